"""x2_to (csrc/common.cuh), the FP32 pair rounded to binary64 on the integer pipes, against the FP64
add of its two parts, bit for bit: every exponent gap, ties and near-ties, powers of two less
something, zero and subnormal parts, infinities and NaNs."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2402_13677_gb300", "csrc")
INCLUDE = os.path.join(HERE, "..", "include")

SRC = r'''
#include <cstdio>
#include "common.cuh"
using namespace ebit;

__device__ unsigned long long mix(unsigned long long z) {   // splitmix64 finaliser
    z += 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}
__device__ unsigned mantissa(unsigned long long r) {
    const unsigned few[8] = {0u, 1u, 2u, 0x7fffffu, 0x7ffffeu, 0x400000u, 0x400001u, 0x3fffffu};
    return (r & 8u) ? (unsigned)(r >> 8) & 0x7fffffu : few[r & 7u];
}
__global__ void k_check(long long n, unsigned long long* bad) {
    long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= n) return;
    unsigned long long r = mix((unsigned long long)t), q = mix(r);
    unsigned eh = (unsigned)(q & 0xffu), gap = (unsigned)((q >> 8) % 80u);
    unsigned el = (q >> 20) & 15u ? (eh > gap ? eh - gap : 0u) : (unsigned)(q >> 24) & 0xffu;
    float hi = __uint_as_float(((unsigned)(r >> 63) << 31) | (eh << 23) | mantissa(mix(q)));
    float lo = __uint_as_float(((unsigned)(r >> 62) << 31) | (el << 23) | mantissa(mix(q + 1)));
    double a = x2_to({hi, lo}), b = (double)hi + (double)lo;
    if (__double_as_longlong(a) != __double_as_longlong(b) && !(a != a && b != b)) atomicAdd(bad, 1ull);
}
int main() {
    unsigned long long *d, h = 1;
    if (cudaMalloc(&d, 8) != cudaSuccess || cudaMemset(d, 0, 8) != cudaSuccess) return 2;
    const long long n = 1ll << 24;
    k_check<<<(unsigned)(n / 256), 256>>>(n, d);
    if (cudaMemcpy(&h, d, 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    printf("%llu\n", h);
    return h == 0 ? 0 : 1;
}
'''


def test_pair_to_binary64_equals_the_fp64_sum(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "pair.cu"
    src.write_text(SRC)
    exe = tmp_path / "pair"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", f"-I{CSRC}", f"-I{INCLUDE}",
                    "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
