// Multigrid-preconditioned conjugate gradients for the implicit solves of the step
// (energy diffusion, viscous Helmholtz, ghost-fluid Poisson).
//
// Operator (integrated five-point form, cell-centred coefficients), applied in flux form:
//     (A x)_i = D_i x_i + wl_i (x_i - x_{i-1}) + wl_{i+1} (x_i - x_{i+1})
//                       + wb_i (x_i - x_{i-nx}) + wb_{i+nx} (x_i - x_{i+nx}),   D_i = cd_i + dd_i
// The flux form keeps the zero row sum of the conductance part exact in any precision: a
// diagonal stored as cd + dd + sum w and rounded to FP32 separately from the w would add a
// spurious diagonal of relative size 6e-8, above the smallest eigenvalue of a 4096^2 Poisson
// operator (condition number ~1e9), and the FP32 solve would stall.  Smoothers use
// diag = D + sum w computed on the fly.
// with cd the h^2 (rho cp / dt or rho / dt) term, dd the Dirichlet contributions (ghost-fluid
// interface links, fixed-temperature or no-slip walls, outflow pressure), wl/wb the left and
// bottom face conductances (zero on domain faces).
//
// Preconditioner: one symmetric V(2,2)-cycle.  Red-black Gauss-Seidel (red-black before,
// black-red after), restriction = sum of the four children, prolongation = injection, coarse
// operators re-discretised (cd summed, dd summed and halved, face weights averaged along the
// coarse face), a fixed symmetric sweep sequence on the coarsest grid.
//
// Kernel structure (few launches per CG iteration):
//   * large levels: k_pre  = 2 red-black sweeps from zero + residual + restriction, and
//                   k_post = prolongation + 2 black-red sweeps (+ r.z at the finest level),
//     each a shared-memory tile with a halo of recomputed cells, so one launch performs
//     several Gauss-Seidel half-sweeps; halo cells are recomputed from the same inputs with
//     the same formula, so the result equals global red-black Gauss-Seidel exactly;
//   * every level of at most 1024 cells: one single-block kernel (k_small) runs the rest of
//     the V-cycle in shared memory;
//   * CG: k_apply (p = z + beta p fused into q = A p, p.q) and k_update (x, r, r.r, test).
// Loop control lives on the device (SolveState); kernels can drive CUDA-graph conditional
// WHILE nodes (cudaGraphSetConditional), or the host can poll the state.
//
// Precision modes:
//   FP64  : CG + V-cycle in double.
//   MIXED : iterative refinement: r = b - A x in FP64, correction A e = r solved in FP32 by
//           the same MG-PCG to a relative 1e-5, x += e in FP64, until ||r|| <= rtol ||b||.
//
// Reductions are deterministic: per-block partial sums, the last block adds them in block order.
#include <algorithm>
#include <atomic>
#include <vector>
#include <cfloat>
#include <type_traits>
#include <cstdio>
#include "common.cuh"
#include "kernels.h"
#include "solver.h"

namespace ebit {

constexpr int RB = 256;          // threads of grid-stride kernels
constexpr int NRED = 608;        // blocks of grid-stride kernels (4 x 152 SMs)
constexpr int SMALL_MAX_F = 1024; // default: levels with at most this many cells run inside k_small (FP32)
constexpr int SMALL_MAX_F_LIMIT = 4096;   // the shared memory of k_small holds at most this level
constexpr int SMALL_MAX_D = 1024; // (FP64: half the shared memory per value)
// the most that the single-block levels of any grid hold: cells (64 x 64 and its levels, rounded up) and
// entries of the bordered x arrays (2048 x 2 and 1024 x 1: their two border rows double them)
constexpr int SMALL_CELLS = 5464, SMALL_XENTRIES = 12296;
constexpr int SMALL_THREADS = 512;   // of the single-block levels (k_small, and block 0 of a cooperative launch)
constexpr size_t SMEM_MAX = 216 * 1024;   // dynamic shared memory of the cluster kernels and the single-block levels, at most
constexpr int SMALL_INV = 32 * 32;   // entries of the coarsest operator's dense inverse, at most
constexpr int TX = 32, TY = 32;  // tile of the large-level kernels
constexpr int NU = 2;            // smoothing sweeps (red-black pairs) before and after
constexpr int NU_SMALL = 2;      // the same on the levels of the single-block kernel
// halo of the tile kernels: every half-sweep after the first leaves one more ring of the region
// stale.  Pre-smoothing starts from x = 0, so its first half-sweep needs no neighbours and is
// exact up to the region edge: 2 NU - 1 further half-sweeps and the residual need 2 NU rings.
// Post-smoothing: 2 NU half-sweeps, then the core only.
constexpr int HPRE = 2 * NU, HPOST = 2 * NU;
constexpr int COARSE_PAIRS = 12; // symmetric sweeps on the coarsest grid (at most 16 cells)

template <typename T, int NR>
struct alignas(sizeof(T) * NR) Vec {
    T v[NR];
};

template <typename T>
struct Lev {
    int nx, ny;
    const T* diag;
    const T* wl;
    const T* wb;
    long long zs;   // byte stride between the instances of a batched launch (0: one instance)
    const T* id;    // FP64: reciprocal of the full diagonal (k_diag_inverse); null in FP32
};

// Reciprocal of a smoother's diagonal.  FP32 (the preconditioner of the inner solves): the
// hardware approximation (one MUFU instruction, within about an ulp; the diagonals are normal
// numbers), the same in every kernel, so that the tile, cooperative and single-block paths stay
// identical; a preconditioner need only be fixed and symmetric, not correctly rounded.  FP64:
// correctly rounded.
__device__ inline float rcp_diag(float v) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}
__device__ inline double rcp_diag(double v) { return __drcp_rn(v); }

__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// residual b - A x of one cell in the smoothers, in flux form (row sums stay exactly D in FP32)
template <typename T>
__device__ inline T cell_residual(T b, T d, T w0, T w1, T w2, T w3, T x, T xl, T xr, T xd, T xu) {
    T ax = d * x + w0 * (x - xl) + w1 * (x - xr) + w2 * (x - xd) + w3 * (x - xu);
    return b - ax;
}

// a state word read now, not at its first use: the words a kernel needs before its work travel
// together with the skip flags (one L2 round trip at the head of these short kernels, not three)
__device__ __forceinline__ int ld_now(const int* p) {
    int v;
    asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ double ld_now(const double* p) {
    double v;
    asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
}
__device__ inline bool skip(const SolveState* s) {
    const int a = ld_now(&s->done), b = ld_now(&s->odone);
    return (a | b) != 0;
}

__device__ inline unsigned long long gtimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Device timing of a tile-kernel launch (one timer per launch; the instances of a batched launch
// share their lead's).  Every block arrives once: a block that runs records its start and end
// (and the first block of each instance counts that instance as active), a block of a converged
// instance only arrives.  The last block to arrive adds the launch's span (first start to last
// end), its launch and the algorithmic bytes of its active instances, and resets the timer.
// Outside ebit_timing_begin / ebit_timing_end the timer is off (KTimer::on, read once at the start
// of a launch): no atomics and no fence at the end of every smoother launch.
__device__ inline bool timer_on(const KTimer* tm) { return tm && threadIdx.x == 0 && ld_now(&tm->on) != 0; }
__device__ inline void timer_begin(KTimer* tm, bool on) {   // on: timer_on, thread 0
    if (on) {
        atomicMin(&tm->start, gtimer());
        if (blockIdx.x == 0 && blockIdx.y == 0) atomicAdd(&tm->active, 1u);
    }
}
__device__ inline void timer_arrive(KTimer* tm, bool on, double bytes_per_instance, bool ran) {
    __syncthreads();
    if (on) {
        if (ran) atomicMax(&tm->end, gtimer());
        __threadfence();
        unsigned int n = gridDim.x * gridDim.y * gridDim.z;
        if (atomicAdd(&tm->ticket, 1u) == n - 1) {
            __threadfence();
            unsigned long long s = atomicAdd(&tm->start, 0ull), e = atomicAdd(&tm->end, 0ull);
            unsigned act = atomicAdd(&tm->active, 0u);
            if (act > 0) {
                tm->total_ns += e > s ? e - s : 0ull;
                tm->launches += 1;
                tm->bytes += bytes_per_instance * act;
            }
            tm->start = ~0ull;
            tm->end = 0ull;
            tm->ticket = 0u;
            tm->active = 0u;
        }
    }
}

// ---- block reductions ---------------------------------------------------------------
__device__ inline double bsum(double v, double* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) sh[w] = v;
    __syncthreads();
    double r = 0.0;
    if (w == 0) {
        r = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
    }
    __syncthreads();
    return r;
}

// Grid reductions in a fixed order.  block_partial writes the block sum of NV per-thread values
// into slot `slot` of partial (partial[k * nslot + slot], thread 0); once every block of the grid
// has written its slots, last_block_total returns true in thread 0 of the last block to arrive,
// with the totals over the nslot slots in tot[0..NV).
// the NV sums share the two block barriers (their shuffle chains overlap)
template <int NV>
__device__ inline void block_partial(const double* v, double* partial, int nslot, int slot) {
    __shared__ double sh[NV][32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double r[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) r[k] = v[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < NV; ++k) r[k] += __shfl_down_sync(0xffffffffu, r[k], o);
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < NV; ++k) sh[k][w] = r[k];
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) r[k] = lane < (int)(blockDim.x >> 5) ? sh[k][lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int k = 0; k < NV; ++k) r[k] += __shfl_down_sync(0xffffffffu, r[k], o);
        if (lane == 0)
#pragma unroll
            for (int k = 0; k < NV; ++k) partial[k * nslot + slot] = r[k];
    }
    __syncthreads();
}
// the same block sum in the solver precision T, converted once (thread 0): the r.z of a tile's
// FP32 cells is summed in FP32 (its slot then joins the FP64 total in tile order), so the tile
// kernels issue no FP64 shuffles
template <typename T>
__device__ inline T bsum_t(T v, T* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) sh[w] = v;
    __syncthreads();
    T r = T(0);
    if (w == 0) {
        r = lane < (int)(blockDim.x >> 5) ? sh[lane] : T(0);
        for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
    }
    __syncthreads();
    return r;
}
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ double widen(float v) { return f2d(v); }
template <typename T, int NV>
__device__ inline void block_partial_t(const T* v, double* partial, int nslot, int slot) {
    __shared__ T sh[32];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        T r = bsum_t(v[k], sh);
        if (threadIdx.x == 0) partial[k * nslot + slot] = widen(r);
    }
}
// Arrival is one atomic add with acquire-release semantics by thread 0, which wrote the block's
// slots itself: it publishes them, and in the last block it (and, through the block barrier,
// every thread) sees the other blocks' slots.  Full fences by every thread around a relaxed
// add cost about a microsecond per launch at the end of these kernels' dependent chain.
__device__ inline unsigned arrive_acq_rel(unsigned* p) {
    unsigned v;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(v) : "l"(p) : "memory");
    return v;
}
template <int NV>
__device__ inline bool last_block_total(double* partial, int nslot, unsigned* ticket, double* tot) {
    __shared__ double sh[NV][32];
    __shared__ bool last;
    if (threadIdx.x == 0) last = arrive_acq_rel(ticket) == gridDim.x * gridDim.y - 1;
    __syncthreads();
    if (!last) return false;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double s[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) s[k] = 0.0;
    for (int b = threadIdx.x; b < nslot; b += blockDim.x)
#pragma unroll
        for (int k = 0; k < NV; ++k) s[k] += __ldcg(partial + k * nslot + b);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < NV; ++k) s[k] += __shfl_down_sync(0xffffffffu, s[k], o);
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < NV; ++k) sh[k][w] = s[k];
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) s[k] = lane < (int)(blockDim.x >> 5) ? sh[k][lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int k = 0; k < NV; ++k) s[k] += __shfl_down_sync(0xffffffffu, s[k], o);
#pragma unroll
        for (int k = 0; k < NV; ++k) tot[k] = s[k];
    }
    if (threadIdx.x == 0) *ticket = 0u;
    return threadIdx.x == 0;
}
// use 1: the loop condition is this solve's own (assigned); use 2: a batched launch, where the
// condition is the OR over the instances (reset to 0 at the top of each loop body by
// k_cond_reset, raised to 1 by every instance that continues)
__device__ inline void set_cond(cudaGraphConditionalHandle h, int use, unsigned v) {
    if (use == 1 || (use == 2 && v)) cudaGraphSetConditional(h, v);
}

__global__ void k_cond_reset(cudaGraphConditionalHandle h0, cudaGraphConditionalHandle h1, int two) {
    if (threadIdx.x == 0) {
        cudaGraphSetConditional(h0, 0u);
        if (two) cudaGraphSetConditional(h1, 0u);
    }
}

// ---- large-level kernels: tiles with recomputed halos ------------------------------------
// A tile kernel owns a TX x TY block of cells and recomputes a halo of H cells around it, so one
// launch performs several red-black half-sweeps with no exchange between blocks (halo cells
// are recomputed from the same inputs with the same formula, so the result equals global
// red-black Gauss-Seidel exactly).
//
// Thread (k, seg) owns the cells of region columns 2k and 2k + 1 in the two rows 2 seg and
// 2 seg + 1; in every row exactly one of its two cells has the colour being swept.  A thread
// keeps its four cells' coefficients (b, the reciprocal of the full diagonal, the four face
// weights, D) in registers; only x lives in shared memory, split by colour.  The region starts
// at an even global cell (tile origins are multiples of TX, TY and the halos are even), so
// region cell (rx, ry) has colour c = (rx + ry) & 1, known at compile time for each of a
// thread's cells.  Colour c's array holds the even rows' cells, then the odd rows', each in thread
// order: cell (r, c) of thread t is entry r TH + t, so a warp's accesses are consecutive words (one
// row of columns after another in the array gave 2.5-way bank conflicts where a warp spans two row
// pairs; with this layout and the paired loads of tile_load_cells k_pre / k_post of 1024x2048 cells take
// 17.1 / 23.4 us, 20.3 / 25.5 before; bound: issue slots and the barriers between half-sweeps).  A
// colour-c cell with e = rx & 1 finds its left / right neighbours (colour 1 - c) at
// threads t - 1 + e / t + e of its row r, its lower / upper ones at row 1 - r of threads t - HX / t
// (r = 0) or t / t + HX (r = 1).
template <typename T, int NR, int H>
struct Region {
    static constexpr int SX = TX + 2 * H, SY = TY + 2 * H, HX = SX / 2, NC = SY * HX;
    static constexpr int NSEG = SY / 2, THREADS = HX * NSEG;
    static_assert(SX % 2 == 0 && SY % 2 == 0, "region sides must be even");
    T* x0;   // x of colour 0 (NR per cell), then colour 1
    __device__ Region(unsigned char* base) { x0 = (T*)base; }
    __device__ T* x(int c) const { return x0 + c * (NR * NC); }
    __device__ static int at(int r, int t) { return r * THREADS + t; }
    static constexpr size_t BYTES = (size_t)2 * NC * NR * sizeof(T);
    __host__ __device__ static constexpr size_t bytes() { return BYTES; }
};
template <int H>
constexpr int tile_block() { return (((TX + 2 * H) / 2) * ((TY + 2 * H) / 2) + 31) / 32 * 32; }
// blocks per SM the FP32 tile kernels are compiled for (register budget: two blocks, 72
// registers, measured 1.2 % faster on the 4096^2 film than three blocks with spills); the FP64
// ones keep the compiler's choice
template <typename T, int NR>
constexpr int tile_min_blocks() { return sizeof(T) == 4 ? 2 : 1; }

// ---- TMA staging of the tile regions ------------------------------------------------------
// One elected thread issues a 2-D tensor copy (cp.async.bulk.tensor) per operand array into
// dense shared-memory boxes and arms an mbarrier with their byte count; every thread waits on
// the barrier (bounded) and then reads its cells from the boxes.  A copy must start at an x
// coordinate whose byte offset is a multiple of 16, so each box starts up to A - 1 cells left
// of the region (A = 16 / bytes per cell) and the region indexes it from that offset; cells
// outside the grid are filled with zeros by the copy.
__device__ inline uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ inline void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ inline void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ inline void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ inline bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ inline void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            smem_u32(dst)),
        "l"((uint64_t)map), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}
// wait for the phase of the barrier with the given parity; false if it did not complete within
// the bound
__device__ inline bool mbar_wait_bounded(uint64_t* bar, uint32_t parity = 0) {
    for (int it = 0; it < (1 << 22); ++it)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}
// order this thread's earlier generic-proxy accesses to shared memory (the block's reads of a
// box, made visible to it by a block barrier) before its next async-proxy (TMA) writes there
__device__ inline void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__host__ __device__ constexpr int pmod(int a, int m) { return ((a % m) + m) % m; }
__host__ __device__ constexpr int floordiv2(int a) { return a >= 0 ? a / 2 : -((-a + 1) / 2); }
__host__ __device__ constexpr int round_up(int a, int m) { return (a + m - 1) / m * m; }
__host__ __device__ constexpr size_t align128(size_t b) { return (b + 127) & ~size_t(127); }

// box geometry of a tile kernel with halo H; POST: k_post (also the pre-smoothed x and the
// coarse x)
template <typename T, int NR, int H, bool POST>
struct Stage {
    static constexpr int SX = TX + 2 * H, SY = TY + 2 * H;
    static constexpr int AS = 16 / (int)sizeof(T);          // x alignment of D, wl, wb (cells)
    static constexpr int AV = 16 / (NR * (int)sizeof(T));   // x alignment of the NR-vector arrays
    static constexpr int OXS = pmod(-H, AS), OXV = pmod(-H, AV), OXC = pmod(floordiv2(-H), AV);
    static constexpr int BWS = round_up(OXS + SX + 1, AS), BHS = SY + 1;   // +1: right / upper faces
    static constexpr int BWV = round_up(OXV + SX, AV), BHV = SY;
    static constexpr int BWC = round_up(OXC + SX / 2 + 1, AV), BHC = SY / 2 + 1;
    static constexpr size_t SB = (size_t)BWS * BHS * sizeof(T);
    static constexpr size_t VB = (size_t)BWV * NR * BHV * sizeof(T);
    static constexpr size_t CB = (size_t)BWC * NR * BHC * sizeof(T);
    // FP64: pre-smoothing also needs the reciprocal diagonal; post-smoothing needs it instead of D
    static constexpr bool ID_BOX = sizeof(T) == 8 && !POST;
    static constexpr int NS = ID_BOX ? 4 : 3;
    static constexpr size_t OFF_D = 0, OFF_WL = align128(SB), OFF_WB = 2 * align128(SB), OFF_ID = 3 * align128(SB);
    static constexpr size_t OFF_B = NS * align128(SB);
    static constexpr size_t OFF_XIN = OFF_B + align128(VB), OFF_XC = OFF_XIN + (POST ? align128(VB) : 0);
    static constexpr size_t OFF_BAR = OFF_XC + (POST ? align128(CB) : 0);
    static constexpr size_t BYTES = OFF_BAR + 128;
    static constexpr uint32_t TX_BYTES = (uint32_t)(NS * SB + VB + (POST ? VB + CB : 0));
    static_assert(BWS <= 256 && BWV * NR <= 256 && BWC * NR <= 256 && BHS <= 256, "TMA box too large");
};

// the copies of one region into the boxes (thread 0): arms the barrier with their byte count
template <typename T, int NR, int H, bool POST>
__device__ inline void stage_issue(unsigned char* sbase, const TileMaps& M, int gx0, int gy0) {
    using Sg = Stage<T, NR, H, POST>;
    uint64_t* bar = reinterpret_cast<uint64_t*>(sbase + Sg::OFF_BAR);
    mbar_expect_tx(bar, Sg::TX_BYTES);
    int xs = gx0 - Sg::OXS, xv = (gx0 - Sg::OXV) * NR;
    tma_load_2d(sbase + Sg::OFF_D, sizeof(T) == 8 && POST ? &M.id : &M.d, xs, gy0, bar);
    if constexpr (Sg::ID_BOX) tma_load_2d(sbase + Sg::OFF_ID, &M.id, xs, gy0, bar);
    tma_load_2d(sbase + Sg::OFF_WL, &M.wl, xs, gy0, bar);
    tma_load_2d(sbase + Sg::OFF_WB, &M.wb, xs, gy0, bar);
    tma_load_2d(sbase + Sg::OFF_B, &M.b, xv, gy0, bar);
    if (POST) {
        tma_load_2d(sbase + Sg::OFF_XIN, &M.xin, xv, gy0, bar);
        tma_load_2d(sbase + Sg::OFF_XC, &M.xc, ((gx0 >> 1) - Sg::OXC) * NR, gy0 >> 1, bar);
    }
}

// barrier set-up and the copies of the block's first tile (thread 0), at the very start of the
// kernel so that they overlap the reads of the solve state
template <typename T, int NR, int H, bool POST>
__device__ inline void stage_first(unsigned char* sbase, const TileMaps& M, int tx) {
    if (threadIdx.x == 0) {
        mbar_init(reinterpret_cast<uint64_t*>(sbase + Stage<T, NR, H, POST>::OFF_BAR), 1);
        mbar_fence_init();
        stage_issue<T, NR, H, POST>(sbase, M, ((int)blockIdx.x % tx) * TX - H, ((int)blockIdx.x / tx) * TY - H);
    }
}

// a block that leaves without work waits (bounded) for the copies it has in flight
template <typename T, int NR, int H, bool POST>
__device__ inline void stage_drain(unsigned char* sbase) {
    if (threadIdx.x == 0) mbar_wait_bounded(reinterpret_cast<uint64_t*>(sbase + Stage<T, NR, H, POST>::OFF_BAR), 0);
}

// The tiles of a TMA-staged tile kernel, persistent: block b takes tiles b, b + G, ... (G blocks,
// at most one per tile; stage_first has requested the first one).
// The next tile's boxes are requested as soon as the current tile has been read out of them
// (into registers and the region), so the copies overlap the current tile's sweeps.  work(t,
// after_load) runs tile t and calls after_load() once the boxes have been read and the block has
// passed a barrier.  A copy that does not land within the bound sets st->fault bit 0 and ends
// the loop (the decision is the same in every thread) after one more bounded wait for that
// copy, the only one in flight.
template <typename T, int NR, int H, bool POST, class Work>
__device__ inline void staged_tiles(unsigned char* sbase, const TileMaps& M, int tx, int nt, SolveState* st,
                                    Work&& work) {
    using Sg = Stage<T, NR, H, POST>;
    uint64_t* bar = reinterpret_cast<uint64_t*>(sbase + Sg::OFF_BAR);
    __syncthreads();   // the barrier's set-up
    // tile t = by tx + bx, advanced by gridDim.x = gq tx + gr without a division per tile
    int t = blockIdx.x, bx = t % tx, by = t / tx;
    const int gq = (int)gridDim.x / tx, gr = (int)gridDim.x % tx;
    for (uint32_t i = 0; t < nt; ++i) {
        bool landed = mbar_wait_bounded(bar, i & 1u);
        if (__syncthreads_or(!landed)) {
            if (threadIdx.x == 0) atomicOr(&st->fault, 1);
            mbar_wait_bounded(bar, i & 1u);
            __syncthreads();
            break;
        }
        int tn = t + gridDim.x, bxn = bx + gr, byn = by + gq;
        if (bxn >= tx) { bxn -= tx; ++byn; }
        work(t, bx, by, [&]() {
            if (threadIdx.x == 0 && tn < nt) {
                fence_proxy_async();
                stage_issue<T, NR, H, POST>(sbase, M, bxn * TX - H, byn * TY - H);
            }
        });
        __syncthreads();   // the region is rewritten by the next tile
        t = tn;
        bx = bxn;
        by = byn;
    }
}


// the thread's four cells: [r][c] = row ry0 + r (ry0 even), colour c; its column is 2k + (c ^ r)
template <typename T, int NR>
struct Cells {
    T b[2][2][NR], id[2][2], wl[2][2], wr[2][2], wb[2][2], wt[2][2], d[2][2];
    // the cells' current x (the copy in shared memory is for the neighbour threads): two of a
    // cell's four neighbours are the thread's own cells of the other colour
    T x[2][2][NR];
};

// n consecutive elements (4, 8 or a multiple of 16 bytes, so aligned)
template <int N, typename T>
__device__ inline void load_row(const T* s, T* o) {
    constexpr int W = N * sizeof(T) > 16 ? 16 / (int)sizeof(T) : N;
    static_assert(N % W == 0, "whole words");
#pragma unroll
    for (int q = 0; q < N; q += W) {
        const Vec<T, W> v = *reinterpret_cast<const Vec<T, W>*>(s + q);
#pragma unroll
        for (int w = 0; w < W; ++w) o[q + w] = v.v[w];
    }
}

// load the thread's cells (coefficients to registers, x to shared memory: for pre-smoothing
// the result of the first colour-0 half-sweep from x = 0, for post-smoothing xin + the
// prolongated coarse x); cells outside the domain get D = 1, zero weights, b = x = 0, so
// sweeps leave them 0.  The two cells of a row are adjacent, in the boxes and in the level's arrays:
// one 8 or 16 byte load per operand (all tiled levels have even sides, their arrays and offsets are
// aligned to a pair)
template <typename T, int NR, int H, bool POST, bool STAGED, bool CHECK>
__device__ inline void tile_load_cells(Region<T, NR, H>& R, Cells<T, NR>& C, int k, int ry0, const Lev<T>& L,
                                       const T* __restrict__ b, const T* __restrict__ xin, const T* __restrict__ xc,
                                       int cnx, int gx0, int gy0, const unsigned char* stage) {
    using Rg = Region<T, NR, H>;
    using Sg = Stage<T, NR, H, POST>;
    static_assert(H % 2 == 0 && TX % 2 == 0 && TY % 2 == 0, "regions must start at an even cell");
    static_assert(Sg::OXS % 2 == 0 && Sg::OXV % 2 == 0, "a cell pair is aligned in its box");
    constexpr bool ID = sizeof(T) == 8;
    T dp[2][2], idp[2][2], wlp[2][3], wbp[3][2], bp[2][2 * NR], xp[2][2 * NR];   // [row][column]
    if constexpr (STAGED) {
        // from the TMA boxes (zeros outside the grid)
        const T* sd = reinterpret_cast<const T*>(stage + Sg::OFF_D);
        const T* swl = reinterpret_cast<const T*>(stage + Sg::OFF_WL);
        const T* swb = reinterpret_cast<const T*>(stage + Sg::OFF_WB);
        const T* sb = reinterpret_cast<const T*>(stage + Sg::OFF_B);
        const int q0 = ry0 * Sg::BWS + 2 * k + Sg::OXS;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int qs = q0 + r * Sg::BWS, qv = ((ry0 + r) * Sg::BWV + 2 * k + Sg::OXV) * NR;
            load_row<2>(sd + qs, dp[r]);
            if constexpr (Sg::ID_BOX) load_row<2>(reinterpret_cast<const T*>(stage + Sg::OFF_ID) + qs, idp[r]);
            load_row<2>(swl + qs, wlp[r]);
            wlp[r][2] = swl[qs + 2];
            load_row<2>(swb + qs, wbp[r]);
            load_row<2 * NR>(sb + qv, bp[r]);
            if constexpr (POST) load_row<2 * NR>(reinterpret_cast<const T*>(stage + Sg::OFF_XIN) + qv, xp[r]);
        }
        load_row<2>(swb + q0 + 2 * Sg::BWS, wbp[2]);
        if constexpr (POST) {   // the block's four cells have one coarse parent
            T cv[NR];
            load_row<NR>(reinterpret_cast<const T*>(stage + Sg::OFF_XC) + ((ry0 >> 1) * Sg::BWC + k + Sg::OXC) * NR, cv);
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int q = 0; q < 2 * NR; ++q) xp[r][q] += cv[q % NR];
        }
    }
    // the block is in the grid or out of it as a whole (sides and tile origins are even)
    const int gi0 = gx0 + 2 * k, gj0 = gy0 + ry0;
    const bool in = !CHECK || (gj0 >= 0 && gj0 < L.ny && gi0 >= 0 && gi0 < L.nx);
    if constexpr (!STAGED) {
        // unconditional loads (clamped, then masked): all of them can be in flight at once
        const int gic = CHECK ? min(max(gi0, 0), L.nx - 2) : gi0, gjc = CHECK ? min(max(gj0, 0), L.ny - 2) : gj0;
        const bool rgt = !CHECK || gic + 2 < L.nx, up = !CHECK || gjc + 2 < L.ny;
        const T* D = ID && POST ? L.id : L.diag;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int g = (gjc + r) * L.nx + gic;
            load_row<2>(D + g, dp[r]);
            if constexpr (Sg::ID_BOX) load_row<2>(L.id + g, idp[r]);
            load_row<2>(L.wl + g, wlp[r]);
            wlp[r][2] = L.wl[rgt ? g + 2 : g];
            if (CHECK && !rgt) wlp[r][2] = T(0);
            load_row<2>(L.wb + g, wbp[r]);
            load_row<2 * NR>(b + (size_t)g * NR, bp[r]);
            if constexpr (POST) load_row<2 * NR>(xin + (size_t)g * NR, xp[r]);
        }
        load_row<2>(L.wb + (up ? gjc + 2 : gjc) * L.nx + gic, wbp[2]);
        if (CHECK && !up) wbp[2][0] = wbp[2][1] = T(0);
        if constexpr (POST) {
            T cv[NR];
            load_row<NR>(xc + (size_t)((gjc >> 1) * cnx + (gic >> 1)) * NR, cv);
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int q = 0; q < 2 * NR; ++q) xp[r][q] += cv[q % NR];
        }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            Vec<T, NR> bv, xv;
            T dv = dp[r][e], wlv = wlp[r][e], wbv = wbp[r][e], wrv = wlp[r][e + 1], wtv = wbp[r + 1][e];
            T idv = !ID ? T(1) : Sg::ID_BOX ? idp[r][e] : dv;   // FP64: loaded (and D only where a residual follows)
#pragma unroll
            for (int k2 = 0; k2 < NR; ++k2) {
                bv.v[k2] = bp[r][e * NR + k2];
                xv.v[k2] = POST ? xp[r][e * NR + k2] : T(0);
            }
            if (CHECK && !in) {
#pragma unroll
                for (int k2 = 0; k2 < NR; ++k2) { bv.v[k2] = T(0); xv.v[k2] = T(0); }
                dv = idv = T(1);
                wlv = wbv = wrv = wtv = T(0);
            }
            // this cell's colour is e ^ r (both known at compile time)
            bool mine0 = (e ^ r) == 0;
            if (!ID) idv = rcp_diag(dv + wlv + wrv + wbv + wtv);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                bool m = (c == 0) == mine0;
                if (m) {
#pragma unroll
                    for (int k2 = 0; k2 < NR; ++k2) C.b[r][c][k2] = bv.v[k2];
                    C.id[r][c] = idv;
                    C.wl[r][c] = wlv;
                    C.wr[r][c] = wrv;
                    C.wb[r][c] = wbv;
                    C.wt[r][c] = wtv;
                    if (!(ID && POST)) C.d[r][c] = dv;
                }
            }
            int cc = e ^ r;
            if (!POST && cc == 0) {
                // pre-smoothing starts from x = 0: its first (colour-0) half-sweep reads only
                // zeros and reduces to x = b / (full diagonal), done here
#pragma unroll
                for (int k2 = 0; k2 < NR; ++k2) xv.v[k2] = bv.v[k2] * idv;
            }
            T* xd = R.x(cc) + Rg::at(r, threadIdx.x) * NR;
#pragma unroll
            for (int k2 = 0; k2 < NR; ++k2) {
                xd[k2] = xv.v[k2];
                C.x[r][cc][k2] = xv.v[k2];
            }
        }
    }
}

// A region wholly inside the grid, with the right and upper faces of its last cells too (all
// but the tiles along the grid's edges), needs no range tests or masks
template <typename T, int NR, int H, bool POST, bool STAGED>
__device__ inline void tile_load(Region<T, NR, H>& R, Cells<T, NR>& C, int k, int ry0, const Lev<T>& L,
                                 const T* __restrict__ b, const T* __restrict__ xin, const T* __restrict__ xc,
                                 int cnx, int gx0, int gy0, const unsigned char* stage) {
    constexpr int SX = Region<T, NR, H>::SX, SY = Region<T, NR, H>::SY;
    if (gx0 >= 0 && gy0 >= 0 && gx0 + SX < L.nx && gy0 + SY < L.ny)
        tile_load_cells<T, NR, H, POST, STAGED, false>(R, C, k, ry0, L, b, xin, xc, cnx, gx0, gy0, stage);
    else
        tile_load_cells<T, NR, H, POST, STAGED, true>(R, C, k, ry0, L, b, xin, xc, cnx, gx0, gy0, stage);
}

// A thread's place in a tile region, the same for every tile of a launch (computed once per
// launch, one register): bit 2 (S - 1) + r is set if half-sweep S updates the thread's cell
// (r, COLOR ^ r) (distance >= S from the region's edge; COLOR, the sweep's colour, is S & 1),
// bit 8 + 2 r + c if cell (r, c) lies in the tile's core, bit 12 if the thread owns cells.  The
// column pair k and the row pair ry0 follow from threadIdx (a division by a constant).
struct TileThread {
    unsigned m;
    __device__ bool act() const { return (m >> 12) & 1u; }
    __device__ bool sweeps(int S, int r) const { return (m >> (2 * (S - 1) + r)) & 1u; }
    __device__ bool core(int r, int c) const { return (m >> (8 + 2 * r + c)) & 1u; }
};
template <int H>
__device__ inline TileThread tile_thread() {
    constexpr int SX = TX + 2 * H, SY = TY + 2 * H, HX = SX / 2, THREADS = HX * (SY / 2);
    const int k = threadIdx.x % HX, ry0 = 2 * (threadIdx.x / HX);
    unsigned m = threadIdx.x < THREADS ? 1u << 12 : 0u;
#pragma unroll
    for (int S = 1; S <= 4; ++S)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            int ry = ry0 + r, rx = 2 * k + ((S & 1) ^ r);
            if (ry >= S && ry < SY - S && rx >= S && rx < SX - S) m |= 1u << (2 * (S - 1) + r);
        }
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            int ry = ry0 + r, rx = 2 * k + (c ^ r);
            if (rx >= H && rx < H + TX && ry >= H && ry < H + TY) m |= 1u << (8 + 2 * r + c);
        }
    return TileThread{m};
}

// one Gauss-Seidel half-sweep of colour COLOR over the region cells at distance >= S from its
// edge; both rows' operands are loaded before either result is stored.  Cell (r, e) of the
// thread (colour COLOR, e = COLOR ^ r) has its horizontal neighbour 2k + 1 - e and its vertical
// neighbour in row 1 - r among the thread's own cells (registers); the other two come from the
// neighbour threads through shared memory.
template <typename T, int NR, int H, int S, int COLOR>
__device__ inline void tile_sweep(Region<T, NR, H>& R, Cells<T, NR>& C, const TileThread& tt) {
    static_assert(COLOR == (S & 1), "half-sweep S has colour S & 1");
    using Rg = Region<T, NR, H>;
    constexpr int HX = Rg::HX;
    if (tt.act()) {
        const T* xo = R.x(1 - COLOR);
        T acc[2][NR];
        bool ok[2];
        int qs[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int e = COLOR ^ r;
            ok[r] = tt.sweeps(S, r);
            const int t = ok[r] ? threadIdx.x : HX + 1;   // a harmless in-range slot otherwise
            const int q = Rg::at(r, t), qv = r == 1 ? Rg::at(0, t + HX) : Rg::at(1, t - HX);
            qs[r] = q;
#pragma unroll
            for (int k2 = 0; k2 < NR; ++k2) {
                const T own_h = C.x[r][1 - COLOR][k2], own_v = C.x[1 - r][1 - COLOR][k2];
                T xl = e == 1 ? own_h : xo[(q - 1) * NR + k2];
                T xrt = e == 0 ? own_h : xo[(q + 1) * NR + k2];
                T xd = r == 1 ? own_v : xo[qv * NR + k2];
                T xu = r == 0 ? own_v : xo[qv * NR + k2];
                acc[r][k2] = (C.b[r][COLOR][k2] + C.wl[r][COLOR] * xl + C.wr[r][COLOR] * xrt +
                              C.wb[r][COLOR] * xd + C.wt[r][COLOR] * xu) *
                             C.id[r][COLOR];
            }
        }
        T* xs = R.x(COLOR);
#pragma unroll
        for (int r = 0; r < 2; ++r)
            if (ok[r])
#pragma unroll
                for (int k2 = 0; k2 < NR; ++k2) {
                    xs[qs[r] * NR + k2] = acc[r][k2];
                    C.x[r][COLOR][k2] = acc[r][k2];
                }
    }
    __syncthreads();
}

// the thread's core cells (inside the TX x TY tile and the domain): f(r, c, gi, gj)
template <typename T, int NR, int H, class Fn>
__device__ inline void tile_core_cells(const Cells<T, NR>& C, const TileThread& tt, int gx0, int gy0,
                                       const Lev<T>& L, Fn&& f) {
    constexpr int HX = Region<T, NR, H>::HX;
    const int k = threadIdx.x % HX, ry0 = 2 * (threadIdx.x / HX);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        int ry = ry0 + r;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            int rx = 2 * k + (c ^ r);
            int gi = gx0 + rx, gj = gy0 + ry;
            if (tt.core(r, c) && gi < L.nx && gj < L.ny) f(r, c, gi, gj);
        }
    }
}

struct NoOp {
    __device__ void operator()() const {}
};

// pre-smoothing of tile (bx, by): x = S^nu(0; b) on the tile (red-black order), coarse
// b = R (b - A x); smem holds the region (STAGED: `stage` its TMA boxes, already landed);
// after_load() runs in every thread once the boxes have been read
template <typename T, int NR, bool STAGED = false, class AfterLoad = NoOp>
__device__ inline void pre_tile(const Lev<T>& L, const T* __restrict__ b, T* __restrict__ x, T* __restrict__ bc,
                                int bx, int by, unsigned char* smem, const unsigned char* stage,
                                const TileThread& tt, AfterLoad after_load = AfterLoad()) {
    constexpr int H = HPRE;
    static_assert(NU == 2, "the sweep sequence below is written out for two pairs");
    using Rg = Region<T, NR, H>;
    constexpr int HX = Rg::HX;
    Rg R(smem);
    int gx0 = bx * TX - H, gy0 = by * TY - H;
    const bool act = tt.act();
    const int k = threadIdx.x % HX, ry0 = 2 * (threadIdx.x / HX);
    Cells<T, NR> C;
    if (act) tile_load<T, NR, H, false, STAGED>(R, C, k, ry0, L, b, nullptr, nullptr, 0, gx0, gy0, stage);
    __syncthreads();
    after_load();
    // the first colour-0 half-sweep (from x = 0) was done by tile_load
    tile_sweep<T, NR, H, 1, 1>(R, C, tt);
    tile_sweep<T, NR, H, 2, 0>(R, C, tt);
    tile_sweep<T, NR, H, 3, 1>(R, C, tt);
    // x of the core cells to global memory, their residuals in registers ([r][e]: row ry0 + r,
    // column 2k + e)
    T res[2][2][NR];
    if (act)
        tile_core_cells<T, NR, H>(C, tt, gx0, gy0, L, [&](int r, int c, int gi, int gj) {
            const T* xo = R.x(1 - c);
            const int e = c ^ r;   // column 2k + e
            const int q = Rg::at(r, threadIdx.x), qv = r == 1 ? Rg::at(0, threadIdx.x + HX) : Rg::at(1, threadIdx.x - HX);
            Vec<T, NR> xv;
#pragma unroll
            for (int k2 = 0; k2 < NR; ++k2) {
                T x0v = C.x[r][c][k2];
                xv.v[k2] = x0v;
                const T own_h = C.x[r][1 - c][k2], own_v = C.x[1 - r][1 - c][k2];
                T xl = e == 1 ? own_h : xo[(q - 1) * NR + k2];
                T xrt = e == 0 ? own_h : xo[(q + 1) * NR + k2];
                T xd = r == 1 ? own_v : xo[qv * NR + k2];
                T xu = r == 0 ? own_v : xo[qv * NR + k2];
                res[r][e][k2] = cell_residual(C.b[r][c][k2], C.d[r][c], C.wl[r][c], C.wr[r][c], C.wb[r][c],
                                              C.wt[r][c], x0v, xl, xrt, xd, xu);
            }
            reinterpret_cast<Vec<T, NR>*>(x)[gj * L.nx + gi] = xv;
        });
    // restriction: sum of the four children.  The region starts H (even) cells before the tile,
    // so a thread's 2 x 2 block is the four children of coarse cell (k - H/2, ry0/2 - H/2) of the
    // tile; a coarse cell of the grid has all four children inside the grid, hence computed above
    int cnx = L.nx / 2, cny = L.ny / 2;
    int ti = k - H / 2, tj = ry0 / 2 - H / 2;
    if (act && ti >= 0 && ti < TX / 2 && tj >= 0 && tj < TY / 2) {
        int ci = bx * (TX / 2) + ti, cj = by * (TY / 2) + tj;
        if (ci < cnx && cj < cny) {
            Vec<T, NR> acc;
#pragma unroll
            for (int k2 = 0; k2 < NR; ++k2) acc.v[k2] = res[0][0][k2] + res[0][1][k2] + res[1][0][k2] + res[1][1][k2];
            reinterpret_cast<Vec<T, NR>*>(bc)[cj * cnx + ci] = acc;
        }
    }
}

// k_pre: one tile per block
template <typename T, int NR>
__global__ void __launch_bounds__(tile_block<HPRE>(), tile_min_blocks<T, NR>())
k_pre(Lev<T> L, const T* __restrict__ b, T* __restrict__ x, T* __restrict__ bc, SolveState* st, KTimer* tm,
      const __grid_constant__ TileMaps maps, int use_tma, unsigned* coop_bar) {
    // the cooperative coarse-cycle launch that follows this (level-0) launch counts its
    // barrier arrivals from 0; the previous one has completed (stream order)
    if (coop_bar && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0) *coop_bar = 0u;
    const long long zo = zoff(L.zs);
    L.diag = zsh(L.diag, zo);
    L.wl = zsh(L.wl, zo);
    L.wb = zsh(L.wb, zo);
    L.id = zsh(L.id, zo);
    b = zsh(b, zo);
    x = zsh(x, zo);
    bc = zsh(bc, zo);
    st = zsh(st, zo);
    constexpr double bytes_cell = sizeof(T) * (3.0 + NR * 2.25);
    constexpr int H = HPRE;
    using Rg = Region<T, NR, H>;
    extern __shared__ __align__(128) unsigned char smem[];
    // TMA boxes 128-byte aligned after the region (the launch reserves 128 bytes of slack)
    unsigned char* stage =
        reinterpret_cast<unsigned char*>(align128(reinterpret_cast<uintptr_t>(smem) + Rg::BYTES));
    if (use_tma) stage_first<T, NR, H, false>(stage, maps, (L.nx + TX - 1) / TX);
    const bool ton = timer_on(tm);
    if (skip(st)) {
        if (use_tma) stage_drain<T, NR, H, false>(stage);
        timer_arrive(tm, ton, 0.0, false);
        return;
    }
    timer_begin(tm, ton);
    if (use_tma) {
        // persistent blocks over the tiles (1-D grid)
        int tx = (L.nx + TX - 1) / TX, nt = tx * ((L.ny + TY - 1) / TY);
        const TileThread tt = tile_thread<H>();
        staged_tiles<T, NR, H, false>(stage, maps, tx, nt, st, [&](int, int bx, int by, auto after_load) {
            pre_tile<T, NR, true>(L, b, x, bc, bx, by, smem, stage, tt, after_load);
        });
    } else {
        pre_tile<T, NR>(L, b, x, bc, blockIdx.x, blockIdx.y, smem, nullptr, tile_thread<H>());
    }
    // algorithmic bytes: b, diag, wl, wb read; x and the quarter-size coarse b written
    timer_arrive(tm, ton, (double)L.nx * L.ny * bytes_cell, true);
}

// post-smoothing of tile (bx, by): x = xin + P xc, then black-red sweeps; returns the tile's
// part of r.z (each right-hand side) when DOT; after_load() as for pre_tile
template <typename T, int NR, bool DOT, bool STAGED = false, class AfterLoad = NoOp>
__device__ inline Vec<T, 2> post_tile(const Lev<T>& L, const T* __restrict__ b, const T* __restrict__ xin,
                                    T* __restrict__ x, const T* __restrict__ xc, int bx, int by, unsigned char* smem,
                                    const unsigned char* stage, const TileThread& tt,
                                    AfterLoad after_load = AfterLoad()) {
    constexpr int H = HPOST;
    using Rg = Region<T, NR, H>;
    Rg R(smem);
    int gx0 = bx * TX - H, gy0 = by * TY - H;
    constexpr int HX = Rg::HX;
    const bool act = tt.act();
    Cells<T, NR> C;
    if (act)
        tile_load<T, NR, H, true, STAGED>(R, C, threadIdx.x % HX, 2 * (threadIdx.x / HX), L, b, xin, xc, L.nx / 2, gx0, gy0,
                                          stage);
    __syncthreads();
    after_load();
    tile_sweep<T, NR, H, 1, 1>(R, C, tt);
    tile_sweep<T, NR, H, 2, 0>(R, C, tt);
    tile_sweep<T, NR, H, 3, 1>(R, C, tt);
    tile_sweep<T, NR, H, 4, 0>(R, C, tt);
    // r.z of the thread's (at most four) core cells, summed in T
    Vec<T, 2> dot;
    dot.v[0] = dot.v[1] = T(0);
    if (act)
        tile_core_cells<T, NR, H>(C, tt, gx0, gy0, L, [&](int r, int c, int gi, int gj) {
            Vec<T, NR> xv;
#pragma unroll
            for (int k2 = 0; k2 < NR; ++k2) {
                xv.v[k2] = C.x[r][c][k2];
                if (DOT) dot.v[k2] += xv.v[k2] * C.b[r][c][k2];
            }
            reinterpret_cast<Vec<T, NR>*>(x)[gj * L.nx + gi] = xv;
        });
    return dot;
}

// k_post: one tile per block; at the finest level also r.z -> beta
template <typename T, int NR, bool DOT>
__global__ void __launch_bounds__(tile_block<HPOST>(), tile_min_blocks<T, NR>())
k_post(Lev<T> L, const T* __restrict__ b, const T* __restrict__ xin, T* __restrict__ x, const T* __restrict__ xc,
       SolveState* st, double* partial, unsigned* ticket, KTimer* tm, const __grid_constant__ TileMaps maps,
       int use_tma) {
    const long long zo = zoff(L.zs);
    L.diag = zsh(L.diag, zo);
    L.wl = zsh(L.wl, zo);
    L.wb = zsh(L.wb, zo);
    L.id = zsh(L.id, zo);
    b = zsh(b, zo);
    xin = zsh(xin, zo);
    x = zsh(x, zo);
    xc = zsh(xc, zo);
    st = zsh(st, zo);
    partial = zsh(partial, zo);
    ticket = zsh(ticket, zo);
    constexpr double bytes_cell = sizeof(T) * (3.0 + NR * 3.25);
    constexpr int H = HPOST;
    using Rg = Region<T, NR, H>;
    extern __shared__ __align__(128) unsigned char smem[];
    unsigned char* stage =
        reinterpret_cast<unsigned char*>(align128(reinterpret_cast<uintptr_t>(smem) + Rg::BYTES));
    if (use_tma) stage_first<T, NR, H, true>(stage, maps, (L.nx + TX - 1) / TX);
    const bool ton = timer_on(tm);
    double rz_old[NR];
#pragma unroll
    for (int k2 = 0; k2 < NR; ++k2) rz_old[k2] = DOT ? ld_now(&st->rz[k2]) : 0.0;
    if (skip(st)) {
        if (use_tma) stage_drain<T, NR, H, true>(stage);
        timer_arrive(tm, ton, 0.0, false);
        return;
    }
    timer_begin(tm, ton);
    int nslot = gridDim.x * gridDim.y;
    if (use_tma) {
        // persistent blocks over the tiles (1-D grid); r.z summed over the block's tiles
        int tx = (L.nx + TX - 1) / TX, nt = tx * ((L.ny + TY - 1) / TY);
        // r.z: one slot per tile, summed in tile order as with one block per tile
        const TileThread tt = tile_thread<H>();
        staged_tiles<T, NR, H, true>(stage, maps, tx, nt, st, [&](int t, int bx, int by, auto after_load) {
            Vec<T, 2> d = post_tile<T, NR, DOT, true>(L, b, xin, x, xc, bx, by, smem, stage, tt, after_load);
            if (DOT) block_partial_t<T, NR>(d.v, partial, nt, t);
        });
        nslot = nt;
    } else {
        Vec<T, 2> d = post_tile<T, NR, DOT>(L, b, xin, x, xc, blockIdx.x, blockIdx.y, smem, nullptr,
                                            tile_thread<H>());
        if (DOT) block_partial_t<T, NR>(d.v, partial, nslot, blockIdx.y * gridDim.x + blockIdx.x);
    }
    if (DOT) {
        double tot[NR];
        if (last_block_total<NR>(partial, nslot, ticket, tot)) {
#pragma unroll
            for (int k2 = 0; k2 < NR; ++k2) {
                st->beta[k2] = rz_old[k2] != 0.0 ? tot[k2] / rz_old[k2] : 0.0;
                st->rz[k2] = tot[k2];
            }
        }
    }
    // algorithmic bytes: b, x, the quarter-size coarse x, diag, wl, wb read; x written
    timer_arrive(tm, ton, (double)L.nx * L.ny * bytes_cell, true);
}

// 16 bytes from global to shared memory, asynchronously (both 16-byte aligned)
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// n elements, the block's threads together; 16-byte pieces in flight at once, plain copies of the rest
template <typename T>
__device__ inline void copy_async(T* dst, const T* src, int n) {
    constexpr int E = 16 / sizeof(T);
    const bool al = ((reinterpret_cast<uintptr_t>(src) | (uintptr_t)smem_u32(dst)) & 15u) == 0;
    const int nv = al ? n / E : 0;
    for (int i = threadIdx.x; i < nv; i += blockDim.x) cp_async16(dst + i * E, src + i * E);
    for (int i = nv * E + threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}

// ---- small levels: the rest of the V-cycle in one block ---------------------------------
struct SmallPlan {
    int n;             // number of small levels
    int nx[Solver::MAXLEV], ny[Solver::MAXLEV];
    int soff[Solver::MAXLEV];   // cell offset of each small level inside the shared-memory arrays
    int xoff[Solver::MAXLEV];   // first entry of each level in the colour-split x array
    size_t goff[Solver::MAXLEV]; // cell offset in the packed global level arrays
    int cells;         // cells of all small levels
    int total;         // the same rounded up to a multiple of four
    int xtotal;        // entries of the colour-split x array
    long long zs;      // byte stride between the instances of a batched launch
};

// What bounds this part is a chain of about forty dependent half-sweeps of a few cells per
// thread: latency of a shared-memory access, five dependent multiply-adds and a barrier, not
// bandwidth.  Thread t of a level owns the 2 x 2 block of cells (2I + e, 2J + r), the four
// children of one cell of the next level, for the level's whole down or up leg:
//   * coefficients, right-hand side and x of its cells stay in registers through a leg; only x
//     goes through shared memory, split by colour (unit stride), and two of a cell's four
//     neighbours are the thread's own cells;
//   * a level's barriers count only the warps that own cells of it (named barrier 1 + level;
//     a warp barrier below 33 blocks), so the deep levels run on one warp;
//   * the restriction is the sum of the block's four residuals, all in one thread.
//   * x has a zero border, so a half-sweep reads its outer neighbours without a test or branch.
// k_small on 32^2 cells, rows of lanes walking a level with every operand read from shared memory
// before: FP32 11.8 -> 8.2 us (one right-hand side), 14.8 -> 10.1 (two), FP64 29 -> 25 and 45 -> 40;
// with a coarsest level solved by 48 half-sweeps (336^2 grid, 21^2 cells) a step 1.78 -> 1.35 ms.

// shared-memory layout: x (colour-split) and b, NR per cell, then diag, wl, (FP64) the reciprocals of
// the full diagonals, wb per cell and the transposed inverse of the coarsest operator
template <typename T, int NR>
struct SmallMem {
    Vec<T, NR>*x, *b;
    T *d, *wl, *wb, *id, *inv;
    __device__ SmallMem(unsigned char* base, const SmallPlan& P) {
        x = (Vec<T, NR>*)base;
        b = x + P.xtotal;
        d = (T*)(b + P.total);
        wl = d + P.total;
        id = wl + P.total;
        wb = id + (sizeof(T) == 8 ? P.total : 0);
        inv = wb + P.total;
    }
    static size_t bytes(int total, int xtotal) {
        return ((size_t)total * (NR + 3 + (sizeof(T) == 8 ? 1 : 0)) + (size_t)xtotal * NR + SMALL_INV) * sizeof(T);
    }
    static size_t bytes(const SmallPlan& P) { return bytes(P.total, P.xtotal); }
};

__device__ inline void team_sync(int l, int threads) {
    if (threads <= 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(l + 1), "r"(threads) : "memory");
}

// A level's x array: one entry per 2 cells of a colour, rows -1 .. 2 hy of hx entries each and one
// spare entry at either end; rows outside the level and the spare entries stay zero.  Cell (i, j)
// is entry xidx(i >> 1, j) of colour (i + j) & 1.  A block reads its eight outer neighbours without
// a test: beyond a left or right side that is an entry of the next row, times a zero weight.
__host__ __device__ constexpr int x_entries(int hx, int rows) { return (rows + 2) * hx + 2; }   // per colour
__device__ __forceinline__ int xidx(int hx, int I, int j) { return 1 + (j + 1) * hx + I; }
// t / n for 0 <= t < 2^13 (the quotient of t + 1/2 is at least 1 / (2 n) from an integer)
__device__ __forceinline__ int small_div(int t, int n) { return (int)__fdividef((float)t + 0.5f, (float)n); }

// residual of a cell of column parity e on the single-block levels: the flux form with the
// rounding of its first sum fixed (one right-hand side fuses D x in the cells of odd columns, two
// fuse the first flux).  The operands are selected, not the results: one FP64 instruction.
template <typename T, int NR>
__device__ __forceinline__ T small_residual(int e, T b, T d, T w0, T w1, T w2, T w3, T x, T xl, T xr, T xd, T xu) {
    const bool dx = NR == 1 && e == 1;
    const T f = x - xl;
    T ax = fma_rn(dx ? d : w0, dx ? x : f, (dx ? w0 : d) * (dx ? f : x));
    ax = fma_rn(w1, x - xr, ax);
    ax = fma_rn(w2, x - xd, ax);
    ax = fma_rn(w3, x - xu, ax);
    return b - ax;
}

// What a block reads of a level: nx columns, rows [0, ny) of it in these arrays (row pitch nx, and
// one row more of wb), cell weights as in Lev
template <typename T, int NR>
struct BlkSrc {
    int nx, ny;
    const T *d, *wl, *wb, *id;
    const Vec<T, NR>* b;
};
// which neighbours exist (weights of the others are 0)
struct BlkSides {
    bool left, right, down, up;
};

// A thread's cells in FP32: the 2 x 2 block of columns 2I, 2I + 1 and rows j, j + 1 (j even), the four
// children of one coarser cell.  [r][e]: row j + r, column 2I + e, colour e ^ r; wl[r][0..2] the weights of
// the row's three vertical faces, wb[0..2][e] of the column's three horizontal ones.  Cells beyond
// an odd side (ODD levels) have b = x = 0 and zero weights.
template <typename T, int NR>
struct QuadBlk {
    using V = Vec<T, NR>;
    static constexpr int RB = 2;                       // rows of a block
    V b[2][2], x[2][2];
    T id[2][2], d[2][2], wl[2][3], wb[3][2];
    int q;        // x entry of the first row: row r of either colour at q + r hx
    bool own;     // the thread owns a block
    __host__ __device__ static int units(int nx, int ny) { return ((nx + 1) >> 1) * ((ny + 1) >> 1); }
    __device__ void place(int hx, int rows, int t, int& I, int& j) {
        j = small_div(t, hx);
        I = t - j * hx;
        j *= 2;
        own = j < rows;
        q = xidx(hx, I, j);
    }
    template <bool ODD>
    __device__ void load(const BlkSrc<T, NR>& S, int I, int j, const BlkSides& n) {
        const int c0 = j * S.nx + 2 * I;
        using P2 = Vec<T, 2>;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int c = c0 + r * S.nx;
            if constexpr (ODD) {
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const bool in = 2 * I + e < S.nx && j + r < S.ny;
                    const int ce = in ? c + e : 0;
                    wl[r][e] = in ? S.wl[ce] : T(0);
                    wb[r][e] = in ? S.wb[ce] : T(0);
                    d[r][e] = in ? S.d[ce] : T(1);
                    const V bv = S.b[ce];
#pragma unroll
                    for (int k = 0; k < NR; ++k) b[r][e].v[k] = in ? bv.v[k] : T(0);
                }
                wl[r][2] = n.right && j + r < S.ny ? S.wl[c + 2] : T(0);
            } else {
                const P2 w = *reinterpret_cast<const P2*>(S.wl + c), v = *reinterpret_cast<const P2*>(S.wb + c);
                const P2 dv = *reinterpret_cast<const P2*>(S.d + c);
                const Vec<T, 2 * NR> bv = *reinterpret_cast<const Vec<T, 2 * NR>*>(S.b + c);
                const T wr = S.wl[c + 2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    wl[r][e] = w.v[e];
                    wb[r][e] = v.v[e];
                    d[r][e] = dv.v[e];
#pragma unroll
                    for (int k = 0; k < NR; ++k) b[r][e].v[k] = bv.v[e * NR + k];
                }
                wl[r][2] = n.right ? wr : T(0);
            }
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            if constexpr (ODD) {
                wb[2][e] = n.up && 2 * I + e < S.nx ? S.wb[c0 + 2 * S.nx + e] : T(0);
            } else {
                const T wt = S.wb[c0 + 2 * S.nx + e];
                wb[2][e] = n.up ? wt : T(0);
            }
        }
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int e = 0; e < 2; ++e)
                id[r][e] = rcp_diag(d[r][e] + wl[r][e] + wl[r][e + 1] + wb[r][e] + wb[r + 1][e]);
#pragma unroll
        for (int r = 0; r < 2; ++r) wl[r][0] = n.left ? wl[r][0] : T(0);
#pragma unroll
        for (int e = 0; e < 2; ++e) wb[0][e] = n.down ? wb[0][e] : T(0);
    }
    // the first colour-0 half-sweep from x = 0 reduces to x = b / (full diagonal)
    __device__ void first() {
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int k = 0; k < NR; ++k) {
                x[r][r].v[k] = b[r][r].v[k] * id[r][r];
                x[r][1 - r].v[k] = T(0);
            }
    }
    __device__ void zero() {
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int k = 0; k < NR; ++k) x[r][e].v[k] = T(0);
    }
    template <int COLOR>
    __device__ void put(V* xs, int hx) const {   // xs: the colour's array
        xs[q] = x[0][COLOR];
        xs[q + hx] = x[1][1 - COLOR];
    }
    template <int COLOR>
    __device__ void fetch(const V* xs, int hx) {
        x[0][COLOR] = xs[q];
        x[1][1 - COLOR] = xs[q + hx];
    }
    __device__ void add(const V& c) {
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int k = 0; k < NR; ++k) x[r][e].v[k] += c.v[k];
    }
    // the block's cells in the order of the finest post-smoothing's r.z: (row, column parity, left,
    // right, lower, upper weight, D, b, x)
    static constexpr int CELLS = 4;
    template <class F>
    __device__ __forceinline__ void cells(F&& f) {
        f(0, 0, 0, wl[0][0], wl[0][1], wb[0][0], wb[1][0], d[0][0], b[0][0], x[0][0]);
        f(1, 0, 1, wl[0][1], wl[0][2], wb[0][1], wb[1][1], d[0][1], b[0][1], x[0][1]);
        f(2, 1, 1, wl[1][1], wl[1][2], wb[1][1], wb[2][1], d[1][1], b[1][1], x[1][1]);
        f(3, 1, 0, wl[1][0], wl[1][1], wb[1][0], wb[2][0], d[1][0], b[1][0], x[1][0]);
    }
    template <int COLOR>
    __device__ const V& low() const { return x[0][COLOR]; }        // the colour's cell of the first row
    template <int COLOR>
    __device__ const V& high() const { return x[1][1 - COLOR]; }   // of the last row
    // the outer neighbours of the block's two cells of colour COLOR, (0, COLOR) and (1, 1 - COLOR)
    template <int COLOR>
    __device__ void outer(const V* xo, int hx, V& h0, V& v0, V& h1, V& v1) const {
        h0 = xo[q + (COLOR ? 1 : -1)];
        v0 = xo[q - hx];
        h1 = xo[q + hx + (COLOR ? -1 : 1)];
        v1 = xo[q + 2 * hx];
    }
    // (b + sum of w x_n) / diagonal of cell (r, e) with the outer neighbours h and v
    __device__ V update(int r, int e, const V& h, const V& v) const {
        V a;
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            const T xl = e == 1 ? x[r][0].v[k] : h.v[k], xr = e == 0 ? x[r][1].v[k] : h.v[k];
            const T xd = r == 1 ? x[0][e].v[k] : v.v[k], xu = r == 0 ? x[1][e].v[k] : v.v[k];
            a.v[k] = (b[r][e].v[k] + wl[r][e] * xl + wl[r][e + 1] * xr + wb[r][e] * xd + wb[r + 1][e] * xu) * id[r][e];
        }
        return a;
    }
    template <int COLOR>
    __device__ void sweep(const V* xo, int hx) {   // xo: the other colour's array
        V h0, v0, h1, v1;
        outer<COLOR>(xo, hx, h0, v0, h1, v1);
        const V a0 = update(0, COLOR, h0, v0), a1 = update(1, 1 - COLOR, h1, v1);
        x[0][COLOR] = a0;
        x[1][1 - COLOR] = a1;
    }
    // the four cells' residuals summed; TILE: in the form of the tile kernels
    template <bool TILE>
    __device__ V residual(const V* xs, int nxc, int hx) const {
        V h[2][2], v[2][2], acc;   // outer neighbours of cell (r, e)
        outer<0>(xs + nxc, hx, h[0][0], v[0][0], h[1][1], v[1][1]);
        outer<1>(xs, hx, h[0][1], v[0][1], h[1][0], v[1][0]);
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            T res[2][2];
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const T xl = e == 1 ? x[r][0].v[k] : h[r][e].v[k], xr = e == 0 ? x[r][1].v[k] : h[r][e].v[k];
                    const T xd = r == 1 ? x[0][e].v[k] : v[r][e].v[k], xu = r == 0 ? x[1][e].v[k] : v[r][e].v[k];
                    if constexpr (TILE)
                        res[r][e] = cell_residual(b[r][e].v[k], d[r][e], wl[r][e], wl[r][e + 1], wb[r][e], wb[r + 1][e],
                                                  x[r][e].v[k], xl, xr, xd, xu);
                    else
                        res[r][e] = small_residual<T, NR>(e, b[r][e].v[k], d[r][e], wl[r][e], wl[r][e + 1], wb[r][e],
                                                          wb[r + 1][e], x[r][e].v[k], xl, xr, xd, xu);
                }
            acc.v[k] = res[0][0] + res[0][1] + res[1][0] + res[1][1];
        }
        return acc;
    }
};

// A thread's cells in FP64: two neighbours of a row, columns 2I, 2I + 1 of row j, one of each colour
// (arrays by colour).  A dependent FP64 operation takes 64 cycles whatever the lanes do, and a
// scheduler's FP64 unit one warp instruction in that time: with one cell of a colour per thread a
// half-sweep is one chain of six operations instead of two behind each other, and the level
// spreads over twice the warps.  The restriction meets through shared memory.
template <typename T, int NR>
struct PairBlk {
    using V = Vec<T, NR>;
    static constexpr int RB = 1;
    V b[2], x[2];
    T id[2], d[2], wl[2], wr[2], wb[2], wt[2];
    int q;
    int par;      // j & 1: the cell of colour c is column 2I + (c ^ par)
    bool own;
    __host__ __device__ static int units(int nx, int ny) { return ((nx + 1) >> 1) * ny; }
    __device__ void place(int hx, int rows, int t, int& I, int& j) {
        j = small_div(t, hx);
        I = t - j * hx;
        own = j < rows;
        q = xidx(hx, I, j);
        par = j & 1;
    }
    template <bool ODD>
    __device__ void load(const BlkSrc<T, NR>& S, int I, int j, const BlkSides& n) {
        const int c = j * S.nx + 2 * I;
        const bool two = !ODD || 2 * I + 1 < S.nx;   // the second cell exists
        const T w0 = S.wl[c], w1 = two ? S.wl[c + 1] : T(0), w2 = n.right ? S.wl[c + 2] : T(0);
#pragma unroll
        for (int k = 0; k < 2; ++k) {                // colour k
            const int e = k ^ par;
            const bool in = e == 0 || two;
            const int ce = in ? c + e : c;
            wl[k] = e ? w1 : (n.left ? w0 : T(0));
            wr[k] = e ? w2 : w1;
            wb[k] = in && n.down ? S.wb[ce] : T(0);
            wt[k] = in && n.up ? S.wb[ce + S.nx] : T(0);
            d[k] = in ? S.d[ce] : T(1);
            id[k] = in ? S.id[ce] : T(1);
            const V bv = S.b[ce];
#pragma unroll
            for (int r = 0; r < NR; ++r) b[k].v[r] = in ? bv.v[r] : T(0);
        }
    }
    __device__ void first() {
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            x[0].v[k] = b[0].v[k] * id[0];
            x[1].v[k] = T(0);
        }
    }
    __device__ void zero() {
#pragma unroll
        for (int k = 0; k < NR; ++k) x[0].v[k] = x[1].v[k] = T(0);
    }
    template <int COLOR>
    __device__ void put(V* xs, int hx) const { xs[q] = x[COLOR]; }
    template <int COLOR>
    __device__ void fetch(const V* xs, int hx) { x[COLOR] = xs[q]; }
    __device__ void add(const V& c) {
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            x[0].v[k] += c.v[k];
            x[1].v[k] += c.v[k];
        }
    }
    static constexpr int CELLS = 2;
    template <class F>
    __device__ __forceinline__ void cells(F&& f) {
        f(0, 0, par, wl[0], wr[0], wb[0], wt[0], d[0], b[0], x[0]);
        f(1, 0, 1 - par, wl[1], wr[1], wb[1], wt[1], d[1], b[1], x[1]);
    }
    template <int COLOR>
    __device__ const V& low() const { return x[COLOR]; }
    template <int COLOR>
    __device__ const V& high() const { return x[COLOR]; }
    template <int COLOR>
    __device__ void sweep(const V* xo, int hx) {
        const bool e = (COLOR ^ par) != 0;
        const V h = xo[q + (e ? 1 : -1)], vd = xo[q - hx], vu = xo[q + hx];
        V a;
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            const T o = x[1 - COLOR].v[k], xl = e ? o : h.v[k], xr = e ? h.v[k] : o;
            a.v[k] = (b[COLOR].v[k] + wl[COLOR] * xl + wr[COLOR] * xr + wb[COLOR] * vd.v[k] + wt[COLOR] * vu.v[k]) *
                     id[COLOR];
        }
        x[COLOR] = a;
    }
    // the residuals of the cells in columns 2I and 2I + 1
    template <bool TILE>
    __device__ void residual(const V* xs, int nxc, int hx, V& r0, V& r1) const {
        V r[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const V* xo = xs + (1 - c) * nxc;
            const bool e = (c ^ par) != 0;
            const V h = xo[q + (e ? 1 : -1)], vd = xo[q - hx], vu = xo[q + hx];
#pragma unroll
            for (int k = 0; k < NR; ++k) {
                const T o = x[1 - c].v[k], xl = e ? o : h.v[k], xr = e ? h.v[k] : o;
                if constexpr (TILE)
                    r[c].v[k] = cell_residual(b[c].v[k], d[c], wl[c], wr[c], wb[c], wt[c], x[c].v[k], xl, xr, vd.v[k],
                                              vu.v[k]);
                else
                    r[c].v[k] = small_residual<T, NR>(e, b[c].v[k], d[c], wl[c], wr[c], wb[c], wt[c], x[c].v[k], xl, xr,
                                                      vd.v[k], vu.v[k]);
            }
        }
        r0 = par ? r[1] : r[0];
        r1 = par ? r[0] : r[1];
    }
};
template <typename T, int NR>
using Blk = std::conditional_t<sizeof(T) == 8, PairBlk<T, NR>, QuadBlk<T, NR>>;

// the restricted residual of K blocks per thread: put(u, value) for each complete coarse cell; s: an
// entry per coarse cell of the team's rows (one of s's barriers between the two rows of a cell
// in FP64), slot(u) the block's
template <typename T, int NR, int K, bool TILE, class Put, class Sync>
__device__ inline void blk_restrict(const Blk<T, NR> (&B)[K], const int (&slot)[K], Vec<T, NR>* s, const Vec<T, NR>* x,
                                    int nxc, int hx, Put&& put, Sync&& sync) {
    if constexpr (Blk<T, NR>::RB == 2) {
#pragma unroll
        for (int u = 0; u < K; ++u)
            if (B[u].own) put(u, B[u].template residual<TILE>(x, nxc, hx));
    } else {
        Vec<T, NR> r0[K], r1[K];
#pragma unroll
        for (int u = 0; u < K; ++u)
            if (B[u].own) {
                B[u].template residual<TILE>(x, nxc, hx, r0[u], r1[u]);
                if (!B[u].par) {
                    Vec<T, NR> a;
#pragma unroll
                    for (int k = 0; k < NR; ++k) a.v[k] = r0[u].v[k] + r1[u].v[k];
                    s[slot[u]] = a;
                }
            }
        sync();
#pragma unroll
        for (int u = 0; u < K; ++u)
            if (B[u].own && B[u].par) {
                Vec<T, NR> a = s[slot[u]];
#pragma unroll
                for (int k = 0; k < NR; ++k) a.v[k] = a.v[k] + r0[u].v[k] + r1[u].v[k];
                put(u, a);
            }
    }
}

// the team of a level: the first `threads` threads of the block (a multiple of 32)
template <typename T>
__device__ inline int small_team(int nx, int ny) {
    const int n = Blk<T, 1>::units(nx, ny), cap = blockDim.x;
    return n >= cap ? cap : (n + 31) & ~31;
}

// the blocks of a thread on single-block level l
template <typename T, int NR, int K, bool ODD>
__device__ inline void small_blocks(Blk<T, NR> (&B)[K], int (&I)[K], int (&j)[K], const SmallPlan& P, int l,
                                    const SmallMem<T, NR>& M, int team) {
    const int o = P.soff[l], nx = P.nx[l], ny = P.ny[l], hx = (nx + 1) >> 1;
    const BlkSrc<T, NR> S = {nx, ny, M.d + o, M.wl + o, M.wb + o, M.id + o, M.b + o};
#pragma unroll
    for (int u = 0; u < K; ++u) {
        B[u].place(hx, ny, threadIdx.x + u * team, I[u], j[u]);
        if (B[u].own)
            B[u].template load<ODD>(S, I[u], j[u],
                                    {I[u] > 0, 2 * I[u] + 2 < nx, j[u] > 0, j[u] + Blk<T, NR>::RB < ny});
    }
}
// one red-black half-sweep of colour COLOR over the K blocks of a thread (x: nxc entries per colour)
template <typename T, int NR, int K, int COLOR>
__device__ inline void small_sweep(Blk<T, NR> (&B)[K], Vec<T, NR>* x, int nxc, int hx, int l, int team) {
#pragma unroll
    for (int u = 0; u < K; ++u)
        if (B[u].own) {
            B[u].template sweep<COLOR>(x + (1 - COLOR) * nxc, hx);
            B[u].template put<COLOR>(x + COLOR * nxc, hx);
        }
    team_sync(l, team);
}

// down leg of level l from x = 0, then the residual restricted to level l + 1
template <typename T, int NR, int K>
__device__ inline void small_down(const SmallPlan& P, int l, SmallMem<T, NR>& M, int team) {
    static_assert(NU_SMALL == 2, "the sweep sequences below are written out for two pairs");
    const int hx = P.nx[l] >> 1, nxc = x_entries(hx, P.ny[l]);
    Vec<T, NR>* x = M.x + P.xoff[l];
    Blk<T, NR> B[K];
    int I[K], j[K];
    small_blocks<T, NR, K, false>(B, I, j, P, l, M, team);
#pragma unroll
    for (int u = 0; u < K; ++u)
        if (B[u].own) {
            B[u].first();
            B[u].template put<0>(x, hx);
        }
    team_sync(l, team);
    small_sweep<T, NR, K, 1>(B, x, nxc, hx, l, team);
    small_sweep<T, NR, K, 0>(B, x, nxc, hx, l, team);
    small_sweep<T, NR, K, 1>(B, x, nxc, hx, l, team);
    Vec<T, NR>* bc = M.b + P.soff[l + 1];
    int slot[K];
#pragma unroll
    for (int u = 0; u < K; ++u) slot[u] = (j[u] >> 1) * hx + I[u];
    blk_restrict<T, NR, K, false>(
        B, slot, bc, x, nxc, hx, [&](int u, const Vec<T, NR>& v) { bc[slot[u]] = v; }, [&]() { team_sync(l, team); });
    team_sync(l, team);
}

// coarsest level: exact solve with the precomputed inverse (up to 32 cells), else a symmetric
// red-black sweep sequence from zero
template <typename T, int NR, int K>
__device__ inline void small_coarsest(const SmallPlan& P, SmallMem<T, NR>& M, bool exact) {
    const int l = P.n - 1, o = P.soff[l], nx = P.nx[l], ny = P.ny[l], n = nx * ny;
    const int hx = (nx + 1) >> 1, nxc = x_entries(hx, (ny + 1) & ~1);
    Vec<T, NR>* x = M.x + P.xoff[l];
    const int team = exact ? 32 : small_team<T>(nx, ny);
    if (threadIdx.x >= team) return;
    if (exact) {
        const int r = threadIdx.x;
        if (r < n) {
            Vec<T, NR> acc;
#pragma unroll
            for (int k = 0; k < NR; ++k) acc.v[k] = T(0);
#pragma unroll 8
            for (int c = 0; c < n; ++c) {
                const T a = M.inv[c * n + r];
                const Vec<T, NR> bv = M.b[o + c];
#pragma unroll
                for (int k = 0; k < NR; ++k) acc.v[k] += a * bv.v[k];
            }
            const int j = small_div(r, nx), i = r - j * nx;
            x[((i + j) & 1) * nxc + xidx(hx, i >> 1, j)] = acc;
        }
        return;
    }
    // (x is zero from the start in a single cycle, not in the later ones of a kernel that runs several)
    Blk<T, NR> B[K];
    int I[K], j[K];
    small_blocks<T, NR, K, true>(B, I, j, P, l, M, team);
#pragma unroll
    for (int u = 0; u < K; ++u)
        if (B[u].own) {
            B[u].zero();
            B[u].template put<0>(x, hx);
            B[u].template put<1>(x + nxc, hx);
        }
    team_sync(l, team);
    for (int k = 0; k < COARSE_PAIRS; ++k) {
        small_sweep<T, NR, K, 0>(B, x, nxc, hx, l, team);
        small_sweep<T, NR, K, 1>(B, x, nxc, hx, l, team);
    }
    for (int k = 0; k < COARSE_PAIRS; ++k) {
        small_sweep<T, NR, K, 1>(B, x, nxc, hx, l, team);
        small_sweep<T, NR, K, 0>(B, x, nxc, hx, l, team);
    }
}

// up leg of level l: x += P x_{l+1}, then the post-smoothing half-sweeps.  The opening barrier
// joins the level's team with the warps that worked on the coarser levels.
template <typename T, int NR, int K>
__device__ inline void small_up(const SmallPlan& P, int l, SmallMem<T, NR>& M, int team) {
    const int hx = P.nx[l] >> 1, nxc = x_entries(hx, P.ny[l]);
    const int chx = (P.nx[l + 1] + 1) >> 1, cnxc = x_entries(chx, (P.ny[l + 1] + 1) & ~1);
    Vec<T, NR>* x = M.x + P.xoff[l];
    const Vec<T, NR>* xc = M.x + P.xoff[l + 1];
    Blk<T, NR> B[K];
    int I[K], j[K];
    small_blocks<T, NR, K, false>(B, I, j, P, l, M, team);
#pragma unroll
    for (int u = 0; u < K; ++u)
        if (B[u].own) {
            B[u].template fetch<0>(x, hx);
            B[u].template fetch<1>(x + nxc, hx);
        }
    team_sync(l, team);
#pragma unroll
    for (int u = 0; u < K; ++u) {
        if (!B[u].own) continue;
        const int J = j[u] >> 1;
        B[u].add(xc[((I[u] + J) & 1) * cnxc + xidx(chx, I[u] >> 1, J)]);
        B[u].template put<0>(x, hx);
        B[u].template put<1>(x + nxc, hx);
    }
    team_sync(l, team);
    small_sweep<T, NR, K, 1>(B, x, nxc, hx, l, team);
    small_sweep<T, NR, K, 0>(B, x, nxc, hx, l, team);
    small_sweep<T, NR, K, 1>(B, x, nxc, hx, l, team);
    small_sweep<T, NR, K, 0>(B, x, nxc, hx, l, team);
}

// the cycle on levels whose operators and level-0 right-hand side are in shared memory: every
// level's down leg on its team, the coarsest solve, the up legs.  A warp leaves at the first level
// it owns no cells of and waits for the others at the up leg of the level before.  BIG: the first
// level may have more blocks than the team has threads (two per thread).
// CALL: the legs as calls of their own (inlined into a kernel of many phases they spill).
template <typename T, int NR>
__device__ __noinline__ void small_down_call(const SmallPlan& P, int l, SmallMem<T, NR>& M, int team) {
    small_down<T, NR, 1>(P, l, M, team);
}
template <typename T, int NR, int K>
__device__ __noinline__ void small_coarsest_call(const SmallPlan& P, SmallMem<T, NR>& M, bool exact) {
    small_coarsest<T, NR, K>(P, M, exact);
}
template <typename T, int NR>
__device__ __noinline__ void small_up_call(const SmallPlan& P, int l, SmallMem<T, NR>& M, int team) {
    small_up<T, NR, 1>(P, l, M, team);
}
template <typename T, int NR, bool BIG, bool CALL = false>
__device__ inline void small_core(const SmallPlan& P, SmallMem<T, NR>& M, bool exact) {
    const int tid = threadIdx.x;
    int lmax = 0;   // levels [0, lmax) with this thread in the team
    while (lmax < P.n - 1 && tid < small_team<T>(P.nx[lmax], P.ny[lmax])) ++lmax;
    const bool two = BIG && Blk<T, NR>::units(P.nx[0], P.ny[0]) > (int)blockDim.x;   // level 0: two blocks per thread
    for (int l = 0; l < lmax; ++l) {
        const int team = small_team<T>(P.nx[l], P.ny[l]);
        bool done = false;
        if constexpr (BIG)
            if (l == 0 && two) {
                small_down<T, NR, 2>(P, l, M, team);
                done = true;
            }
        if constexpr (CALL) small_down_call<T, NR>(P, l, M, team);
        else if (!done) small_down<T, NR, 1>(P, l, M, team);
    }
    if (lmax == P.n - 1) {
        // up to 1024 cells: blocks of four one per thread, pairs one or two
        const bool pair2 = sizeof(T) == 8 && Blk<T, NR>::units(P.nx[P.n - 1], P.ny[P.n - 1]) > (int)blockDim.x;
        if constexpr (CALL) {
            if (!pair2) small_coarsest_call<T, NR, 1>(P, M, exact);
            else if constexpr (sizeof(T) == 8) small_coarsest_call<T, NR, 2>(P, M, exact);
        } else {
            if (!pair2) small_coarsest<T, NR, 1>(P, M, exact);
            else if constexpr (sizeof(T) == 8) small_coarsest<T, NR, 2>(P, M, exact);
        }
        if (tid < 32) __syncwarp();
    }
    for (int l = lmax - 1; l >= 0; --l) {
        const int team = small_team<T>(P.nx[l], P.ny[l]);
        bool done = false;
        if constexpr (BIG)
            if (l == 0 && two) {
                small_up<T, NR, 2>(P, l, M, team);
                done = true;
            }
        if constexpr (CALL) small_up_call<T, NR>(P, l, M, team);
        else if (!done) small_up<T, NR, 1>(P, l, M, team);
    }
    __syncthreads();
}

// the small levels' operators into shared memory (asynchronous copies: the caller waits and meets
// at a block barrier), x zeroed; true if the coarsest level has its inverse
template <typename T, int NR>
__device__ inline bool small_operators(const SmallPlan& P, SmallMem<T, NR>& M, const T* diag, const T* id, const T* wl,
                                       const T* wb, const T* inv) {
    const size_t g = P.goff[0];
    const int n = P.nx[P.n - 1] * P.ny[P.n - 1];
    const bool try_inv = n <= 32;
    copy_async(M.d, diag + g, P.cells);
    copy_async(M.wl, wl + g, P.cells);
    copy_async(M.wb, wb + g, P.cells);
    if (sizeof(T) == 8) copy_async(M.id, id + g, P.cells);
    // the inverse is copied whether usable or not, beside the word that says so
    T usable = T(0), v[2] = {T(0), T(0)};
    if (try_inv) {
        usable = inv[n * n];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int c = threadIdx.x + u * blockDim.x;
            if (c < n * n) v[u] = inv[c];
        }
    }
    for (int c = threadIdx.x; c < P.xtotal; c += blockDim.x) {
        Vec<T, NR> z;
#pragma unroll
        for (int k = 0; k < NR; ++k) z.v[k] = T(0);
        M.x[c] = z;
    }
    if (try_inv)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int c = threadIdx.x + u * blockDim.x;
            if (c < n * n) {
                const int r = small_div(c, n);
                M.inv[(c - r * n) * n + r] = v[u];
            }
        }
    if (try_inv)
        for (int c = threadIdx.x + 2 * blockDim.x; c < n * n; c += blockDim.x) M.inv[(c % n) * n + c / n] = inv[c];
    return try_inv && usable == T(1);
}

// the V-cycle on the small levels in one block of SMALL_THREADS threads, from the level-(first
// small) rhs b_in to its correction x_out; with DOT (the cycle starts at the finest level) also
// r.z -> beta
template <typename T, int NR, bool DOT>
__device__ void small_cycle(const SmallPlan& P, const T* __restrict__ diag, const T* __restrict__ id,
                            const T* __restrict__ wl, const T* __restrict__ wb, const T* __restrict__ inv, const T* __restrict__ b_in,
                            T* __restrict__ x_out, SolveState* st, unsigned char* smem) {
    SmallMem<T, NR> M(smem, P);
    const int n0 = P.nx[0] * P.ny[0];
    // the small levels are contiguous in the packed level arrays and in shared memory: one flat
    // asynchronous copy per array, all in flight together
    copy_async((T*)M.b, b_in, n0 * NR);
    const bool exact = small_operators<T, NR>(P, M, diag, id, wl, wb, inv);
    cp_async_wait_all();
    __syncthreads();
    small_core<T, NR, sizeof(T) == 4>(P, M, exact);
    const int nx0 = P.nx[0], hx0 = (nx0 + 1) >> 1, nxc0 = x_entries(hx0, (P.ny[0] + 1) & ~1);
    const Vec<T, NR>* x0 = M.x + P.xoff[0];
    auto xat = [&](int c) {
        const int j = small_div(c, nx0), i = c - j * nx0;
        return x0[((i + j) & 1) * nxc0 + xidx(hx0, i >> 1, j)];
    };
    for (int c = threadIdx.x; c < n0; c += blockDim.x) reinterpret_cast<Vec<T, NR>*>(x_out)[c] = xat(c);
    if (DOT) {
        // the cycle started at the finest level: r.z -> beta, summed as by 1024 threads (virtual
        // thread t takes the cells t, t + 1024, ...; 32 warp sums, then their sum)
        __shared__ double sh[32];
#pragma unroll
        for (int k = 0; k < NR; ++k) {
#pragma unroll
            for (int h = 0; h < 1024 / SMALL_THREADS; ++h) {
                double a = 0.0;
                for (int c = h * SMALL_THREADS + threadIdx.x; c < n0; c += 1024)
                    a += (double)xat(c).v[k] * (double)M.b[c].v[k];
                for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
                if ((threadIdx.x & 31) == 0) sh[(h * SMALL_THREADS + threadIdx.x) >> 5] = a;
            }
            __syncthreads();
            if (threadIdx.x < 32) {
                double a = sh[threadIdx.x];
                for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
                if (threadIdx.x == 0) {
                    double old = st->rz[k];
                    st->beta[k] = old != 0.0 ? a / old : 0.0;
                    st->rz[k] = a;
                }
            }
            __syncthreads();
        }
    }
}

template <typename T, int NR, bool DOT>
__global__ void __launch_bounds__(SMALL_THREADS) k_small(SmallPlan P, const T* __restrict__ diag,
                                                         const T* __restrict__ id, const T* __restrict__ wl, const T* __restrict__ wb,
                                                         const T* __restrict__ inv, const T* __restrict__ b_in,
                                                         T* __restrict__ x_out, SolveState* st) {
    const long long zo = zoff(P.zs);
    diag = zsh(diag, zo);
    id = zsh(id, zo);
    wl = zsh(wl, zo);
    wb = zsh(wb, zo);
    inv = zsh(inv, zo);
    b_in = zsh(b_in, zo);
    x_out = zsh(x_out, zo);
    st = zsh(st, zo);
    if (skip(st)) return;
    extern __shared__ __align__(128) unsigned char smem[];
    small_cycle<T, NR, DOT>(P, diag, id, wl, wb, inv, b_in, x_out, st, smem);
}


// ---- the coarse part of the V-cycle in one cooperative launch -----------------------------
// Tiled levels with few tiles are latency-bound: each launch costs more than its work.  The
// tiled levels [l0, nb) and the single-block levels run in one cooperative launch whose blocks
// take the tiles of a level in turn and meet at a grid barrier between the phases:
// pre-smoothing down the levels, the single-block cycle (block 0), post-smoothing up.
template <typename T>
struct CoarsePlan {
    int l0, nb;                      // levels handled: tiled [l0, nb), then the single-block ones
    int spin;                        // polls of a grid barrier before it gives up (fault bit 1)
    Lev<T> L[Solver::MAXLEV];
    const T* b[Solver::MAXLEV];      // rhs of level l
    T* x2[Solver::MAXLEV];           // pre-smoothed x of level l
    T* bc[Solver::MAXLEV];           // rhs of level l + 1 (written by the pre phase of level l)
    T* xo[Solver::MAXLEV];           // final x of level l
    const T* xc[Solver::MAXLEV];     // x of level l + 1 (read by the post phase of level l)
};
constexpr int CC_THREADS = SMALL_THREADS;

// grid-wide barrier of a cooperative launch (all blocks resident).  bar[0] counts arrivals and
// only grows during a launch (the level-0 pre-smoothing kernel, which precedes every launch,
// zeroes it): barrier k of the launch is passed once it reaches k x (number of blocks).  One
// release reduction per block (it publishes the writes the block's threads made before the
// block barrier) and acquire loads while waiting (the writes of the other blocks are visible to
// this block's threads after the closing block barrier); the wait is bounded and a timeout is
// recorded in st->fault.
__device__ inline unsigned ld_acquire_gpu(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ inline void red_release_gpu_add(unsigned* p, unsigned v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ inline void grid_sync(unsigned* bar, unsigned& target, SolveState* st, int spin) {
    target += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) {
        red_release_gpu_add(&bar[0], 1u);
        for (int it = 0; (int)(ld_acquire_gpu(&bar[0]) - target) < 0; ++it)
            if (it > spin) {
                atomicOr(&st->fault, 2);
                break;
            }
    }
    __syncthreads();
}

template <typename T, int NR>
__global__ void __launch_bounds__(CC_THREADS) k_coarse_cycle(CoarsePlan<T> C, SmallPlan P, const T* __restrict__ diag,
                                                             const T* __restrict__ id, const T* __restrict__ wl, const T* __restrict__ wb,
                                                             const T* __restrict__ inv, SolveState* st,
                                                             unsigned* bar) {
    if (skip(st)) return;   // written by an earlier launch: the same for every block
    extern __shared__ __align__(128) unsigned char smem[];
    unsigned gen = 0;   // arrivals that pass the next barrier (bar[0] starts the launch at 0)
    const TileThread tpre = tile_thread<HPRE>(), tpost = tile_thread<HPOST>();
    for (int l = C.l0; l < C.nb; ++l) {
        const Lev<T>& L = C.L[l];
        int tx = (L.nx + TX - 1) / TX, nt = tx * ((L.ny + TY - 1) / TY);
        for (int t = blockIdx.x; t < nt; t += gridDim.x) {
            pre_tile<T, NR>(L, C.b[l], C.x2[l], C.bc[l], t % tx, t / tx, smem, nullptr, tpre);
            __syncthreads();
        }
        grid_sync(bar, gen, st, C.spin);
    }
    if (blockIdx.x == 0) small_cycle<T, NR, false>(P, diag, id, wl, wb, inv, C.bc[C.nb - 1], C.xo[C.nb], st, smem);
    grid_sync(bar, gen, st, C.spin);
    for (int l = C.nb - 1; l >= C.l0; --l) {
        const Lev<T>& L = C.L[l];
        int tx = (L.nx + TX - 1) / TX, nt = tx * ((L.ny + TY - 1) / TY);
        for (int t = blockIdx.x; t < nt; t += gridDim.x) {
            post_tile<T, NR, false>(L, C.b[l], C.x2[l], C.xo[l], C.xc[l], t % tx, t / tx, smem, nullptr, tpost);
            __syncthreads();
        }
        if (l > C.l0) grid_sync(bar, gen, st, C.spin);
    }
}

// ---- the coarse part of the V-cycle in one thread-block cluster ----------------------------
// The coarse levels of a single instance are latency-bound: in the grid-barrier launch above a
// phase costs 2 to 3 us (load a tile from L2, sweep, store) and a barrier 0.9 to 1.4 us.  Here one
// cluster of up to 16 blocks (16 SMs) keeps the levels [l0, nb) in its shared memory: block k of
// the cluster owns rows [k rp, (k + 1) rp) of a level (rp even), thread t of it 2 x 2 blocks of
// cells as in the single-block levels.  After a half-sweep of one colour the edge rows' new
// values are stored into the neighbour blocks' halo rows through distributed shared memory, and
// a cluster barrier (0.2 us; store, barrier and read of a pushed value 0.3 to 0.4 us) ends the
// phase.  Operators are copied from global memory once per launch, the levels exchange their
// right-hand sides and corrections through distributed shared memory, and block 0 runs the
// single-block levels.  The arithmetic of every cell is that of the tile kernels.
// Measured per launch against the grid-barrier launch or the separate ones (one right-hand side):
// FP32 on a 128^2 grid 17.6 -> 12.8 us, on 512^2 31.2 -> 26 (28 with cold caches; its 256^2 level costs
// what two separate launches do); FP64 from the 128^2 level down 80 -> 46 us.  A 64^2 level of four rows per block
// spends about 1000 cycles a phase, 750 of them push and barrier.
constexpr int CL_MAX = 6;            // levels kept by the cluster, at most
constexpr int CL_BLOCKS = 16;        // blocks of the cluster (16 needs the non-portable attribute)
constexpr int CL_THREADS = 512;      // threads per block, at most (the registers are budgeted for it)
struct ClPlan {
    int nl;                          // levels kept by the cluster
    int nt;                          // of these, the first nt are tiled levels of the separate launches
    int nx[CL_MAX], ny[CL_MAX], rp[CL_MAX];
    int off[CL_MAX];                 // byte offset of the level's arrays in every block's shared memory
    size_t goff[CL_MAX];             // cell offset in the packed level arrays
    SmallPlan S;                     // the single-block levels, at byte offset soff of block 0
    int soff;
};

__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// the same shared-memory object in block `rank` of the cluster (a generic address)
template <class P>
__device__ __forceinline__ P* cluster_map(P* p, unsigned rank) {
    unsigned long long r;
    asm("mapa.u64 %0, %1, %2;" : "=l"(r) : "l"((unsigned long long)(uintptr_t)p), "r"(rank));
    return reinterpret_cast<P*>((uintptr_t)r);
}
// a level's arrays in a block's shared memory: x (rows -1 .. rp, as on the single-block levels),
// b, (FP64) the restriction's partial sums, then D, wl, (FP64) the reciprocal diagonals, wb (one row
// more)
template <typename T, int NR>
struct ClMem {
    static constexpr bool F64 = sizeof(T) == 8;
    Vec<T, NR>*x, *b, *s;
    T *d, *wl, *wb, *id;
    __host__ __device__ static int xn(int nx, int rp) { return (2 * x_entries(nx >> 1, rp) + 3) & ~3; }
    __host__ __device__ static int sn(int nx, int rp) { return F64 ? (rp * nx / 4 + 3) & ~3 : 0; }
    __device__ ClMem(unsigned char* base, int nx, int rp) {
        x = (Vec<T, NR>*)base;
        b = x + xn(nx, rp);
        s = b + rp * nx;
        d = (T*)(s + sn(nx, rp));
        wl = d + rp * nx;
        id = wl + rp * nx;
        wb = id + (F64 ? rp * nx : 0);
    }
    static int bytes(int nx, int rp) {
        size_t v = (size_t)(xn(nx, rp) + rp * nx + sn(nx, rp)) * NR, c = (size_t)(3 * rp + 1) * nx + (F64 ? rp * nx : 0);
        return (int)(((v + c + 2) * sizeof(T) + 127) & ~size_t(127));
    }
};
// a block's slab of a level
struct ClSlab {
    int nx, hx, rp, j0, j1, nxc;     // rows [j0, j1); nxc entries per colour of x
    __device__ ClSlab(const ClPlan& P, int l, int rank) {
        nx = P.nx[l];
        hx = nx >> 1;
        rp = P.rp[l];
        j0 = min(rank * rp, P.ny[l]);
        j1 = min(j0 + rp, P.ny[l]);
        nxc = x_entries(hx, rp);
    }
};
// edge of a slab that a block of cells lies on (its new values are pushed there)
constexpr unsigned CL_DOWN = 1, CL_UP = 2;

// the blocks of a thread on level l of the cluster
template <typename T, int NR, int K>
__device__ inline void cl_blocks(Blk<T, NR> (&B)[K], unsigned (&edge)[K], int (&I)[K], int (&j)[K], const ClSlab& S,
                                 int ny, const ClMem<T, NR>& M) {
    const BlkSrc<T, NR> src = {S.nx, S.j1 - S.j0, M.d, M.wl, M.wb, M.id, M.b};
#pragma unroll
    for (int u = 0; u < K; ++u) {
        B[u].place(S.hx, S.j1 - S.j0, threadIdx.x + u * blockDim.x, I[u], j[u]);
        edge[u] = 0;
        if (!B[u].own) continue;
        // the rows below and above are halo rows (zero beyond the grid)
        B[u].template load<false>(src, I[u], j[u],
                                  {I[u] > 0, I[u] + 1 < S.hx, S.j0 + j[u] > 0, S.j0 + j[u] + Blk<T, NR>::RB < ny});
        edge[u] = (j[u] == 0 && S.j0 > 0 ? CL_DOWN : 0u) |
                  (S.j0 + j[u] + Blk<T, NR>::RB == S.j1 && S.j1 < ny ? CL_UP : 0u);
    }
}
// the new values of colour COLOR in the block's edge rows, into the neighbour slabs' halo rows
template <typename T, int NR, int COLOR>
__device__ __forceinline__ void cl_push(const Blk<T, NR>& B, unsigned edge, int I, const ClSlab& S, Vec<T, NR>* xdn,
                                        Vec<T, NR>* xup) {
    if (edge & CL_DOWN) xdn[COLOR * S.nxc + xidx(S.hx, I, S.rp)] = B.template low<COLOR>();
    if (edge & CL_UP) xup[COLOR * S.nxc + xidx(S.hx, I, -1)] = B.template high<COLOR>();
}
template <typename T, int NR, int K, int COLOR, bool LAST = false>
__device__ inline void cl_sweep(Blk<T, NR> (&B)[K], const unsigned (&edge)[K], const int (&I)[K], const ClSlab& S,
                                Vec<T, NR>* x, Vec<T, NR>* xdn, Vec<T, NR>* xup) {
#pragma unroll
    for (int u = 0; u < K; ++u) {
        if (!B[u].own) continue;
        B[u].template sweep<COLOR>(x + (1 - COLOR) * S.nxc, S.hx);
        if (!LAST) {
            B[u].template put<COLOR>(x + COLOR * S.nxc, S.hx);
            if (edge[u]) cl_push<T, NR, COLOR>(B[u], edge[u], I[u], S, xdn, xup);
        }
    }
    if (!LAST) cluster_barrier();
}

// down leg; TILE: the residual as in the tile kernels, else as on the single-block levels
template <typename T, int NR, int K, bool TILE>
__device__ inline void cl_down(const ClPlan& P, int l, int rank, unsigned char* smem) {
    const ClSlab S(P, l, rank);
    const ClMem<T, NR> M(smem + P.off[l], S.nx, S.rp);
    Vec<T, NR>* xdn = cluster_map(M.x, rank > 0 ? rank - 1 : 0);
    Vec<T, NR>* xup = cluster_map(M.x, rank + 1 < CL_BLOCKS ? rank + 1 : rank);
    Blk<T, NR> B[K];
    unsigned edge[K];
    int I[K], j[K];
    cl_blocks<T, NR, K>(B, edge, I, j, S, P.ny[l], M);
#pragma unroll
    for (int u = 0; u < K; ++u) {
        if (!B[u].own) continue;
        B[u].first();
        B[u].template put<0>(M.x, S.hx);
        if (edge[u]) cl_push<T, NR, 0>(B[u], edge[u], I[u], S, xdn, xup);
    }
    cluster_barrier();
    cl_sweep<T, NR, K, 1>(B, edge, I, S, M.x, xdn, xup);
    cl_sweep<T, NR, K, 0>(B, edge, I, S, M.x, xdn, xup);
    cl_sweep<T, NR, K, 1>(B, edge, I, S, M.x, xdn, xup);
    // the restricted residual into the right-hand side of the next level, in the shared memory of
    // the block that owns that cell
    int slot[K];
#pragma unroll
    for (int u = 0; u < K; ++u) slot[u] = (j[u] >> 1) * S.hx + I[u];
    blk_restrict<T, NR, K, TILE>(
        B, slot, M.s, M.x, S.nxc, S.hx,
        [&](int u, const Vec<T, NR>& v) {
            const int J = (S.j0 + j[u]) >> 1;
            if (l + 1 < P.nl) {
                const int own = small_div(J, P.rp[l + 1]);
                const ClMem<T, NR> N(smem + P.off[l + 1], P.nx[l + 1], P.rp[l + 1]);
                cluster_map(N.b, own)[(J - own * P.rp[l + 1]) * P.nx[l + 1] + I[u]] = v;
            } else {
                const SmallMem<T, NR> N(smem + P.soff, P.S);
                cluster_map(N.b, 0)[J * P.S.nx[0] + I[u]] = v;
            }
        },
        [&]() { __syncthreads(); });
    cluster_barrier();
}

// up leg on the blocks B of the thread (their x is the result); the last half-sweep of the first
// kept level (TOP) stays in the registers
template <typename T, int NR, int K, bool TOP>
__device__ inline void cl_up_blocks(Blk<T, NR> (&B)[K], unsigned (&edge)[K], int (&I)[K], int (&j)[K], const ClSlab& S,
                                    const ClMem<T, NR>& M, const ClPlan& P, int l, int rank, unsigned char* smem) {
    Vec<T, NR>* xdn = cluster_map(M.x, rank > 0 ? rank - 1 : 0);
    Vec<T, NR>* xup = cluster_map(M.x, rank + 1 < CL_BLOCKS ? rank + 1 : rank);
    cl_blocks<T, NR, K>(B, edge, I, j, S, P.ny[l], M);
#pragma unroll
    for (int u = 0; u < K; ++u) {
        if (!B[u].own) continue;
        const int J = (S.j0 + j[u]) >> 1;
        Vec<T, NR> cv;
        if (l + 1 < P.nl) {
            const int own = small_div(J, P.rp[l + 1]), chx = P.nx[l + 1] >> 1, cnxc = x_entries(chx, P.rp[l + 1]);
            const ClMem<T, NR> N(smem + P.off[l + 1], P.nx[l + 1], P.rp[l + 1]);
            cv = cluster_map(N.x, own)[((I[u] + J) & 1) * cnxc + xidx(chx, I[u] >> 1, J - own * P.rp[l + 1])];
        } else {
            const int chx = (P.S.nx[0] + 1) >> 1, cnxc = x_entries(chx, (P.S.ny[0] + 1) & ~1);
            const SmallMem<T, NR> N(smem + P.soff, P.S);
            cv = cluster_map(N.x, 0)[P.S.xoff[0] + ((I[u] + J) & 1) * cnxc + xidx(chx, I[u] >> 1, J)];
        }
        B[u].template fetch<0>(M.x, S.hx);
        B[u].template fetch<1>(M.x + S.nxc, S.hx);
        B[u].add(cv);
        B[u].template put<0>(M.x, S.hx);
        B[u].template put<1>(M.x + S.nxc, S.hx);
        if (edge[u]) cl_push<T, NR, 0>(B[u], edge[u], I[u], S, xdn, xup);
    }
    cluster_barrier();
    cl_sweep<T, NR, K, 1>(B, edge, I, S, M.x, xdn, xup);
    cl_sweep<T, NR, K, 0>(B, edge, I, S, M.x, xdn, xup);
    cl_sweep<T, NR, K, 1>(B, edge, I, S, M.x, xdn, xup);
    cl_sweep<T, NR, K, 0, TOP>(B, edge, I, S, M.x, xdn, xup);
}
// up leg; the result of the first kept level (TOP) goes to x_out, the others' stay in shared memory
template <typename T, int NR, int K, bool TOP>
__device__ inline void cl_up(const ClPlan& P, int l, int rank, unsigned char* smem, T* __restrict__ x_out) {
    const ClSlab S(P, l, rank);
    const ClMem<T, NR> M(smem + P.off[l], S.nx, S.rp);
    Blk<T, NR> B[K];
    unsigned edge[K];
    int I[K], j[K];
    cl_up_blocks<T, NR, K, TOP>(B, edge, I, j, S, M, P, l, rank, smem);
    if (TOP) {
#pragma unroll
        for (int u = 0; u < K; ++u) {
            if (!B[u].own) continue;
#pragma unroll
            for (int r = 0; r < Blk<T, NR>::RB; ++r) {
                Vec<T, 2 * NR> o;   // columns 2I, 2I + 1 of row j + r
#pragma unroll
                for (int k = 0; k < NR; ++k) {
                    if constexpr (Blk<T, NR>::RB == 2) {
                        o.v[k] = B[u].x[r][0].v[k];
                        o.v[NR + k] = B[u].x[r][1].v[k];
                    } else {
                        o.v[k] = B[u].par ? B[u].x[1].v[k] : B[u].x[0].v[k];
                        o.v[NR + k] = B[u].par ? B[u].x[0].v[k] : B[u].x[1].v[k];
                    }
                }
                reinterpret_cast<Vec<T, 2 * NR>*>(x_out)[(size_t)(S.j0 + j[u] + r) * S.hx + I[u]] = o;
            }
        }
    }
}

// the cluster's levels into shared memory: operators and the first level's right-hand side, all
// copies in flight at once (the caller waits and meets at a cluster barrier), x zeroed; block 0
// also the single-block levels (true if their coarsest one has its inverse)
template <typename T, int NR>
__device__ inline bool cl_operators(const ClPlan& P, int rank, unsigned char* smem, const T* diag, const T* id,
                                    const T* wl, const T* wb, const T* inv, const T* b_in) {
    for (int l = 0; l < P.nl; ++l) {
        const ClSlab S(P, l, rank);
        const ClMem<T, NR> M(smem + P.off[l], S.nx, S.rp);
        const int nr = S.j1 - S.j0, n = nr * S.nx;
        const size_t g = P.goff[l] + (size_t)S.j0 * S.nx;
        const int nwb = nr > 0 && S.j1 < P.ny[l] ? n + S.nx : n;
        copy_async(M.d, diag + g, n);
        copy_async(M.wl, wl + g, n);
        copy_async(M.wb, wb + g, nwb);
        if (sizeof(T) == 8) copy_async(M.id, id + g, n);
        if (l == 0) copy_async((T*)M.b, b_in + (size_t)S.j0 * S.nx * NR, n * NR);
        if (nwb == n)
            for (int i = threadIdx.x; i < S.nx; i += blockDim.x) M.wb[n + i] = T(0);   // the grid's upper side
        for (int i = threadIdx.x; i < 2 * S.nxc; i += blockDim.x) {
            Vec<T, NR> z;
#pragma unroll
            for (int k = 0; k < NR; ++k) z.v[k] = T(0);
            M.x[i] = z;
        }
    }
    bool exact = false;
    if (rank == 0) {
        SmallMem<T, NR> M(smem + P.soff, P.S);
        exact = small_operators<T, NR>(P.S, M, diag, id, wl, wb, inv);
    }
    return exact;
}
// (as above) the legs as calls of their own
template <typename T, int NR, bool TILE>
__device__ __noinline__ void cl_down_call(const ClPlan& P, int l, int rank, unsigned char* smem) {
    cl_down<T, NR, 1, TILE>(P, l, rank, smem);
}
template <typename T, int NR>
__device__ __noinline__ void cl_up_call(const ClPlan& P, int l, int rank, unsigned char* smem) {
    cl_up<T, NR, 1, false>(P, l, rank, smem, nullptr);
}
// the down legs, the single-block levels in block 0, and the up legs of the levels below the first;
// CALL: as calls, one block of cells per thread (else two on the first level where it needs them)
template <typename T, int NR, bool CALL>
__device__ inline void cl_cycle(const ClPlan& P, int rank, unsigned char* smem, bool exact) {
    auto two = [&](int l) { return Blk<T, NR>::units(P.nx[l], P.rp[l]) > (int)blockDim.x; };
    for (int l = 0; l < P.nl; ++l) {
        const bool tile = sizeof(T) == 4 || l < P.nt;
        if constexpr (CALL) {
            if (tile) cl_down_call<T, NR, true>(P, l, rank, smem);
            else if constexpr (sizeof(T) == 8) cl_down_call<T, NR, false>(P, l, rank, smem);
        } else if (!tile) {
            if constexpr (sizeof(T) == 8) cl_down<T, NR, 1, false>(P, l, rank, smem);
        } else if (two(l)) {
            cl_down<T, NR, 2, true>(P, l, rank, smem);
        } else {
            cl_down<T, NR, 1, true>(P, l, rank, smem);
        }
    }
    if (rank == 0) {
        SmallMem<T, NR> M(smem + P.soff, P.S);
        small_core<T, NR, false, CALL>(P.S, M, exact);
    }
    cluster_barrier();
    for (int l = P.nl - 1; l >= 1; --l) {
        if constexpr (CALL) cl_up_call<T, NR>(P, l, rank, smem);
        else if (two(l)) cl_up<T, NR, 2, false>(P, l, rank, smem, nullptr);
        else cl_up<T, NR, 1, false>(P, l, rank, smem, nullptr);
    }
}

template <typename T, int NR>
__global__ void __launch_bounds__(CL_THREADS, 1)
k_coarse_cluster(const __grid_constant__ ClPlan P, const T* __restrict__ diag, const T* __restrict__ id,
                 const T* __restrict__ wl, const T* __restrict__ wb, const T* __restrict__ inv,
                 const T* __restrict__ b_in, T* __restrict__ x_out, const SolveState* st) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int rank = cluster_rank();
    const bool exact = cl_operators<T, NR>(P, rank, smem, diag, id, wl, wb, inv, b_in);
    const bool off = skip(st);   // written by an earlier launch: the same for every block
    cp_async_wait_all();
    if (off) return;
    cluster_barrier();
    cl_cycle<T, NR, false>(P, rank, smem, exact);
    if (Blk<T, NR>::units(P.nx[0], P.rp[0]) > (int)blockDim.x) cl_up<T, NR, 2, true>(P, 0, rank, smem, x_out);
    else cl_up<T, NR, 1, true>(P, 0, rank, smem, x_out);
}

// dense inverse of the coarsest operator (at most 32 cells), Gauss-Jordan in precision T by the
// block's warps: per pivot warp 0 scales the pivot row (one reciprocal), then warp w eliminates
// rows w, w + W, ... of [A | I] (A: 32 x 65 values of shared memory; columns past 2 n stay zero and
// are left out).  inv[n * n] = 1 marks a usable inverse; a non-positive or non-finite pivot (a
// singular coarsest operator, e.g. a pure-Neumann pressure problem) leaves 0 there and the cycle
// falls back to sweeps.  The chain of n dependent reciprocals remains (FP64: about 700 cycles each).
template <typename T>
__device__ inline void coarse_inverse_block(int nx, int ny, const T* diag, const T* wl, const T* wb, T* inv, T (*A)[65],
                                            T* row) {
    const int n = nx * ny, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const bool wide = 2 * n > 32;
    for (int r = warp; r < n; r += nw) {
        A[r][lane] = T(0);
        A[r][lane + 32] = T(0);
    }
    __syncthreads();
    if (threadIdx.x < n) {
        int r = threadIdx.x, i = r % nx, j = r / nx;
        T w0 = wl[r], w1 = i < nx - 1 ? wl[r + 1] : T(0), w2 = wb[r], w3 = j < ny - 1 ? wb[r + nx] : T(0);
        A[r][r] = diag[r] + w0 + w1 + w2 + w3;
        if (i > 0) A[r][r - 1] = -w0;
        if (i < nx - 1) A[r][r + 1] = -w1;
        if (j > 0) A[r][r - nx] = -w2;
        if (j < ny - 1) A[r][r + nx] = -w3;
        A[r][n + r] = T(1);
    }
    __syncthreads();
    bool ok = true;
    for (int p = 0; p < n; ++p) {
        if (warp == 0) {
            T piv = A[p][p];
            ok = ok && piv > T(0) && piv < T(INFINITY);
            T rp = T(1) / piv;
            T a0 = A[p][lane] * rp, a1 = wide ? A[p][lane + 32] * rp : T(0);
            __syncwarp();   // every lane has read the pivot
            row[lane] = A[p][lane] = a0;
            if (wide) row[lane + 32] = A[p][lane + 32] = a1;
        }
        __syncthreads();
        for (int r = warp; r < n; r += nw) {
            if (r == p) continue;
            T f = A[r][p];
            T v0 = A[r][lane], v1 = wide ? A[r][lane + 32] : T(0);
            __syncwarp();   // every lane has read the factor
            A[r][lane] = v0 - f * row[lane];
            if (wide) A[r][lane + 32] = v1 - f * row[lane + 32];
        }
        __syncthreads();
    }
    for (int c = threadIdx.x; c < n * n; c += blockDim.x) inv[c] = A[c / n][n + c % n];
    if (threadIdx.x == 0) inv[n * n] = ok ? T(1) : T(0);
}


// an FP64 operator value in the solver precision (FP32: rounded on the integer pipes)
template <typename T>
__device__ __forceinline__ T to_prec(double v);
template <>
__device__ __forceinline__ double to_prec<double>(double v) { return v; }
template <>
__device__ __forceinline__ float to_prec<float>(double v) { return d2f_rn(v); }

// Levels of the hierarchy as the setup kernel sees them.
struct SetupPlan {
    int nlev, nx[Solver::MAXLEV], ny[Solver::MAXLEV];
    size_t off[Solver::MAXLEV];
    long long zs;      // byte stride between the instances of a batched launch
};

// the operator of one cell of a level, and its coarsening: cd summed, dd summed and halved, face
// weights averaged over the two fine faces; c[r][e] = cell (2I + e, 2J + r)
template <typename T>
struct OpCell {
    T cd, dd, wl, wb;
};
template <typename T>
__device__ __forceinline__ OpCell<T> coarsen(const OpCell<T> (&c)[2][2]) {
    OpCell<T> o;
    o.cd = c[0][0].cd + c[0][1].cd + c[1][0].cd + c[1][1].cd;
    o.dd = T(0.5) * (c[0][0].dd + c[0][1].dd + c[1][0].dd + c[1][1].dd);
    o.wl = T(0.5) * (c[0][0].wl + c[1][0].wl);
    o.wb = T(0.5) * (c[0][0].wb + c[0][1].wb);
    return o;
}

// The whole multigrid hierarchy in precision T in one launch.  Block (bx, by) converts its
// SB x SB cells of level 0 (D = cd + dd, face weights, cd, dd; with d64 != null also D in FP64
// for the refinement residual), a thread the four children of a level-1 cell, and coarsens its
// own footprint level by level in shared memory while a level-l cell still lies inside it
// (2^l <= SB); the last block to finish builds the remaining levels from the others' results (in
// shared memory too once a level has at most SETUP_CAP cells) and, when the coarsest level has at
// most 32 cells, its dense inverse.
// Small grids are bound by the chain of levels: read back from global memory each took about a
// microsecond, and the inverse in one warp 3 us in FP32 and 20 us in FP64: 23.7 -> 15.9 us in FP32 at
// 512^2, 42 -> 19 us in FP64 at 64^2, 281 -> 255 us in FP32 at 4096^2.
// Footprints are SB x SB: 64 x 64 on large grids leave the last block a quarter of the work of
// 32 x 32 ones (its levels run serially after every other block has finished: 140 against
// 155 us on a 2048 x 4096 grid), 32 x 32 on small grids keep more blocks busy.
constexpr int SETUP_CAP = 1024;
template <typename T, int SB>
__global__ void __launch_bounds__(256) k_setup_tree(SetupPlan P, const double* __restrict__ cd,
                                                    const double* __restrict__ dd, const double* __restrict__ wl,
                                                    const double* __restrict__ wb, T* diag, T* owl, T* owb, T* ocd,
                                                    T* odd, double* __restrict__ d64, T* inv, unsigned* ticket) {
    const long long zo = zoff(P.zs);
    cd = zsh(cd, zo);
    dd = zsh(dd, zo);
    wl = zsh(wl, zo);
    wb = zsh(wb, zo);
    diag = zsh(diag, zo);
    owl = zsh(owl, zo);
    owb = zsh(owb, zo);
    ocd = zsh(ocd, zo);
    odd = zsh(odd, zo);
    d64 = zsh(d64, zo);
    inv = zsh(inv, zo);
    ticket = zsh(ticket, zo);
    // two levels of a footprint (or of the whole grid); later [A | I] of the inverse
    __shared__ OpCell<T> lev0[SETUP_CAP], lev1[SETUP_CAP / 4];
    static_assert(SB / 2 * (SB / 2) <= SETUP_CAP && sizeof(lev0) >= sizeof(T) * (32 * 65 + 64), "shared buffers");
    const int nx = P.nx[0], ny = P.ny[0];
    auto fine = [&](int c) {   // level-0 cell c: converted, stored, returned
        const double ddv = dd ? dd[c] : 0.0, cdv = cd[c], dg = cdv + ddv;
        OpCell<T> o = {to_prec<T>(cdv), to_prec<T>(ddv), to_prec<T>(wl[c]), to_prec<T>(wb[c])};
        diag[c] = to_prec<T>(dg);
        owl[c] = o.wl;
        owb[c] = o.wb;
        ocd[c] = o.cd;
        odd[c] = o.dd;
        if (d64) d64[c] = dg;
        return o;
    };
    auto store = [&](size_t c, const OpCell<T>& o) {
        ocd[c] = o.cd;
        odd[c] = o.dd;
        owl[c] = o.wl;
        owb[c] = o.wb;
        diag[c] = o.cd + o.dd;
    };
    int l = 1;
    if (P.nlev == 1) {
        for (int k = threadIdx.x; k < SB * SB; k += blockDim.x) {
            const int i = blockIdx.x * SB + k % SB, j = blockIdx.y * SB + k / SB;
            if (i < nx && j < ny) fine(j * nx + i);
        }
    } else {
        constexpr int W = SB / 2;
        for (int k = threadIdx.x; k < W * W; k += blockDim.x) {
            const int I = blockIdx.x * W + k % W, J = blockIdx.y * W + k / W;
            if (I >= P.nx[1] || J >= P.ny[1]) continue;
            const int c = 2 * J * nx + 2 * I;
            const OpCell<T> f[2][2] = {{fine(c), fine(c + 1)}, {fine(c + nx), fine(c + nx + 1)}};
            const OpCell<T> o = coarsen(f);
            store(P.off[1] + (size_t)J * P.nx[1] + I, o);
            lev0[k] = o;
        }
        OpCell<T>*src = lev0, *dst = lev1;
        for (l = 2; l < P.nlev && (1 << l) <= SB; ++l) {
            __syncthreads();
            const int w = SB >> l;
            for (int k = threadIdx.x; k < w * w; k += blockDim.x) {
                const int i = k % w, j = k / w, I = blockIdx.x * w + i, J = blockIdx.y * w + j;
                if (I >= P.nx[l] || J >= P.ny[l]) continue;
                const int q = 2 * j * 2 * w + 2 * i;
                const OpCell<T> f[2][2] = {{src[q], src[q + 1]}, {src[q + 2 * w], src[q + 2 * w + 1]}};
                const OpCell<T> o = coarsen(f);
                store(P.off[l] + (size_t)J * P.nx[l] + I, o);
                dst[k] = o;
            }
            OpCell<T>* t = src;
            src = dst;
            dst = t;
        }
    }
    // the last block: the levels above every block's footprint, then the coarsest inverse
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = arrive_acq_rel(ticket) == gridDim.x * gridDim.y - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    OpCell<T>*src = nullptr, *dst = lev0;   // src: the level below in shared memory, or null
    for (; l < P.nlev; ++l) {
        const int fnx = P.nx[l - 1], n = P.nx[l] * P.ny[l];
        const size_t fo = P.off[l - 1], co = P.off[l];
        const bool keep = n <= (dst == lev0 ? SETUP_CAP : SETUP_CAP / 4);
        for (int k = threadIdx.x; k < n; k += blockDim.x) {
            const int q = 2 * (k / P.nx[l]) * fnx + 2 * (k % P.nx[l]);
            OpCell<T> f[2][2];
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int c = q + r * fnx + e;
                    if (src) f[r][e] = src[c];
                    else f[r][e] = {__ldcg(ocd + fo + c), __ldcg(odd + fo + c), __ldcg(owl + fo + c), __ldcg(owb + fo + c)};
                }
            const OpCell<T> o = coarsen(f);
            store(co + k, o);
            if (keep) dst[k] = o;
        }
        __syncthreads();
        if (keep) {
            src = dst;
            dst = dst == lev0 ? lev1 : lev0;
        } else {
            src = nullptr;
            dst = lev0;
        }
    }
    const int lc = P.nlev - 1;
    if (P.nx[lc] * P.ny[lc] <= 32) {
        T(*A)[65] = reinterpret_cast<T(*)[65]>(lev0);
        coarse_inverse_block<T>(P.nx[lc], P.ny[lc], diag + P.off[lc], owl + P.off[lc], owb + P.off[lc], inv, A,
                                &A[0][0] + 32 * 65);
    }
    if (threadIdx.x == 0) *ticket = 0u;
}

// FP64 levels: the reciprocal of every cell's full diagonal D + its four face weights, correctly
// rounded, once per solve.  The FP64 pipe (one warp instruction per 19 cycles and SM) bounds the
// FP64 smoothers, and the four sums and the reciprocal were 14 of the 24 to 28 FP64 instructions
// that a region cell cost in every smoother launch (the reciprocal stored is the same value).
__global__ void __launch_bounds__(256) k_diag_inverse(SetupPlan P, const double* __restrict__ diag,
                                                      const double* __restrict__ wl, const double* __restrict__ wb,
                                                      double* __restrict__ id) {
    const long long zo = zoff(P.zs);
    diag = zsh(diag, zo);
    wl = zsh(wl, zo);
    wb = zsh(wb, zo);
    id = zsh(id, zo);
    for (int l = 0; l < P.nlev; ++l) {
        const int nx = P.nx[l], ny = P.ny[l];
        const size_t o = P.off[l];
        for (CellWalk cw(nx); cw.c < nx * ny; cw.next()) {
            const size_t c = o + cw.c;
            id[c] = rcp_diag(diag[c] + wl[c] + (cw.i + 1 < nx ? wl[c + 1] : 0.0) + wb[c] +
                             (cw.j + 1 < ny ? wb[c + nx] : 0.0));
        }
    }
}

// ---- CG kernels ---------------------------------------------------------------------------
// p_new = z + beta p_old; q = A p_new; p.q -> alpha = r.z / p.q
// Dot-product accumulation of a thread: FP64 for FP64 data; for FP32 data an FP32-pair running
// sum (48-bit, FP32 instructions only), written to the FP64 total by flush().  An earlier form
// summed FP32 chunks of eight cells into FP64 with a counter tested in the per-cell body, which
// the compiler issued as a predicated FP64 add for every cell (the FP64 pipe 40-60 % busy in
// these memory-bound kernels).  The loop of k_update walks its cells in chunks of DOT_CHUNK (more
// loads in flight per thread).  The inner FP32 solves of the
// refinement work on a residual scaled to values of order one (k_ir_residual), so FP32 products
// neither underflow nor overflow there.
constexpr int DOT_CHUNK = 8;
template <typename T, int NR>
struct DotAcc {
    double tot[NR];
    __device__ DotAcc() {
#pragma unroll
        for (int k = 0; k < NR; ++k) tot[k] = 0.0;
    }
    __device__ void add(int k, T a, T b) { tot[k] += (double)a * (double)b; }
    __device__ void flush() {}
};
// FP32 data: each product added to an FP32-pair running sum (TwoSum, FP32 instructions only);
// flush() writes the sum so far to tot in FP64 (one FP64 add), so it may be called once at the
// end or after every chunk
template <int NR>
struct DotAcc<float, NR> {
    double tot[NR];
    f32x2 sum[NR];
    __device__ DotAcc() {
#pragma unroll
        for (int k = 0; k < NR; ++k) { tot[k] = 0.0; sum[k] = {0.0f, 0.0f}; }
    }
    __device__ void add(int k, float a, float b) {
        f32x2 t = two_sum(sum[k].hi, a * b);
        sum[k] = quick_two_sum(t.hi, t.lo + sum[k].lo);
    }
    __device__ void flush() {
#pragma unroll
        for (int k = 0; k < NR; ++k) tot[k] = x2_to(sum[k]);
    }
};

template <typename T, int NR>
__global__ void __launch_bounds__(256) k_apply(Lev<T> L, const T* __restrict__ z, T* __restrict__ p0,
                                                T* __restrict__ p1, T* __restrict__ q, SolveState* st,
                                                double* partial, unsigned* ticket, int vb) {
    const long long zo = zoff(L.zs);
    L.diag = zsh(L.diag, zo);
    L.wl = zsh(L.wl, zo);
    L.wb = zsh(L.wb, zo);
    z = zsh(z, zo);
    p0 = zsh(p0, zo);
    p1 = zsh(p1, zo);
    q = zsh(q, zo);
    st = zsh(st, zo);
    partial = zsh(partial, zo);
    ticket = zsh(ticket, zo);
    const int it = ld_now(&st->iters);
    T beta[NR];
    double rz[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) {
        beta[k] = (T)ld_now(&st->beta[k]);
        rz[k] = ld_now(&st->rz[k]);
    }
    if (skip(st)) return;
    const Vec<T, NR>* __restrict__ Z = reinterpret_cast<const Vec<T, NR>*>(z);
    const Vec<T, NR>* __restrict__ Po = reinterpret_cast<const Vec<T, NR>*>((it & 1) ? p1 : p0);
    Vec<T, NR>* __restrict__ Pn = reinterpret_cast<Vec<T, NR>*>((it & 1) ? p0 : p1);
    Vec<T, NR>* __restrict__ Q = reinterpret_cast<Vec<T, NR>*>(q);
    int N = L.nx * L.ny;
    for (int v = blockIdx.x; v < vb; v += gridDim.x) {
        DotAcc<T, NR> acc;
#pragma unroll 2
        for (CellWalk cw(L.nx, v, vb); cw.c < N; cw.next()) {
            int c = cw.c, i = cw.i, j = cw.j;
            auto pn = [&](int cc) {
                Vec<T, NR> a = Z[cc], b = Po[cc];
#pragma unroll
                for (int k = 0; k < NR; ++k)
                    if (beta[k] != T(0)) a.v[k] += beta[k] * b.v[k];   // beta = 0: p = z (old p unused)
                return a;
            };
            Vec<T, NR> pc = pn(c), qv;
            T d = L.diag[c];
#pragma unroll
            for (int k = 0; k < NR; ++k) qv.v[k] = d * pc.v[k];
            if (i > 0) {
                T w = L.wl[c];
                Vec<T, NR> a = pn(c - 1);
                for (int k = 0; k < NR; ++k)
                    qv.v[k] += w * (pc.v[k] - a.v[k]);
            }
            if (i < L.nx - 1) {
                T w = L.wl[c + 1];
                Vec<T, NR> a = pn(c + 1);
                for (int k = 0; k < NR; ++k)
                    qv.v[k] += w * (pc.v[k] - a.v[k]);
            }
            if (j > 0) {
                T w = L.wb[c];
                Vec<T, NR> a = pn(c - L.nx);
                for (int k = 0; k < NR; ++k)
                    qv.v[k] += w * (pc.v[k] - a.v[k]);
            }
            if (j < L.ny - 1) {
                T w = L.wb[c + L.nx];
                Vec<T, NR> a = pn(c + L.nx);
                for (int k = 0; k < NR; ++k)
                    qv.v[k] += w * (pc.v[k] - a.v[k]);
            }
#pragma unroll
            for (int k = 0; k < NR; ++k) acc.add(k, pc.v[k], qv.v[k]);
            Pn[c] = pc;
            Q[c] = qv;
        }
        acc.flush();
        block_partial<NR>(acc.tot, partial, vb, v);
    }
    double tot[NR];
    if (last_block_total<NR>(partial, vb, ticket, tot)) {
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            st->pq[k] = tot[k];
            st->alpha[k] = tot[k] != 0.0 ? rz[k] / tot[k] : 0.0;
        }
    }
}

// x += alpha p_new; r -= alpha q; r.r; convergence test; loop condition
template <typename T, int NR>
__global__ void __launch_bounds__(256) k_update(int N, long long zs, T* __restrict__ x, T* __restrict__ r,
                                                 const T* __restrict__ p0,
                                                 const T* __restrict__ p1, const T* __restrict__ q, SolveState* st,
                                                 double* partial, unsigned* ticket, cudaGraphConditionalHandle h,
                                                 int use_h, int vb) {
    const long long zo = zoff(zs);
    x = zsh(x, zo);
    r = zsh(r, zo);
    p0 = zsh(p0, zo);
    p1 = zsh(p1, zo);
    q = zsh(q, zo);
    st = zsh(st, zo);
    partial = zsh(partial, zo);
    ticket = zsh(ticket, zo);
    const int it = ld_now(&st->iters);
    T alpha[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) alpha[k] = (T)ld_now(&st->alpha[k]);
    if (skip(st)) return;
    const Vec<T, NR>* __restrict__ Pn = reinterpret_cast<const Vec<T, NR>*>((it & 1) ? p0 : p1);
    const Vec<T, NR>* __restrict__ Q = reinterpret_cast<const Vec<T, NR>*>(q);
    Vec<T, NR>* __restrict__ X = reinterpret_cast<Vec<T, NR>*>(x);
    Vec<T, NR>* __restrict__ Rr = reinterpret_cast<Vec<T, NR>*>(r);
    for (int v = blockIdx.x; v < vb; v += gridDim.x) {
        DotAcc<T, NR> acc;
        const int stride = vb * blockDim.x;
        auto cell = [&](int c) {
            Vec<T, NR> xv = X[c], rv = Rr[c], pv = Pn[c], qv = Q[c];
#pragma unroll
            for (int k = 0; k < NR; ++k) {
                xv.v[k] += alpha[k] * pv.v[k];
                rv.v[k] -= alpha[k] * qv.v[k];
                acc.add(k, rv.v[k], rv.v[k]);
            }
            X[c] = xv;
            Rr[c] = rv;
        };
        // whole chunks unrolled (their loads in flight at once); the rest of the walk as a loop: a
        // guarded body issues its FP64 instructions whether the cell exists or not, and on a 512^2
        // grid a thread has one or two cells (FP64, 64^2: 7.2 -> 5.9 us)
        int c0 = v * blockDim.x + threadIdx.x;
        for (; c0 + (DOT_CHUNK - 1) * stride < N; c0 += DOT_CHUNK * stride) {
#pragma unroll
            for (int u = 0; u < DOT_CHUNK; ++u) cell(c0 + u * stride);
            acc.flush();
        }
        for (; c0 < N; c0 += stride) cell(c0);
        acc.flush();
        block_partial<NR>(acc.tot, partial, vb, v);
    }
    double tot[NR];
    if (last_block_total<NR>(partial, vb, ticket, tot)) {
        bool done = true, bad = false;
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            st->rr[k] = tot[k];
            if (!(tot[k] <= st->tol2[k])) done = false;
            bad = bad || !isfinite(tot[k]);
        }
        st->iters += 1;
        if (bad) {   // a NaN or infinity: no further iteration can recover
            st->nonfinite = 1;
            done = true;
        }
        if (done) st->done = 1;
        set_cond(h, use_h, (!done && st->iters < st->max_iters) ? 1u : 0u);
    }
}

// ---- the same two kernels for FP32 and one right-hand side, four cells per thread ---------------
// On rows whose length is a multiple of four (and 16-byte aligned arrays) a thread takes four
// consecutive cells of a row: 16-byte loads and stores, a quarter of the index work and four
// times the bytes in flight per load.  Each cell's arithmetic is k_apply's / k_update's (the
// same flux form, terms in the same order); the dot products add a thread's four cells in order
// to its FP32-pair sum.  Virtual blocks over the quads as in the per-cell kernels, so a batched
// instance still sums exactly as the instance launched alone.

// walk over the groups of a thread (row j, group m of the row: cells G m .. G m + G - 1, G = 4
// or 2) of virtual block v of vb, without a division per step
struct QuadWalk {
    int t, m, j, stride, dm, dj, nq;
    __device__ QuadWalk(int nq_, int v, int nv) : nq(nq_) {
        t = v * blockDim.x + threadIdx.x;
        stride = nv * blockDim.x;
        m = t % nq;
        j = t / nq;
        dm = stride % nq;
        dj = stride / nq;
    }
    __device__ void next() {
        t += stride;
        m += dm;
        j += dj;
        if (m >= nq) { m -= nq; ++j; }
    }
};

__device__ __forceinline__ float f4(const float4& a, int k) { return k == 0 ? a.x : k == 1 ? a.y : k == 2 ? a.z : a.w; }

__global__ void __launch_bounds__(256) k_apply4(Lev<float> L, const float* __restrict__ z, float* __restrict__ p0,
                                                float* __restrict__ p1, float* __restrict__ q, SolveState* st,
                                                double* partial, unsigned* ticket, int vb) {
    const long long zo = zoff(L.zs);
    L.diag = zsh(L.diag, zo);
    L.wl = zsh(L.wl, zo);
    L.wb = zsh(L.wb, zo);
    z = zsh(z, zo);
    p0 = zsh(p0, zo);
    p1 = zsh(p1, zo);
    q = zsh(q, zo);
    st = zsh(st, zo);
    partial = zsh(partial, zo);
    ticket = zsh(ticket, zo);
    const int it = ld_now(&st->iters);
    const float beta = (float)ld_now(&st->beta[0]);
    const double rz = ld_now(&st->rz[0]);
    if (skip(st)) return;
    const float* __restrict__ Po = (it & 1) ? p1 : p0;
    float* __restrict__ Pn = (it & 1) ? p0 : p1;
    const int nx = L.nx, ny = L.ny, nq = nx / 4, NQ = nq * ny;
    // p = z + beta p_old of one cell / of four (beta = 0: p = z, the old p unused)
    auto pn1 = [&](int cc) { return beta != 0.0f ? z[cc] + beta * Po[cc] : z[cc]; };
    auto pn4 = [&](int cc) {
        float4 a = *reinterpret_cast<const float4*>(z + cc);
        if (beta != 0.0f) {
            float4 o = *reinterpret_cast<const float4*>(Po + cc);
            a.x += beta * o.x;
            a.y += beta * o.y;
            a.z += beta * o.z;
            a.w += beta * o.w;
        }
        return a;
    };
    for (int v = blockIdx.x; v < vb; v += gridDim.x) {
        DotAcc<float, 1> acc;
#pragma unroll 2
        for (QuadWalk w(nq, v, vb); w.t < NQ; w.next()) {
            const int i0 = 4 * w.m, j = w.j, c = j * nx + i0;
            float4 pc = pn4(c);
            float4 dg = *reinterpret_cast<const float4*>(L.diag + c);
            float4 wl = *reinterpret_cast<const float4*>(L.wl + c);
            float4 wb = *reinterpret_cast<const float4*>(L.wb + c);
            float pl = i0 > 0 ? pn1(c - 1) : 0.0f;
            float pr = i0 + 4 < nx ? pn1(c + 4) : 0.0f;
            float wr3 = i0 + 4 < nx ? L.wl[c + 4] : 0.0f;
            float4 pd = j > 0 ? pn4(c - nx) : make_float4(0.f, 0.f, 0.f, 0.f);
            float4 pu = j < ny - 1 ? pn4(c + nx) : make_float4(0.f, 0.f, 0.f, 0.f);
            float4 wt = j < ny - 1 ? *reinterpret_cast<const float4*>(L.wb + c + nx) : make_float4(0.f, 0.f, 0.f, 0.f);
            float qv[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const float p = f4(pc, a);
                float s = f4(dg, a) * p;
                const int i = i0 + a;
                if (i > 0) s += f4(wl, a) * (p - (a == 0 ? pl : f4(pc, a - 1)));
                if (i < nx - 1) s += (a == 3 ? wr3 : f4(wl, a + 1)) * (p - (a == 3 ? pr : f4(pc, a + 1)));
                if (j > 0) s += f4(wb, a) * (p - f4(pd, a));
                if (j < ny - 1) s += f4(wt, a) * (p - f4(pu, a));
                qv[a] = s;
                acc.add(0, p, s);
            }
            *reinterpret_cast<float4*>(Pn + c) = pc;
            *reinterpret_cast<float4*>(q + c) = make_float4(qv[0], qv[1], qv[2], qv[3]);
        }
        acc.flush();
        block_partial<1>(acc.tot, partial, vb, v);
    }
    double tot[1];
    if (last_block_total<1>(partial, vb, ticket, tot)) {
        st->pq[0] = tot[0];
        st->alpha[0] = tot[0] != 0.0 ? rz / tot[0] : 0.0;
    }
}

// two right-hand sides (liquid and vapour values of a cell interleaved): a thread takes two
// consecutive cells of a row, one float4 of each vector, a float2 of each coefficient array
__global__ void __launch_bounds__(256) k_apply2(Lev<float> L, const float* __restrict__ z, float* __restrict__ p0,
                                                float* __restrict__ p1, float* __restrict__ q, SolveState* st,
                                                double* partial, unsigned* ticket, int vb) {
    const long long zo = zoff(L.zs);
    L.diag = zsh(L.diag, zo);
    L.wl = zsh(L.wl, zo);
    L.wb = zsh(L.wb, zo);
    z = zsh(z, zo);
    p0 = zsh(p0, zo);
    p1 = zsh(p1, zo);
    q = zsh(q, zo);
    st = zsh(st, zo);
    partial = zsh(partial, zo);
    ticket = zsh(ticket, zo);
    const int it = ld_now(&st->iters);
    const float b0 = (float)ld_now(&st->beta[0]), b1 = (float)ld_now(&st->beta[1]);
    const double rz[2] = {ld_now(&st->rz[0]), ld_now(&st->rz[1])};
    if (skip(st)) return;
    const float* __restrict__ Po = (it & 1) ? p1 : p0;
    float* __restrict__ Pn = (it & 1) ? p0 : p1;
    const int nx = L.nx, ny = L.ny, np = nx / 2, NP = np * ny;
    // p = z + beta p_old of one cell (float2) / of two (float4), per right-hand side
    auto pn2 = [&](int cc) {
        float2 a = *reinterpret_cast<const float2*>(z + 2 * cc);
        float2 o = *reinterpret_cast<const float2*>(Po + 2 * cc);
        if (b0 != 0.0f) a.x += b0 * o.x;
        if (b1 != 0.0f) a.y += b1 * o.y;
        return a;
    };
    auto pn4 = [&](int cc) {
        float4 a = *reinterpret_cast<const float4*>(z + 2 * cc);
        float4 o = *reinterpret_cast<const float4*>(Po + 2 * cc);
        if (b0 != 0.0f) { a.x += b0 * o.x; a.z += b0 * o.z; }
        if (b1 != 0.0f) { a.y += b1 * o.y; a.w += b1 * o.w; }
        return a;
    };
    for (int v = blockIdx.x; v < vb; v += gridDim.x) {
        DotAcc<float, 2> acc;
#pragma unroll 2
        for (QuadWalk w(np, v, vb); w.t < NP; w.next()) {
            const int i0 = 2 * w.m, j = w.j, c = j * nx + i0;
            float4 pc = pn4(c);
            float2 dg = *reinterpret_cast<const float2*>(L.diag + c);
            float2 wl = *reinterpret_cast<const float2*>(L.wl + c);
            float2 wb = *reinterpret_cast<const float2*>(L.wb + c);
            float2 pl = i0 > 0 ? pn2(c - 1) : make_float2(0.f, 0.f);
            float2 pr = i0 + 2 < nx ? pn2(c + 2) : make_float2(0.f, 0.f);
            float wr1 = i0 + 2 < nx ? L.wl[c + 2] : 0.0f;
            float4 pd = j > 0 ? pn4(c - nx) : make_float4(0.f, 0.f, 0.f, 0.f);
            float4 pu = j < ny - 1 ? pn4(c + nx) : make_float4(0.f, 0.f, 0.f, 0.f);
            float2 wt = j < ny - 1 ? *reinterpret_cast<const float2*>(L.wb + c + nx) : make_float2(0.f, 0.f);
            float qv[4];
#pragma unroll
            for (int a = 0; a < 2; ++a) {          // cell i0 + a
                const int i = i0 + a;
                const float d = a == 0 ? dg.x : dg.y, wlf = a == 0 ? wl.x : wl.y, wbf = a == 0 ? wb.x : wb.y;
                const float wrf = a == 0 ? wl.y : wr1, wtf = a == 0 ? wt.x : wt.y;
#pragma unroll
                for (int k = 0; k < 2; ++k) {      // right-hand side k
                    const float p = f4(pc, 2 * a + k);
                    float s = d * p;
                    const float left = a == 0 ? (k == 0 ? pl.x : pl.y) : f4(pc, k);
                    const float right = a == 1 ? (k == 0 ? pr.x : pr.y) : f4(pc, 2 + k);
                    if (i > 0) s += wlf * (p - left);
                    if (i < nx - 1) s += wrf * (p - right);
                    if (j > 0) s += wbf * (p - f4(pd, 2 * a + k));
                    if (j < ny - 1) s += wtf * (p - f4(pu, 2 * a + k));
                    qv[2 * a + k] = s;
                    acc.add(k, p, s);
                }
            }
            *reinterpret_cast<float4*>(Pn + 2 * c) = pc;
            *reinterpret_cast<float4*>(q + 2 * c) = make_float4(qv[0], qv[1], qv[2], qv[3]);
        }
        acc.flush();
        block_partial<2>(acc.tot, partial, vb, v);
    }
    double tot[2];
    if (last_block_total<2>(partial, vb, ticket, tot)) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            st->pq[k] = tot[k];
            st->alpha[k] = tot[k] != 0.0 ? rz[k] / tot[k] : 0.0;
        }
    }
}

template <int NR>
__global__ void __launch_bounds__(256) k_update4(int N, long long zs, float* __restrict__ x, float* __restrict__ r,
                                                 const float* __restrict__ p0, const float* __restrict__ p1,
                                                 const float* __restrict__ q, SolveState* st, double* partial,
                                                 unsigned* ticket, cudaGraphConditionalHandle h, int use_h, int vb) {
    const long long zo = zoff(zs);
    x = zsh(x, zo);
    r = zsh(r, zo);
    p0 = zsh(p0, zo);
    p1 = zsh(p1, zo);
    q = zsh(q, zo);
    st = zsh(st, zo);
    partial = zsh(partial, zo);
    ticket = zsh(ticket, zo);
    const int it = ld_now(&st->iters);
    // element e of a float4 belongs to right-hand side e % NR (NR = 2: liquid, vapour interleaved)
    const float a0 = (float)ld_now(&st->alpha[0]), a1 = NR > 1 ? (float)ld_now(&st->alpha[1]) : a0;
    if (skip(st)) return;
    const float4* __restrict__ Pn = reinterpret_cast<const float4*>((it & 1) ? p0 : p1);
    const float4* __restrict__ Q = reinterpret_cast<const float4*>(q);
    float4* __restrict__ X = reinterpret_cast<float4*>(x);
    float4* __restrict__ R = reinterpret_cast<float4*>(r);
    const int NQ = N * NR / 4;
    for (int v = blockIdx.x; v < vb; v += gridDim.x) {
        DotAcc<float, NR> acc;
#pragma unroll 2
        for (int t = v * blockDim.x + threadIdx.x; t < NQ; t += vb * blockDim.x) {
            float4 xv = X[t], rv = R[t], pv = Pn[t], qv = Q[t];
            xv.x += a0 * pv.x;
            xv.y += a1 * pv.y;
            xv.z += a0 * pv.z;
            xv.w += a1 * pv.w;
            rv.x -= a0 * qv.x;
            rv.y -= a1 * qv.y;
            rv.z -= a0 * qv.z;
            rv.w -= a1 * qv.w;
            acc.add(0, rv.x, rv.x);
            acc.add(NR - 1, rv.y, rv.y);
            acc.add(0, rv.z, rv.z);
            acc.add(NR - 1, rv.w, rv.w);
            X[t] = xv;
            R[t] = rv;
        }
        acc.flush();
        block_partial<NR>(acc.tot, partial, vb, v);
    }
    double tot[NR];
    if (last_block_total<NR>(partial, vb, ticket, tot)) {
        bool done = true, bad = false;
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            st->rr[k] = tot[k];
            if (!(tot[k] <= st->tol2[k])) done = false;
            bad = bad || !isfinite(tot[k]);
        }
        st->iters += 1;
        if (bad) {   // a NaN or infinity: no further iteration can recover
            st->nonfinite = 1;
            done = true;
        }
        if (done) st->done = 1;
        set_cond(h, use_h, (!done && st->iters < st->max_iters) ? 1u : 0u);
    }
}

// ---- a whole inner solve in one cooperative launch (small grids) ---------------------------
// On small grids a CG iteration is a handful of short kernels (the V-cycle legs, p/q, x/r), each
// a graph node whose launch costs as much as its work.  k_cg_persist runs the whole inner FP32
// MG-PCG solve of one refinement pass in one cooperative launch: the V-cycle as in the
// cooperative coarse cycle but from the finest level, then p = z + beta p with q = A p, then x
// and r, with a bounded grid barrier between the phases.  The dot products of a phase are
// written as per-tile (r.z) or per-block (p.q, r.r) slots; after the barrier every block sums
// the slots in the same order with the same code, so all blocks hold the same alpha, beta and
// convergence decision without another barrier; block 0 alone writes the solve state.  The
// arithmetic of each cell is that of the separate kernels; only the grouping of the dot
// products differs (per block instead of per launch block).

// the single-block levels as a call: inlined into the whole-solve kernel they add to its spills
template <typename T, int NR>
__device__ __noinline__ void small_cycle_call(const SmallPlan& P, const T* diag, const T* wl, const T* wb,
                                              const T* inv, const T* b_in, T* x_out, SolveState* st,
                                              unsigned char* smem) {
    small_cycle<T, NR, false>(P, diag, nullptr, wl, wb, inv, b_in, x_out, st, smem);
}

// grid barrier that gives up: false if this block's wait ran out or a fault is already recorded
// (every block then leaves at its next barrier, so a fault ends the launch after a bounded time)
__device__ inline bool grid_sync_ok(unsigned* bar, unsigned& target, SolveState* st, int spin) {
    __shared__ int bad;
    target += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) {
        int b = *((volatile int*)&st->fault);
        if (!b) {
            red_release_gpu_add(&bar[0], 1u);
            for (int it = 0; (int)(ld_acquire_gpu(&bar[0]) - target) < 0; ++it)
                if (it > spin) {
                    atomicOr(&st->fault, 2);
                    b = 1;
                    break;
                }
        }
        bad = b;
    }
    __syncthreads();
    return bad == 0;
}

// sum of nslot slots per right-hand side (partial[k * nslot + s]) in a fixed order, in every
// block (the result is in every thread)
template <int NR>
__device__ inline void sum_slots(const double* partial, int nslot, double* tot) {
    __shared__ double sh[32];
    __shared__ double res[2];
#pragma unroll
    for (int k = 0; k < NR; ++k) {
        double a = 0.0;
        for (int b = threadIdx.x; b < nslot; b += blockDim.x) a += ((const volatile double*)partial)[k * nslot + b];
        a = bsum(a, sh);
        if (threadIdx.x == 0) res[k] = a;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NR; ++k) tot[k] = res[k];
    __syncthreads();
}

template <typename T, int NR>
__global__ void __launch_bounds__(CC_THREADS, 1)
k_cg_persist(CoarsePlan<T> C, SmallPlan P, const T* __restrict__ diag, const T* __restrict__ wl,
             const T* __restrict__ wb, const T* __restrict__ inv, T* __restrict__ x, T* __restrict__ r,
             T* __restrict__ p0, T* __restrict__ p1, T* __restrict__ q, SolveState* st, double* partial,
             unsigned* bar) {
    if (skip(st)) return;   // the refinement has converged: the same in every block
    extern __shared__ __align__(128) unsigned char smem[];
    unsigned gen = 0;
    const TileThread tpre = tile_thread<HPRE>(), tpost = tile_thread<HPOST>();
    const int G = gridDim.x;
    const Lev<T>& L0 = C.L[0];
    const int N = L0.nx * L0.ny;
    const int tx0 = (L0.nx + TX - 1) / TX, nt0 = tx0 * ((L0.ny + TY - 1) / TY);
    double* prz = partial;                // r.z per finest tile
    double* ppq = partial + 2 * nt0;      // p.q per block
    double* prr = ppq + 2 * G;            // r.r per block
    double rz[2], tol2[2], alpha[2] = {0.0, 0.0}, beta[2] = {0.0, 0.0}, pq[2] = {0.0, 0.0}, rr[2] = {0.0, 0.0};
    int iters = st->iters;
    const int maxit = st->max_iters;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        rz[k] = st->rz[k];
        tol2[k] = st->tol2[k];
    }
    bool done = false, bad = false, ok = true;
    while (!done) {
        // ---- z = M r: the V-cycle from the finest level
        for (int l = 0; l < C.nb && ok; ++l) {
            const Lev<T>& L = C.L[l];
            int tx = (L.nx + TX - 1) / TX, nt = tx * ((L.ny + TY - 1) / TY);
            for (int t = blockIdx.x; t < nt; t += G) {
                pre_tile<T, NR>(L, C.b[l], C.x2[l], C.bc[l], t % tx, t / tx, smem, nullptr, tpre);
                __syncthreads();
            }
            ok = grid_sync_ok(bar, gen, st, C.spin);
        }
        if (!ok) break;
        if (blockIdx.x == 0) small_cycle_call<T, NR>(P, diag, wl, wb, inv, C.bc[C.nb - 1], C.xo[C.nb], st, smem);
        if (!grid_sync_ok(bar, gen, st, C.spin)) break;
        for (int l = C.nb - 1; l >= 1 && ok; --l) {
            const Lev<T>& L = C.L[l];
            int tx = (L.nx + TX - 1) / TX, nt = tx * ((L.ny + TY - 1) / TY);
            for (int t = blockIdx.x; t < nt; t += G) {
                post_tile<T, NR, false>(L, C.b[l], C.x2[l], C.xo[l], C.xc[l], t % tx, t / tx, smem, nullptr, tpost);
                __syncthreads();
            }
            ok = grid_sync_ok(bar, gen, st, C.spin);
        }
        if (!ok) break;
        for (int t = blockIdx.x; t < nt0; t += G) {
            Vec<T, 2> d =
                post_tile<T, NR, true>(L0, C.b[0], C.x2[0], C.xo[0], C.xc[0], t % tx0, t / tx0, smem, nullptr, tpost);
            block_partial_t<T, NR>(d.v, prz, nt0, t);
            __syncthreads();
        }
        if (!grid_sync_ok(bar, gen, st, C.spin)) break;
        double rzn[2] = {0.0, 0.0};
        sum_slots<NR>(prz, nt0, rzn);
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            beta[k] = rz[k] != 0.0 ? rzn[k] / rz[k] : 0.0;
            rz[k] = rzn[k];
        }
        // ---- p = z + beta p; q = A p; p.q (the new p of the neighbours recomputed, as k_apply)
        const Vec<T, NR>* __restrict__ Z = reinterpret_cast<const Vec<T, NR>*>(C.xo[0]);
        const Vec<T, NR>* __restrict__ Po = reinterpret_cast<const Vec<T, NR>*>((iters & 1) ? p1 : p0);
        Vec<T, NR>* __restrict__ Pn = reinterpret_cast<Vec<T, NR>*>((iters & 1) ? p0 : p1);
        Vec<T, NR>* __restrict__ Q = reinterpret_cast<Vec<T, NR>*>(q);
        {
            T bt[NR];
#pragma unroll
            for (int k = 0; k < NR; ++k) bt[k] = (T)beta[k];
            DotAcc<T, NR> acc;
            for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += G * blockDim.x) {
                int i = c % L0.nx, j = c / L0.nx;
                auto pn = [&](int cc) {
                    Vec<T, NR> a = Z[cc], b = Po[cc];
#pragma unroll
                    for (int k = 0; k < NR; ++k)
                        if (bt[k] != T(0)) a.v[k] += bt[k] * b.v[k];
                    return a;
                };
                Vec<T, NR> pc = pn(c), qv;
                T dg = L0.diag[c];
#pragma unroll
                for (int k = 0; k < NR; ++k) qv.v[k] = dg * pc.v[k];
                if (i > 0) {
                    T w = L0.wl[c];
                    Vec<T, NR> a = pn(c - 1);
                    for (int k = 0; k < NR; ++k) qv.v[k] += w * (pc.v[k] - a.v[k]);
                }
                if (i < L0.nx - 1) {
                    T w = L0.wl[c + 1];
                    Vec<T, NR> a = pn(c + 1);
                    for (int k = 0; k < NR; ++k) qv.v[k] += w * (pc.v[k] - a.v[k]);
                }
                if (j > 0) {
                    T w = L0.wb[c];
                    Vec<T, NR> a = pn(c - L0.nx);
                    for (int k = 0; k < NR; ++k) qv.v[k] += w * (pc.v[k] - a.v[k]);
                }
                if (j < L0.ny - 1) {
                    T w = L0.wb[c + L0.nx];
                    Vec<T, NR> a = pn(c + L0.nx);
                    for (int k = 0; k < NR; ++k) qv.v[k] += w * (pc.v[k] - a.v[k]);
                }
#pragma unroll
                for (int k = 0; k < NR; ++k) acc.add(k, pc.v[k], qv.v[k]);
                Pn[c] = pc;
                Q[c] = qv;
            }
            acc.flush();
            block_partial<NR>(acc.tot, ppq, G, blockIdx.x);
        }
        if (!grid_sync_ok(bar, gen, st, C.spin)) break;
        sum_slots<NR>(ppq, G, pq);
#pragma unroll
        for (int k = 0; k < NR; ++k) alpha[k] = pq[k] != 0.0 ? rz[k] / pq[k] : 0.0;
        // ---- x += alpha p; r -= alpha q; r.r
        {
            T al[NR];
#pragma unroll
            for (int k = 0; k < NR; ++k) al[k] = (T)alpha[k];
            Vec<T, NR>* __restrict__ X = reinterpret_cast<Vec<T, NR>*>(x);
            Vec<T, NR>* __restrict__ Rr = reinterpret_cast<Vec<T, NR>*>(r);
            DotAcc<T, NR> acc;
            const int stride = G * blockDim.x;
            for (int c0 = blockIdx.x * blockDim.x + threadIdx.x; c0 < N; c0 += DOT_CHUNK * stride) {
#pragma unroll
                for (int u = 0; u < DOT_CHUNK; ++u) {
                    int c = c0 + u * stride;
                    if (c < N) {
                        Vec<T, NR> xv = X[c], rv = Rr[c], pv = Pn[c], qv = Q[c];
#pragma unroll
                        for (int k = 0; k < NR; ++k) {
                            xv.v[k] += al[k] * pv.v[k];
                            rv.v[k] -= al[k] * qv.v[k];
                            acc.add(k, rv.v[k], rv.v[k]);
                        }
                        X[c] = xv;
                        Rr[c] = rv;
                    }
                }
                acc.flush();
            }
            block_partial<NR>(acc.tot, prr, G, blockIdx.x);
        }
        if (!grid_sync_ok(bar, gen, st, C.spin)) break;
        sum_slots<NR>(prr, G, rr);
        iters += 1;
        done = true;
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            if (!(rr[k] <= tol2[k])) done = false;
            bad = bad || !isfinite(rr[k]);
        }
        if (bad || iters >= maxit) done = true;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            st->rz[k] = rz[k];
            st->beta[k] = beta[k];
            st->pq[k] = pq[k];
            st->alpha[k] = alpha[k];
            st->rr[k] = rr[k];
        }
        st->iters = iters;
        if (bad) st->nonfinite = 1;
        st->done = 1;
    }
}

// ---- a whole CG solve in one thread-block cluster (grids of up to 16384 cells, instances alone) ---
// On these grids a CG iteration is five launches of 5 to 50 us whose work is a microsecond or two:
// launch, first reads of the state, the reduction's tail.  The cluster of the coarse levels also
// keeps level 0: r and x (z) with its slab, the search direction p with halo rows, the solution;
// an iteration is the V-cycle's phases, four reductions' worth of cluster barriers and no launch.
// A reduction's partial sums are stored into every block's shared memory, so all blocks form the
// same totals, alpha, beta and convergence decision.
//   * r.z: the sums of the post-smoothing tiles (32 x 32, the shuffle trees of its 13 warps) are
//     formed by the block tile t belongs to (t % 16), in the tile kernel's precision and order.
//   * p.q and r.r: the sums of the element kernels.  A unit is what one of their threads sums (FP64
//     a cell; FP32, by FP32-pair sums, four cells of a row, two with two right-hand sides, one where
//     rows are not a multiple of four), units go in groups of 32 (a warp's tree), eight groups a
//     block's slot, then the slots' tree.  Four lanes take a group: a lane-parallel tree is nine
//     FP64 instructions per 8 groups where shuffle trees are 40.
// So a solve is bit for bit that of the separate launches.  Bound: latency, a chain of some 60
// cluster and block barriers and FP64 sweeps (64 cycles an operation) an iteration.  Measured, one
// solve of the separate launches -> this kernel: 120x104 FP64 to 1e-10 1.27 -> 0.94 ms; ten steps on
// 64x64 in FP64 8.7 -> 6.5 ms.
struct CgPlan {
    ClPlan C;
    int p_off, x_off, prod_off, w_off, tb_off, tw_off, ts_off;   // byte offsets in shared memory
    int tx, nt, tslots;          // 32 x 32 tiles: a row, all, per block
    int unit;                    // cells of a unit of p.q and r.r
    int pstride;                 // entries of prod per right-hand side
    int ngrp, nslot;             // slots of 8 groups of 32 units, and their groups
};
constexpr int CG_GRP = 36;       // a group of 32 products takes 36 (fewer bank conflicts)

// totals over the whole cluster; buf: which of the two sets of partial sums.  The FP64 work on a
// total (a division is ten dependent operations) is one lane's, fin(k, total) by lane 0 of warp k:
// every thread of the block doing it would keep the FP64 pipe busy for 2 us.
template <typename T, int NR>
struct CgSum {
    const CgPlan& P;
    unsigned char* smem;
    int rank, buf;
    // prod[k][unit] is in shared memory (every unit of the slab written): its `units` units, the first
    // one of group g0
    template <class Fin>
    __device__ void total(int units, int g0, Fin&& fin) {
        double* prod = (double*)(smem + P.prod_off);
        double* W = (double*)(smem + P.w_off) + buf * NR * P.ngrp;
        const int ps = P.pstride, ng = (units + 31) / 32, m = threadIdx.x & 3, lane = threadIdx.x & 31;
        __syncthreads();
        for (int q0 = 0; q0 < ng * NR; q0 += blockDim.x >> 2) {
            const int q = q0 + (threadIdx.x >> 2), k = q >= ng && NR > 1 ? 1 : 0, g = q - k * ng;
            const bool in = q < ng * NR;
            double v[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) v[t] = in ? prod[k * ps + g * CG_GRP + m + 4 * t] : 0.0;
            // lanes i and i + 16, i + 8, i + 4 of the warp tree: i = m + 4 t
            double c = ((v[0] + v[4]) + (v[2] + v[6])) + ((v[1] + v[5]) + (v[3] + v[7]));
            c += __shfl_down_sync(0xffffffffu, c, 2, 4);
            c += __shfl_down_sync(0xffffffffu, c, 1, 4);
            c = __shfl_sync(0xffffffffu, c, lane & ~3);
            if (in)
#pragma unroll
                for (int r = 0; r < CL_BLOCKS / 4; ++r) cluster_map(W, m + 4 * r)[k * P.ngrp + g0 + g] = c;
        }
        cluster_barrier();
        if (threadIdx.x < 32 * NR) {   // warp k
            const int k = threadIdx.x >> 5;
            double s[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int v = lane + 32 * h;
                s[h] = 0.0;
                if (v < P.nslot) {
                    const double* w = W + k * P.ngrp + 8 * v;
                    s[h] = ((w[0] + w[4]) + (w[2] + w[6])) + ((w[1] + w[5]) + (w[3] + w[7]));
                }
            }
            for (int o = 16; o > 0; o >>= 1) {
                s[0] += __shfl_down_sync(0xffffffffu, s[0], o);
                if (P.nslot > 32) s[1] += __shfl_down_sync(0xffffffffu, s[1], o);
            }
            if (lane == 0) fin(k, P.nslot > 32 ? s[0] + s[1] : s[0]);
        }
        __syncthreads();
    }
};

template <typename T, int NR>
__global__ void __launch_bounds__(CL_THREADS, 1)
k_cg_cluster(const __grid_constant__ CgPlan G, const T* __restrict__ diag, const T* __restrict__ id,
             const T* __restrict__ wl, const T* __restrict__ wb, const T* __restrict__ inv, const T* __restrict__ r_in,
             T* x_io, SolveState* st) {
    using V = Vec<T, NR>;
    extern __shared__ __align__(128) unsigned char smem[];
    // the solve's scalars, the same in every block
    __shared__ double rz[2], alpha[2], beta[2], pq[2], rr[2], tol2[2];
    __shared__ int cont[2], nonfin[2];   // the residual is above the tolerance / not finite
    const ClPlan& P = G.C;
    const int rank = cluster_rank();
    const bool exact = cl_operators<T, NR>(P, rank, smem, diag, id, wl, wb, inv, r_in);
    const ClSlab S(P, 0, rank);
    const ClMem<T, NR> M(smem + P.off[0], S.nx, S.rp);
    V* pa = (V*)(smem + G.p_off);            // p, as a level's x array
    V* xs = (V*)(smem + G.x_off);            // the solution, [cell of the block][thread]
    V* xg = reinterpret_cast<V*>(x_io);
    const int nthr = blockDim.x, rows = S.j1 - S.j0;
    for (int i = threadIdx.x; i < 2 * S.nxc; i += nthr) {
        V z;
#pragma unroll
        for (int k = 0; k < NR; ++k) z.v[k] = T(0);
        pa[i] = z;
    }
    {   // partial sums that no block writes count as 0; cells of the last group beyond the grid too
        const int bytes = G.ts_off + (int)sizeof(double) * NR * 64 - G.prod_off;
        for (int i = threadIdx.x; i < bytes / 4; i += nthr) reinterpret_cast<int*>(smem + G.prod_off)[i] = 0;
    }
    if (threadIdx.x < 2) {
        rz[threadIdx.x] = st->rz[threadIdx.x];
        tol2[threadIdx.x] = st->tol2[threadIdx.x];
    }
    int iters = ld_now(&st->iters);
    const int maxit = ld_now(&st->max_iters);
    const bool off = skip(st);   // written by an earlier launch: the same for every block
    Blk<T, NR> B[1];
    unsigned edge[1];
    int I[1], j[1];
    B[0].place(S.hx, rows, threadIdx.x, I[0], j[0]);
    // global index of the block's cell (row r, column e), or of the local one
    auto gcell = [&](int r, int e) { return (S.j0 + j[0] + r) * S.nx + 2 * I[0] + e; };
    if (!off && B[0].own)
        B[0].cells([&](int n, int r, int e, T, T, T, T, T, const V&, const V&) { xs[n * nthr + threadIdx.x] = xg[gcell(r, e)]; });
    cp_async_wait_all();
    if (off) return;
    cluster_barrier();
    V* pdn = cluster_map(pa, rank > 0 ? rank - 1 : 0);
    V* pup = cluster_map(pa, rank + 1 < CL_BLOCKS ? rank + 1 : rank);
    bool done = false, bad = false;
    while (!done && iters < maxit) {
        // ---- z = M r
        cl_cycle<T, NR, true>(P, rank, smem, exact);
        cl_up_blocks<T, NR, 1, true>(B, edge, I, j, S, M, P, 0, rank, smem);
        // ---- r.z of the block's 2 x 2 cells to the owner of its tile
        {
            const int Jg = (S.j0 + j[0]) >> 1, t = (Jg >> 4) * G.tx + (I[0] >> 4);
            T* TB = (T*)(smem + G.tb_off);
            V dot;
#pragma unroll
            for (int k = 0; k < NR; ++k) dot.v[k] = T(0);
            auto add = [&]() {
                B[0].cells([&](int, int, int, T, T, T, T, T, const V& bv, const V& xv) {
#pragma unroll
                    for (int k = 0; k < NR; ++k) dot.v[k] = fma_rn(xv.v[k], bv.v[k], dot.v[k]);
                });
            };
            bool send = B[0].own;
            if constexpr (Blk<T, NR>::RB == 1) {   // the even row's two cells, then the odd row's
                const int slot = (j[0] >> 1) * S.hx + I[0];
                if (B[0].own && !(j[0] & 1)) {
                    add();
                    M.s[slot] = dot;
                    send = false;
                }
                __syncthreads();
                if (B[0].own && (j[0] & 1)) {
                    dot = M.s[slot];
                    add();
                }
            } else if (B[0].own) {
                add();
            }
            if (send) {
                T* dst = cluster_map(TB, t & (CL_BLOCKS - 1)) + (t / CL_BLOCKS) * NR * 256 + (Jg & 15) * 16 + (I[0] & 15);
#pragma unroll
                for (int k = 0; k < NR; ++k) dst[k * 256] = dot.v[k];
            }
            cluster_barrier();
            // the trees of the tile kernel's 13 warps over its 20 x 20 threads (16 x 16 of them with cells)
            T* TW = (T*)(smem + G.tw_off);
            double* TS = (double*)(smem + G.ts_off);
            const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = nthr >> 5, jobs = G.tslots * NR;
            for (int q = warp; q < jobs * 13; q += nw) {
                const int sk = q / 13, ix = 32 * (q - sk * 13) + lane, kk = ix % 20 - 2, sg = ix / 20 - 2;
                T v = kk >= 0 && kk < 16 && sg >= 0 && sg < 16 ? TB[sk * 256 + sg * 16 + kk] : T(0);
                for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
                if (lane == 0) TW[sk * 16 + q - sk * 13] = v;
            }
            __syncthreads();
            for (int sk = warp; sk < jobs; sk += nw) {
                T v = lane < 13 ? TW[sk * 16 + lane] : T(0);
                for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
                const double w = widen(__shfl_sync(0xffffffffu, v, 0));
                const int tt = (sk / NR) * CL_BLOCKS + rank;
                if (tt < G.nt && lane < CL_BLOCKS) cluster_map(TS, lane)[(sk % NR) * 64 + tt] = w;
            }
            cluster_barrier();
            if (warp < NR) {
                double a = TS[warp * 64 + lane], b = TS[warp * 64 + 32 + lane];   // 0 beyond the tiles
                for (int o = 16; o > 0; o >>= 1) {
                    a += __shfl_down_sync(0xffffffffu, a, o);
                    if (G.nt > 32) b += __shfl_down_sync(0xffffffffu, b, o);
                }
                if (lane == 0) {
                    const double tot = G.nt > 32 ? a + b : a, old = rz[warp];
                    beta[warp] = old != 0.0 ? tot / old : 0.0;
                    rz[warp] = tot;
                }
            }
            __syncthreads();
        }
        // ---- p = z + beta p, its edge rows to the neighbours
        T bt[NR];
#pragma unroll
        for (int k = 0; k < NR; ++k) bt[k] = (T)beta[k];
        auto pidx = [&](int r, int e) { return ((e ^ r ^ (j[0] & 1)) ? S.nxc : 0) + xidx(S.hx, I[0], j[0] + r); };
        if (B[0].own)
            B[0].cells([&](int, int r, int e, T, T, T, T, T, const V&, V& xv) {
                V* q = pa + pidx(r, e);
                const V po = *q;
#pragma unroll
                for (int k = 0; k < NR; ++k)
                    if (bt[k] != T(0)) xv.v[k] = fma_rn(bt[k], po.v[k], xv.v[k]);
                *q = xv;   // the block's x is now p
                if ((edge[0] & CL_DOWN) && r == 0) pdn[(q - pa) + S.rp * S.hx] = xv;
                if ((edge[0] & CL_UP) && r == Blk<T, NR>::RB - 1) pup[(q - pa) - rows * S.hx] = xv;
            });
        cluster_barrier();
        // ---- q = A p, p.q
        V qv[Blk<T, NR>::CELLS];
        // the cells' terms a.b summed by unit into shared memory, then over the cluster
        auto dot = [&](const V (&a)[Blk<T, NR>::CELLS], const V (&b)[Blk<T, NR>::CELLS], int buf, auto&& fin) {
            double* prod = (double*)(smem + G.prod_off);
            auto put = [&](int k, int c, double v) {   // unit of local cell c (its last one)
                const int u = c / G.unit;
                prod[k * G.pstride + u + 4 * (u >> 5)] = v;
            };
            if constexpr (sizeof(T) == 8) {
                if (B[0].own)
#pragma unroll
                    for (int n = 0; n < 2; ++n)
#pragma unroll
                        for (int k = 0; k < NR; ++k)
                            put(k, j[0] * S.nx + 2 * I[0] + (n ^ B[0].par), a[n].v[k] * b[n].v[k]);
            } else {
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int c = (j[0] + r) * S.nx + 2 * I[0], n0 = r ? 3 : 0, n1 = r ? 2 : 1;   // columns 2I, 2I + 1
                    DotAcc<T, NR> acc;
                    if (G.unit == 1) {
                        if (B[0].own)
#pragma unroll
                            for (int k = 0; k < NR; ++k) {
                                DotAcc<T, NR> one;
                                one.add(k, a[n0].v[k], b[n0].v[k]);
                                one.flush();
                                put(k, c, one.tot[k]);
                                acc.add(k, a[n1].v[k], b[n1].v[k]);
                                acc.flush();
                                put(k, c + 1, acc.tot[k]);
                            }
                        continue;
                    }
                    if (B[0].own)
#pragma unroll
                        for (int k = 0; k < NR; ++k) {
                            acc.add(k, a[n0].v[k], b[n0].v[k]);
                            acc.add(k, a[n1].v[k], b[n1].v[k]);
                        }
                    if (G.unit == 4) {   // the odd thread of two neighbours goes on from the even one's sum
                        DotAcc<T, NR> go = acc;
#pragma unroll
                        for (int k = 0; k < NR; ++k) {
                            go.sum[k].hi = __shfl_up_sync(0xffffffffu, acc.sum[k].hi, 1);
                            go.sum[k].lo = __shfl_up_sync(0xffffffffu, acc.sum[k].lo, 1);
                        }
                        if (B[0].own && (I[0] & 1))
#pragma unroll
                            for (int k = 0; k < NR; ++k) {
                                go.add(k, a[n0].v[k], b[n0].v[k]);
                                go.add(k, a[n1].v[k], b[n1].v[k]);
                                go.flush();
                                put(k, c, go.tot[k]);
                            }
                    } else if (B[0].own) {
#pragma unroll
                        for (int k = 0; k < NR; ++k) {
                            acc.flush();
                            put(k, c, acc.tot[k]);
                        }
                    }
                }
            }
            CgSum<T, NR>{G, smem, rank, buf}.total(rows * S.nx / G.unit, S.j0 * S.nx / (32 * G.unit), fin);
        };
        V pv_[Blk<T, NR>::CELLS];
        if (B[0].own)
            B[0].cells([&](int n, int r, int e, T w0, T w1, T w2, T w3, T dg, const V&, const V& pv) {
                const int row = j[0] + r;
                const V* q = pa + (((e ^ row) & 1) ? 0 : S.nxc);   // the other colour
                const int x0 = xidx(S.hx, I[0], row);
                const V pl = q[e ? x0 : x0 - 1], pr = q[e ? x0 + 1 : x0], pd = q[x0 - S.hx], pu = q[x0 + S.hx];
#pragma unroll
                for (int k = 0; k < NR; ++k) {
                    const T pc = pv.v[k];
                    T a = fma_rn(w0, pc - pl.v[k], dg * pc);
                    a = fma_rn(w1, pc - pr.v[k], a);
                    a = fma_rn(w2, pc - pd.v[k], a);
                    a = fma_rn(w3, pc - pu.v[k], a);
                    qv[n].v[k] = a;
                }
            });
        if (B[0].own)
            B[0].cells([&](int n, int, int, T, T, T, T, T, const V&, const V& p) { pv_[n] = p; });
        dot(pv_, qv, 0, [&](int k, double t) {
            pq[k] = t;
            alpha[k] = t != 0.0 ? rz[k] / t : 0.0;
        });
        // ---- x += alpha p, r -= alpha q, r.r
        T al[NR];
#pragma unroll
        for (int k = 0; k < NR; ++k) al[k] = (T)alpha[k];
        if (B[0].own)
            B[0].cells([&](int n, int r, int e, T, T, T, T, T, V& bv, const V& pv) {
                V xv = xs[n * nthr + threadIdx.x];
#pragma unroll
                for (int k = 0; k < NR; ++k) {
                    xv.v[k] = fma_rn(al[k], pv.v[k], xv.v[k]);
                    bv.v[k] = fma_rn(-al[k], qv[n].v[k], bv.v[k]);
                }
                qv[n] = bv;
                xs[n * nthr + threadIdx.x] = xv;
                M.b[(j[0] + r) * S.nx + 2 * I[0] + e] = bv;
            });
        dot(qv, qv, 1, [&](int k, double t) {
            rr[k] = t;
            cont[k] = !(t <= tol2[k]);
            nonfin[k] = !isfinite(t);
        });
        iters += 1;
        done = true;
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            if (cont[k]) done = false;
            bad = bad || nonfin[k] != 0;
        }
        if (bad) done = true;   // a NaN or infinity: no further iteration can recover
    }
    if (B[0].own)
        B[0].cells([&](int n, int r, int e, T, T, T, T, T, const V&, const V&) { xg[gcell(r, e)] = xs[n * nthr + threadIdx.x]; });
    if (rank == 0 && threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            st->rz[k] = rz[k];
            st->beta[k] = beta[k];
            st->pq[k] = pq[k];
            st->alpha[k] = alpha[k];
            st->rr[k] = rr[k];
        }
        st->iters = iters;
        if (bad) st->nonfinite = 1;
        if (done) st->done = 1;
    }
}

// FP64 CG start: r = b - A x, r.r, b.b, tolerance, state reset
template <int NR>
__global__ void __launch_bounds__(256)
k_init64(Lev<double> L, const double* __restrict__ b, const double* __restrict__ x, double* __restrict__ r,
         SolveState* st, double* partial, unsigned* ticket, double rtol2, int max_iters,
         cudaGraphConditionalHandle h, int use_h, int vb) {
    const long long zo = zoff(L.zs);
    L.diag = zsh(L.diag, zo);
    L.wl = zsh(L.wl, zo);
    L.wb = zsh(L.wb, zo);
    b = zsh(b, zo);
    x = zsh(x, zo);
    r = zsh(r, zo);
    st = zsh(st, zo);
    partial = zsh(partial, zo);
    ticket = zsh(ticket, zo);
    int N = L.nx * L.ny;
    const Vec<double, NR>* X = reinterpret_cast<const Vec<double, NR>*>(x);
    const Vec<double, NR>* B = reinterpret_cast<const Vec<double, NR>*>(b);
    for (int v = blockIdx.x; v < vb; v += gridDim.x) {
        double acc[2 * NR];
#pragma unroll
        for (int k = 0; k < 2 * NR; ++k) acc[k] = 0.0;
        for (CellWalk cw(L.nx, v, vb); cw.c < N; cw.next()) {
            int c = cw.c, i = cw.i, j = cw.j;
            Vec<double, NR> xv = X[c], bv = B[c], s;   // s = (A x)_i in flux form
            double dg = L.diag[c];
#pragma unroll
            for (int k = 0; k < NR; ++k) s.v[k] = dg * xv.v[k];
            if (i > 0) { double w = L.wl[c]; for (int k = 0; k < NR; ++k) s.v[k] += w * (xv.v[k] - X[c - 1].v[k]); }
            if (i < L.nx - 1) {
                double w = L.wl[c + 1];
                for (int k = 0; k < NR; ++k)
                    s.v[k] += w * (xv.v[k] - X[c + 1].v[k]);
            }
            if (j > 0) { double w = L.wb[c]; for (int k = 0; k < NR; ++k) s.v[k] += w * (xv.v[k] - X[c - L.nx].v[k]); }
            if (j < L.ny - 1) {
                double w = L.wb[c + L.nx];
                for (int k = 0; k < NR; ++k)
                    s.v[k] += w * (xv.v[k] - X[c + L.nx].v[k]);
            }
            Vec<double, NR> rv;
#pragma unroll
            for (int k = 0; k < NR; ++k) {
                rv.v[k] = bv.v[k] - s.v[k];
                acc[k] += rv.v[k] * rv.v[k];
                acc[NR + k] += bv.v[k] * bv.v[k];
            }
            reinterpret_cast<Vec<double, NR>*>(r)[c] = rv;
        }
        block_partial<2 * NR>(acc, partial, vb, v);
    }
    double tot[2 * NR];
    if (last_block_total<2 * NR>(partial, vb, ticket, tot)) {
        bool done = true, bad = false;
        for (int k = 0; k < 2; ++k) {
            double rr = k < NR ? tot[k] : 0.0, bb = k < NR ? tot[NR + k] : 0.0;
            st->rr[k] = rr;
            st->bb[k] = bb;
            st->tol2[k] = rtol2 * (bb > 1e-300 ? bb : 1e-300);
            st->rz[k] = 0.0;
            st->beta[k] = 0.0;
            if (!(rr <= st->tol2[k])) done = false;
            if (!isfinite(rr) || !isfinite(bb)) bad = true;
        }
        st->nonfinite = bad ? 1 : 0;
        if (bad) done = true;   // no iteration: the system holds a NaN or an infinity
        st->iters = 0;
        st->itot = 0;
        st->max_iters = max_iters;
        st->done = done ? 1 : 0;
        st->odone = 0;
        st->oiters = 0;
        st->nr = NR;
        set_cond(h, use_h, done ? 0u : 1u);
    }
}

// power of two s that brings cell values whose sum of squares over n cells is rr to order one
__device__ inline double unit_scale(double rr, int n) {
    double m = sqrt(rr / (double)n);
    int e = (m > 0.0 && isfinite(m)) ? ilogb(m) : 0;
    e = e < -1000 ? -1000 : (e > 1000 ? 1000 : e);
    return ldexp(1.0, -e);
}

// refinement start: b.b and the outer tolerance
template <int NR>
__global__ void __launch_bounds__(256) k_ir_init(int N, long long zs, const double* __restrict__ b, SolveState* st,
                                                  double* partial,
                                                  unsigned* ticket, double rtol2, double inner_rtol, int max_iters,
                                                  int max_outer, int vb) {
    const long long zo = zoff(zs);
    b = zsh(b, zo);
    st = zsh(st, zo);
    partial = zsh(partial, zo);
    ticket = zsh(ticket, zo);
    for (int v = blockIdx.x; v < vb; v += gridDim.x) {
        double acc[NR];
#pragma unroll
        for (int k = 0; k < NR; ++k) acc[k] = 0.0;
        for (int c = v * blockDim.x + threadIdx.x; c < N; c += vb * blockDim.x) {
            Vec<double, NR> bv = reinterpret_cast<const Vec<double, NR>*>(b)[c];
#pragma unroll
            for (int k = 0; k < NR; ++k) acc[k] += bv.v[k] * bv.v[k];
        }
        block_partial<NR>(acc, partial, vb, v);
    }
    double tot[NR];
    if (last_block_total<NR>(partial, vb, ticket, tot)) {
        for (int k = 0; k < 2; ++k) {
            double bb = k < NR ? tot[k] : 0.0;
            st->obb[k] = bb;
            st->otol2[k] = rtol2 * (bb > 1e-300 ? bb : 1e-300);
            st->scale_next[k] = unit_scale(bb, N);
        }
        st->odone = 0;
        st->oiters = 0;
        st->done = 0;
        st->iters = 0;
        st->itot = 0;
        st->max_iters = max_iters;
        st->max_outer = max_outer;
        st->inner_rtol = inner_rtol;
        st->nr = NR;
        st->nonfinite = 0;
    }
}

// refinement sweep: r64 = b - A64 x, outer test, r32 = r64, e = 0, inner state reset
// Bound: the FP64 pipe (19 cycles a warp instruction and SM).  A thread walks R rows of W cells: a
// difference of x across a face serves both its cells (the other one's is its exact negative), 8.6
// FP64 instructions a cell where one cell at a time needs 10, and the vertical ones need no second
// load of x.  W = 2: four cells a row save 0.4 more but leave 16 warps an SM, the pipe half idle
// (1024x2048, two right-hand sides: 112 us); loading a row ahead likewise (110).  Measured, one and two
// right-hand sides: 512^2 16.7 and 25.6 -> 15.6 and 22.4 us; 4096^2 331 and 652 -> 302 and 566 (a step 21.6
// -> 21.0 ms); 1024x2048 gains nothing with one right-hand side (54.1 -> 54.3 cold: fewer FP64
// instructions, but 80 registers leave a third of the warps; the pipe is 52-70 % busy, 79 % with two).
// n consecutive values of a row (one, or an even number at a 16-byte boundary)
template <int n>
__device__ __forceinline__ void row_ld(const double* __restrict__ p, double* o) {
    if constexpr (n == 1) {
        o[0] = p[0];
    } else {
#pragma unroll
        for (int q = 0; q < n; q += 2) {
            const double2 v = *reinterpret_cast<const double2*>(p + q);
            o[q] = v.x;
            o[q + 1] = v.y;
        }
    }
}

constexpr int IR_THREADS = 128;
template <int NR, int W>
__global__ void __launch_bounds__(IR_THREADS) k_ir_residual(Lev<double> L, const double* __restrict__ b,
                                                      const double* __restrict__ x, float* __restrict__ r32,
                                                      float* __restrict__ e32, SolveState* st, double* partial,
                                                      unsigned* ticket, cudaGraphConditionalHandle ho,
                                                      cudaGraphConditionalHandle hi, int use_h, int set_hi,
                                                      unsigned* coop_bar, int R) {
    // the whole-solve cooperative launch that follows counts its barrier arrivals from 0 (its
    // previous launch has completed: stream order)
    if (coop_bar && blockIdx.x == 0 && blockIdx.z == 0 && threadIdx.x == 0) *coop_bar = 0u;
    const long long zo = zoff(L.zs);
    L.diag = zsh(L.diag, zo);
    L.wl = zsh(L.wl, zo);
    L.wb = zsh(L.wb, zo);
    b = zsh(b, zo);
    x = zsh(x, zo);
    r32 = zsh(r32, zo);
    e32 = zsh(e32, zo);
    st = zsh(st, zo);
    partial = zsh(partial, zo);
    ticket = zsh(ticket, zo);
    double sc[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) sc[k] = ld_now(&st->scale_next[k]);
    if (ld_now(&st->odone)) return;
    int N = L.nx * L.ny;
    // the inner FP32 system is solved for s r, s = 2^k a power of two that brings the residual's
    // cell values to order one, set from the previous residual norm (of b on the first pass) by
    // the launch that computed it: the same in every block.  The FP32 copy is rounded from
    // r 2^k on the integer pipes and the norm is summed from that copy (a thread's FP32-pair sum,
    // then FP64; relative accuracy about 1e-7, ample for the convergence test), so the FP64 pipe
    // carries the residual alone.
    int ksc[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) {
        ksc[k] = (int)((__double_as_longlong(sc[k]) >> 52) & 0x7ff) - 1023;
    }
    const int nq = L.nx / W, u = blockIdx.x * IR_THREADS + threadIdx.x;
    const int m = u % nq, j0 = u / nq * R, j1 = min(j0 + R, L.ny);
    DotAcc<float, NR> acc;
    if (j0 < L.ny) {
        constexpr int V = W * NR;
        const int c0 = j0 * L.nx + m * W;
        const bool lft = m > 0, rgt = m < nq - 1;
        // xc: the row's x; dv: its differences to the row below, dv = x_below - x (the sign of the
        // row below's own term); wb: the weights of the faces between
        double xc[V], dv[V], wb[W];
        row_ld<V>(x + (size_t)c0 * NR, xc);
#pragma unroll
        for (int q = 0; q < W; ++q) wb[q] = 0.0;
#pragma unroll
        for (int q = 0; q < V; ++q) dv[q] = 0.0;
        if (j0 > 0) {
            double xd[V];
            row_ld<V>(x + (size_t)(c0 - L.nx) * NR, xd);
            row_ld<W>(L.wb + c0, wb);
#pragma unroll
            for (int q = 0; q < V; ++q) dv[q] = xd[q] - xc[q];
        }
#pragma unroll 2
        for (int j = j0, c = c0; j < j1; ++j, c += L.nx) {
            double xu[V], wt[W], wl[W + 1], dg[W], bv[V], xl[NR], xr[NR];
            const bool up = j + 1 < L.ny;
#pragma unroll
            for (int q = 0; q < W; ++q) wt[q] = 0.0;
#pragma unroll
            for (int q = 0; q < V; ++q) xu[q] = xc[q];
            if (up) {
                row_ld<V>(x + (size_t)(c + L.nx) * NR, xu);
                row_ld<W>(L.wb + c + L.nx, wt);
            }
            row_ld<W>(L.diag + c, dg);
            row_ld<W>(L.wl + c, wl);
            row_ld<V>(b + (size_t)c * NR, bv);
            // the faces on the grid's sides: weight 0, difference 0
            if (!lft) wl[0] = 0.0;
            wl[W] = rgt ? L.wl[c + W] : 0.0;
#pragma unroll
            for (int k = 0; k < NR; ++k) {
                xl[k] = lft ? x[(size_t)(c - 1) * NR + k] : xc[k];
                xr[k] = rgt ? x[(size_t)(c + W) * NR + k] : xc[V - NR + k];
            }
            double s[V];   // A x in flux form
#pragma unroll
            for (int q = 0; q < V; ++q) s[q] = dg[q / NR] * xc[q];
            double h[V + NR];
#pragma unroll
            for (int q = 0; q < V; ++q) h[q] = xc[q] - (q < NR ? xl[q] : xc[q - NR]);
#pragma unroll
            for (int k = 0; k < NR; ++k) h[V + k] = xr[k] - xc[V - NR + k];
            alignas(16) float rf[V], ez[V];
#pragma unroll
            for (int q = 0; q < V; ++q) {
                s[q] = fma(wl[q / NR], h[q], s[q]);
                s[q] = fma(wl[q / NR + 1], -h[q + NR], s[q]);
                s[q] = fma(wb[q / NR], -dv[q], s[q]);
                dv[q] = xc[q] - xu[q];
                s[q] = fma(wt[q / NR], dv[q], s[q]);
                rf[q] = d2f_rn2(bv[q] - s[q], ksc[q % NR]);
                acc.add(q % NR, rf[q], rf[q]);
                ez[q] = 0.0f;
                xc[q] = xu[q];
            }
#pragma unroll
            for (int q = 0; q < W; ++q) wb[q] = wt[q];
            using F = Vec<float, V % 4 == 0 ? 4 : V>;
#pragma unroll
            for (int q = 0; q < V; q += sizeof(F) / 4) {
                *reinterpret_cast<F*>(r32 + (size_t)c * NR + q) = *reinterpret_cast<const F*>(rf + q);
                *reinterpret_cast<F*>(e32 + (size_t)c * NR + q) = *reinterpret_cast<const F*>(ez + q);
            }
        }
        acc.flush();
    }
    // the block's sum: over its warps lane by lane, then one warp's tree (a tree per warp would be a
    // tenth of the kernel's FP64 instructions)
    __shared__ double sh[NR][IR_THREADS];
#pragma unroll
    for (int k = 0; k < NR; ++k) sh[k][threadIdx.x] = acc.tot[k];
    __syncthreads();
    const int vb = gridDim.x;
    if (threadIdx.x < 32 * NR) {
        const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
        double a = sh[k][lane];
#pragma unroll
        for (int w = 1; w < IR_THREADS / 32; ++w) a += sh[k][lane + 32 * w];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
        if (lane == 0) partial[k * vb + blockIdx.x] = a;
    }
    __syncthreads();
    double tot[NR];
    if (last_block_total<NR>(partial, vb, ticket, tot)) {
        bool done = true;
        for (int k = 0; k < 2; ++k) {
            double s2 = k < NR ? sc[k] * sc[k] : 1.0;   // a power of two: the divisions are exact
            double rr = k < NR ? tot[k] / s2 : 0.0;
            st->orr[k] = rr;
            if (!(rr <= st->otol2[k])) done = false;
            if (!isfinite(rr) || !isfinite(st->obb[k])) st->nonfinite = 1;
            st->scale[k] = k < NR ? sc[k] : 1.0;
            st->scale_next[k] = unit_scale(rr, N);
            st->rr[k] = k < NR ? tot[k] : 0.0;
            // the inner solve reduces the residual by inner_rtol, but never below half the
            // outer target: no solve past what the refinement needs (in the scaled units)
            st->tol2[k] = fmax(st->inner_rtol * st->inner_rtol * rr, 0.25 * st->otol2[k]) * s2;
            st->rz[k] = 0.0;
            st->beta[k] = 0.0;
        }
        st->oiters += 1;
        st->itot += st->iters;
        if (st->oiters > st->max_outer || st->nonfinite) done = true;
        st->odone = done ? 1 : 0;
        st->iters = 0;
        st->done = done ? 1 : 0;
        set_cond(ho, use_h, done ? 0u : 1u);
        if (set_hi) set_cond(hi, use_h, done ? 0u : 1u);
    }
}

template <int NR>
__global__ void k_ir_update(int N, long long zs, double* __restrict__ x, const float* __restrict__ e,
                            const SolveState* st) {
    const long long zo = zoff(zs);
    x = zsh(x, zo);
    e = zsh(e, zo);
    st = zsh(st, zo);
    const double s0 = ld_now(&st->scale[0]), s1 = NR > 1 ? ld_now(&st->scale[1]) : s0;
    if (ld_now(&st->odone)) return;
    // powers of two: exact; an even element belongs to the first right-hand side
    const double inv0 = 1.0 / s0, inv1 = NR > 1 ? 1.0 / s1 : inv0;
    const long long n = (long long)N * NR;
    const int t = blockIdx.x * blockDim.x + threadIdx.x, T = gridDim.x * blockDim.x;
    // four elements per step (one 16-byte load of e, two of x) where both arrays allow it
    const bool vec = ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(e)) & 15u) == 0;
    const long long n4 = vec ? n / 4 : 0;
#pragma unroll 2
    for (long long q = t; q < n4; q += T) {
        float4 ev = reinterpret_cast<const float4*>(e)[q];
        double2* xp = reinterpret_cast<double2*>(x) + 2 * q;
        double2 a = xp[0], b = xp[1];
        a.x += f2d(ev.x) * inv0;
        a.y += f2d(ev.y) * inv1;
        b.x += f2d(ev.z) * inv0;
        b.y += f2d(ev.w) * inv1;
        xp[0] = a;
        xp[1] = b;
    }
    for (long long c = 4 * n4 + t; c < n; c += T) x[c] += f2d(e[c]) * ((c & 1) ? inv1 : inv0);
}

// ---------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------
static inline int nblocks(long long n) {
    long long b = (n + RB - 1) / RB;
    return (int)(b < NRED ? (b < 1 ? 1 : b) : NRED);
}
// Blocks per instance of a launch over nz instances.  The reduction kernels are written for
// nblocks(n) blocks per instance (their virtual blocks, a function of the grid alone) and run
// them on this many real blocks, each taking the virtual blocks b, b + launch, ...: the same cells
// in the same order into the same slots, so that an instance's sums do not depend on how many
// instances share the launch.  One instance keeps one real block per virtual block; a batch
// gets about two blocks per SM slot in total (NRED = 4 per SM), instead of thousands of blocks
// that each reduce a few hundred cells.
static inline int lblocks(long long n, int nz) {
    int v = nblocks(n);
    int per = (2 * NRED) / (nz > 0 ? nz : 1);
    return nz <= 1 ? v : (v < per ? v : (per < 1 ? 1 : per));
}

void Solver::plan(int nx_, int ny_) {
    nx = nx_;
    ny = ny_;
    nlev = 0;
    int x = nx, y = ny;
    size_t off = 0;
    while (true) {
        lnx[nlev] = x;
        lny[nlev] = y;
        loff[nlev] = off;
        off += (size_t)x * y;
        ++nlev;
        if (nlev == MAXLEV) break;
        if ((x & 1) || (y & 1) || (long long)x * y <= 16 || x < 2 || y < 2) break;
        x /= 2;
        y /= 2;
    }
    ncells_all = off;
    if (small_max_f <= 0) small_max_f = SMALL_MAX_F;
    nbig_f = 0;
    while (nbig_f < nlev - 1 && (long long)lnx[nbig_f] * lny[nbig_f] > small_max_f) ++nbig_f;
    nbig_d = 0;
    while (nbig_d < nlev - 1 && (long long)lnx[nbig_d] * lny[nbig_d] > SMALL_MAX_D) ++nbig_d;
    nbig = nbig_f;
}

static size_t tiles(int nx, int ny) { return (size_t)((nx + TX - 1) / TX) * ((ny + TY - 1) / TY); }

size_t Solver::bytes(int nx, int ny) {
    Solver s;
    s.plan(nx, ny);
    size_t total = 0;
    auto add = [&](size_t b) { total += (b + 255) & ~size_t(255); };
    size_t A = s.ncells_all, N = (size_t)nx * ny;
    for (int k = 0; k < 5; ++k) add(A * 4);
    for (int k = 0; k < 5; ++k) add(A * 8);
    add(A * 2 * 4); add(A * 2 * 4); add(A * 2 * 4);
    add(A * 2 * 8); add(A * 2 * 8); add(A * 2 * 8);
    add(N * 2 * 4); add(N * 4 * 4); add(N * 2 * 4); add(N * 2 * 4);
    add(N * 2 * 8); add(N * 4 * 8); add(N * 2 * 8);
    add(1040 * 4); add(1040 * 8);
    size_t mb = tiles(nx, ny) > (size_t)NRED ? tiles(nx, ny) : (size_t)NRED;
    add(mb * 4 * 8);
    add(256);
    add(NSLOT * sizeof(SolveState));
    add(4 * sizeof(KTimer));
    return total;
}

template <typename K>
static void allow_smem(K kern, int bytes, cudaError_t* first) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess && *first == cudaSuccess) *first = e;
}

cudaError_t Solver::bind(void* base, int nx_, int ny_, bool make_streams, cudaStream_t init_stream) {
    plan(nx_, ny_);
    tma_ready = false;   // descriptors hold addresses: re-encode after every binding
    char* p = (char*)base;
    auto take = [&](size_t b) { void* r = p; p += (b + 255) & ~size_t(255); return r; };
    size_t A = ncells_all, N = (size_t)nx * ny;
    f_diag = (float*)take(A * 4); f_wl = (float*)take(A * 4); f_wb = (float*)take(A * 4);
    f_cd = (float*)take(A * 4); f_dd = (float*)take(A * 4);
    d_diag = (double*)take(A * 8); d_wl = (double*)take(A * 8); d_wb = (double*)take(A * 8);
    d_cd = (double*)take(A * 8); d_dd = (double*)take(A * 8);
    f_x = (float*)take(A * 2 * 4); f_b = (float*)take(A * 2 * 4); f_x2 = (float*)take(A * 2 * 4);
    d_x = (double*)take(A * 2 * 8); d_b = (double*)take(A * 2 * 8); d_x2 = (double*)take(A * 2 * 8);
    f_r = (float*)take(N * 2 * 4); f_p = (float*)take(N * 4 * 4); f_q = (float*)take(N * 2 * 4);
    f_e = (float*)take(N * 2 * 4);
    d_r = (double*)take(N * 2 * 8); d_p = (double*)take(N * 4 * 8); d_q = (double*)take(N * 2 * 8);
    f_inv = (float*)take(1040 * 4); d_inv = (double*)take(1040 * 8);
    size_t mb = tiles(nx, ny) > (size_t)NRED ? tiles(nx, ny) : (size_t)NRED;
    partial = (double*)take(mb * 4 * 8);
    tickets = (unsigned*)take(256);
    st_base = (SolveState*)take(NSLOT * sizeof(SolveState));
    st = st_base;
    timer = (KTimer*)take(4 * sizeof(KTimer));
    if (make_streams)
        for (int k = 0; k < 3; ++k) cudaStreamCreateWithFlags(&aux[k], cudaStreamNonBlocking);
    // shared-memory opt-in of the tile kernels, and of those that run the single-block levels (2048 x 2
    // cells with two right-hand sides take 204864 bytes; dynamic + static may pass 48 KB)
    const int SM = 200 * 1024, SML = (int)SMEM_MAX;
    cudaError_t err = cudaSuccess;
    allow_smem(k_pre<float, 1>, SM, &err);
    allow_smem(k_pre<float, 2>, SM, &err);
    allow_smem(k_pre<double, 1>, SM, &err);
    allow_smem(k_pre<double, 2>, SM, &err);
    allow_smem(k_post<float, 1, true>, SM, &err);
    allow_smem(k_post<float, 1, false>, SM, &err);
    allow_smem(k_post<float, 2, true>, SM, &err);
    allow_smem(k_post<float, 2, false>, SM, &err);
    allow_smem(k_post<double, 1, true>, SM, &err);
    allow_smem(k_post<double, 1, false>, SM, &err);
    allow_smem(k_post<double, 2, true>, SM, &err);
    allow_smem(k_post<double, 2, false>, SM, &err);
    allow_smem(k_coarse_cycle<float, 1>, SML, &err);
    allow_smem(k_coarse_cycle<float, 2>, SML, &err);
    allow_smem(k_coarse_cycle<double, 1>, SML, &err);
    allow_smem(k_coarse_cycle<double, 2>, SML, &err);
    allow_smem(k_cg_persist<float, 1>, SML, &err);
    allow_smem(k_cg_persist<float, 2>, SML, &err);
    allow_smem(k_small<float, 1, true>, SML, &err);
    allow_smem(k_small<float, 1, false>, SML, &err);
    allow_smem(k_small<float, 2, true>, SML, &err);
    allow_smem(k_small<float, 2, false>, SML, &err);
    allow_smem(k_small<double, 1, true>, SML, &err);
    allow_smem(k_small<double, 1, false>, SML, &err);
    allow_smem(k_small<double, 2, true>, SML, &err);
    allow_smem(k_small<double, 2, false>, SML, &err);
    // device state that must start at zero (tickets, solve states, timers; timer starts at ~0)
    cudaError_t e[4];
    e[0] = cudaMemsetAsync(timer, 0, 4 * sizeof(KTimer), init_stream);
    e[1] = cudaSuccess;
    for (int k = 0; k < 4; ++k) {
        cudaError_t ek = cudaMemsetAsync(&timer[k].start, 0xff, sizeof(unsigned long long), init_stream);
        if (ek != cudaSuccess) e[1] = ek;
    }
    e[2] = cudaMemsetAsync(tickets, 0, 256, init_stream);
    e[3] = cudaMemsetAsync(st_base, 0, NSLOT * sizeof(SolveState), init_stream);
    for (int k = 0; k < 4 && err == cudaSuccess; ++k) err = e[k];
    timing = 1;
    return err;
}

// accessors for precision T
template <typename T> struct PT;
template <> struct PT<float> {
    static float* diag(Solver& s) { return s.f_diag; }
    static float* wl(Solver& s) { return s.f_wl; }
    static float* wb(Solver& s) { return s.f_wb; }
    static float* cd(Solver& s) { return s.f_cd; }
    static float* dd(Solver& s) { return s.f_dd; }
    static float* x(Solver& s) { return s.f_x; }
    static float* x2(Solver& s) { return s.f_x2; }
    static float* inv(Solver& s) { return s.f_inv; }
    static float* b(Solver& s) { return s.f_b; }
    static float* r(Solver& s) { return s.f_r; }
    static constexpr int prec = 1;
};
template <> struct PT<double> {
    static double* diag(Solver& s) { return s.d_diag; }
    static double* wl(Solver& s) { return s.d_wl; }
    static double* wb(Solver& s) { return s.d_wb; }
    static double* cd(Solver& s) { return s.d_cd; }
    static double* dd(Solver& s) { return s.d_dd; }
    static double* x(Solver& s) { return s.d_x; }
    static double* x2(Solver& s) { return s.d_x2; }
    static double* inv(Solver& s) { return s.d_inv; }
    static double* b(Solver& s) { return s.d_b; }
    static double* r(Solver& s) { return s.d_r; }
    static constexpr int prec = 0;
};

// the FP64 levels' reciprocal diagonals, in the storage of the levels' Dirichlet terms (read by the
// set-up alone)
template <typename T> static T* id_of(Solver& s);
template <> float* id_of<float>(Solver&) { return nullptr; }
template <> double* id_of<double>(Solver& s) { return s.d_dd; }

// ---- TMA descriptors (host) ----------------------------------------------------------------
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn tensor_map_encoder() {
    static EncodeTiledFn fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)f;
        else
            cudaGetLastError();
    }
    return fn;
}

// a 2-D row-major array of w x h elements of T, copied in boxes of bw x bh; false when the base
// or the row pitch is not 16-byte aligned or the encoder refuses
template <typename T>
static bool encode_2d(CUtensorMap* m, const void* base, int w, int h, int bw, int bh) {
    EncodeTiledFn fn = tensor_map_encoder();
    if (!fn || (uintptr_t)base % 16 != 0 || ((size_t)w * sizeof(T)) % 16 != 0) return false;
    cuuint64_t dims[2] = {(cuuint64_t)w, (cuuint64_t)h};
    cuuint64_t pitch[1] = {(cuuint64_t)w * sizeof(T)};
    cuuint32_t box[2] = {(cuuint32_t)bw, (cuuint32_t)bh};
    cuuint32_t es[2] = {1, 1};
    CUtensorMapDataType dt = sizeof(T) == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT64;
    return fn(m, dt, 2, const_cast<void*>(base), dims, pitch, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
           CUDA_SUCCESS;
}

static size_t tmap_index(int prec, int nr, int l, int post) {
    return ((size_t)(prec * 2 + (nr - 1)) * Solver::MAXLEV + l) * 2 + post;
}

template <typename T, int NR, bool POST>
static bool encode_tile_maps(Solver& s, int l, TileMaps& M) {
    constexpr int H = POST ? HPOST : HPRE;
    using Sg = Stage<T, NR, H, POST>;
    int nx = s.lnx[l], ny = s.lny[l];
    size_t o = s.loff[l];
    const T* b = l == 0 ? PT<T>::r(s) : PT<T>::b(s) + 2 * o;
    bool ok = encode_2d<T>(&M.d, PT<T>::diag(s) + o, nx, ny, Sg::BWS, Sg::BHS) &&
              (sizeof(T) == 4 || encode_2d<T>(&M.id, id_of<T>(s) + o, nx, ny, Sg::BWS, Sg::BHS)) &&
              encode_2d<T>(&M.wl, PT<T>::wl(s) + o, nx, ny, Sg::BWS, Sg::BHS) &&
              encode_2d<T>(&M.wb, PT<T>::wb(s) + o, nx, ny, Sg::BWS, Sg::BHS) &&
              encode_2d<T>(&M.b, b, nx * NR, ny, Sg::BWV * NR, Sg::BHV);
    if (POST)
        ok = ok && encode_2d<T>(&M.xin, PT<T>::x2(s) + 2 * o, nx * NR, ny, Sg::BWV * NR, Sg::BHV) &&
             encode_2d<T>(&M.xc, PT<T>::x(s) + 2 * s.loff[l + 1], s.lnx[l + 1] * NR, s.lny[l + 1], Sg::BWC * NR,
                          Sg::BHC);
    return ok;
}

template <typename T>
static void encode_precision(Solver& s, int nbig) {
    for (int l = 0; l < nbig; ++l) {
        int p = PT<T>::prec;
        s.tma_ok[tmap_index(p, 1, l, 0)] = encode_tile_maps<T, 1, false>(s, l, s.tmaps[tmap_index(p, 1, l, 0)]);
        s.tma_ok[tmap_index(p, 1, l, 1)] = encode_tile_maps<T, 1, true>(s, l, s.tmaps[tmap_index(p, 1, l, 1)]);
        s.tma_ok[tmap_index(p, 2, l, 0)] = encode_tile_maps<T, 2, false>(s, l, s.tmaps[tmap_index(p, 2, l, 0)]);
        s.tma_ok[tmap_index(p, 2, l, 1)] = encode_tile_maps<T, 2, true>(s, l, s.tmaps[tmap_index(p, 2, l, 1)]);
    }
}

// descriptors of every tiled level, both precisions and right-hand-side counts (host work only)
static void ensure_tile_maps(Solver& s) {
    if (s.tma_ready) return;
    size_t n = tmap_index(1, 2, Solver::MAXLEV - 1, 1) + 1;
    s.tmaps.assign(n, TileMaps{});
    s.tma_ok.assign(n, 0);
    encode_precision<float>(s, s.nbig_f);
    encode_precision<double>(s, s.nbig_d);
    s.tma_ready = true;
}

template <typename T>
static Lev<T> lev(Solver& s, int l) {
    size_t o = s.loff[l];
    const T* id = id_of<T>(s);
    return {s.lnx[l], s.lny[l], PT<T>::diag(s) + o, PT<T>::wl(s) + o, PT<T>::wb(s) + o, s.zs, id ? id + o : nullptr};
}

template <typename T>
static void setup_levels(Solver& s, const double* cd, const double* dd, const double* wl, const double* wb,
                         double* d64, cudaStream_t stm) {
    SetupPlan P;
    P.zs = s.zs;
    P.nlev = s.nlev;
    for (int l = 0; l < s.nlev; ++l) { P.nx[l] = s.lnx[l]; P.ny[l] = s.lny[l]; P.off[l] = s.loff[l]; }
    if ((long long)s.nx * s.ny > (1LL << 21)) {
        constexpr int SB = 64;
        dim3 grid((s.nx + SB - 1) / SB, (s.ny + SB - 1) / SB, s.nz);
        k_setup_tree<T, SB><<<grid, 256, 0, stm>>>(P, cd, dd, wl, wb, PT<T>::diag(s), PT<T>::wl(s), PT<T>::wb(s),
                                                   PT<T>::cd(s), PT<T>::dd(s), d64, PT<T>::inv(s), s.tickets + 6);
    } else {
        constexpr int SB = 32;
        dim3 grid((s.nx + SB - 1) / SB, (s.ny + SB - 1) / SB, s.nz);
        k_setup_tree<T, SB><<<grid, 256, 0, stm>>>(P, cd, dd, wl, wb, PT<T>::diag(s), PT<T>::wl(s), PT<T>::wb(s),
                                                   PT<T>::cd(s), PT<T>::dd(s), d64, PT<T>::inv(s), s.tickets + 6);
    }
    ++s.launches;
    if constexpr (sizeof(T) == 8) {
        k_diag_inverse<<<dim3(lblocks(s.nx * (long long)s.ny, s.nz), 1, s.nz), RB, 0, stm>>>(
            P, PT<T>::diag(s), PT<T>::wl(s), PT<T>::wb(s), id_of<T>(s));
        ++s.launches;
    }
}

// z = M r: r is the level-0 rhs, z the level-0 output (both NR-interleaved)
template <typename T> static int nbig_of(const Solver& s);
template <> int nbig_of<float>(const Solver& s) { return s.nbig_f; }
template <> int nbig_of<double>(const Solver& s) { return s.nbig_d; }

template <typename T>
static SmallPlan small_plan(const Solver& s, int first = -1) {
    SmallPlan P;
    P.zs = s.zs;
    int nb = first >= 0 ? first : nbig_of<T>(s);
    P.n = s.nlev - nb;
    int so = 0, xo = 0;
    for (int k = 0; k < P.n; ++k) {
        int l = nb + k;
        P.nx[k] = s.lnx[l];
        P.ny[k] = s.lny[l];
        P.soff[k] = so;
        P.xoff[k] = xo;
        P.goff[k] = s.loff[l];
        so += s.lnx[l] * s.lny[l];
        xo += (2 * x_entries((s.lnx[l] + 1) / 2, (s.lny[l] + 1) & ~1) + 3) & ~3;
    }
    P.cells = so;
    P.total = (so + 3) & ~3;   // (a multiple of 16 bytes in every array)
    P.xtotal = xo;
    return P;
}

// shared memory of the cooperative coarse cycle: the larger of the tile regions and the
// single-block levels
template <typename T, int NR>
static size_t coarse_smem(const SmallPlan& P) {
    size_t a = Region<T, NR, HPRE>::bytes(), b = Region<T, NR, HPOST>::bytes();
    size_t c = SmallMem<T, NR>::bytes(P);
    size_t m = a > b ? a : b;
    return m > c ? m : c;
}

// first tiled level of the cooperative coarse cycle (nb: none).  A level joins when its tiles
// fit one per co-resident block; the finest level stays separate (its post-smoothing carries
// the r.z of CG).  Single instances only.
template <typename T, int NR>
static int coarse_start(Solver& s) {
    int nb = nbig_of<T>(s);
    if (!s.use_coop || s.nz != 1 || nb < 2) return nb;
    static int resident[2][2] = {{-1, -1}, {-1, -1}};
    int& res = resident[PT<T>::prec][NR - 1];
    if (res < 0) {
        int dev = 0, sms = 0, per = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        size_t smem = Region<T, NR, HPRE>::bytes() > Region<T, NR, HPOST>::bytes()
                          ? Region<T, NR, HPRE>::bytes()
                          : Region<T, NR, HPOST>::bytes();
        smem = smem > SmallMem<T, NR>::bytes(SMALL_CELLS, SMALL_XENTRIES) ? smem
                                                                          : SmallMem<T, NR>::bytes(SMALL_CELLS, SMALL_XENTRIES);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_coarse_cycle<T, NR>, CC_THREADS, smem);
        res = per * sms;
        cudaGetLastError();
    }
    for (int l = 1; l < nb; ++l)
        if ((long long)((s.lnx[l] + TX - 1) / TX) * ((s.lny[l] + TY - 1) / TY) <= res) return l;
    return nb;
}

// whether the current device takes a cluster of CL_BLOCKS blocks of the kernel (asked once per
// device and kernel slot)
static bool cluster_usable(const void* kern, int slot) {
    static std::atomic<int> usable[64][8];   // 0 not asked, 1 yes, 2 no
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return false;
    std::atomic<int>& u = usable[dev][slot];
    if (u.load() == 0) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(CL_BLOCKS);
        cfg.blockDim = dim3(CL_THREADS);
        cfg.dynamicSmemBytes = SMEM_MAX;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = CL_BLOCKS;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
        u.store(e == cudaSuccess && n > 0 ? 1 : 2);
        if (e != cudaSuccess) cudaGetLastError();
    }
    return u.load() == 1;
}

// threads that the single-block levels from ls on want (one block of cells per thread; the
// coarsest FP64 one may have two)
template <typename T, int NR>
static int small_threads(const Solver& s, int ls) {
    int need = 32;
    if (ls < s.nlev - 1) need = Blk<T, NR>::units(s.lnx[ls], s.lny[ls]);
    const int uc = Blk<T, NR>::units(s.lnx[s.nlev - 1], s.lny[s.nlev - 1]);
    return std::max(need, sizeof(T) == 8 ? (uc + 1) / 2 : uc);
}
// first level that block 0 of the cluster runs alone
template <typename T>
static int cluster_small(const Solver& s, int nb) {
    int ls = nb;
    if (sizeof(T) == 8)
        while (ls < s.nlev - 1 && s.lnx[ls] * s.lny[ls] > 256) ++ls;
    return ls;
}

// Plan of the cluster launch: the first tiled level l0 >= 1 from which every level fits the
// cluster's shared memory and threads (l0 = nb: none; the finest level stays separate, its
// post-smoothing carries the r.z of CG).  In FP64, where a half-sweep of 32 x 32 cells takes one
// SM 0.8 us of FP64 issue against 0.45 us over the cluster, the levels above 256 cells stay in the
// cluster; in FP32 those above the single-block size (block 0 has a thread for each block of that
// level's cells or there is no plan: with a single-block size of 4096 cells a first level of more than
// 2048 takes the grid-barrier launch).  Single instances; a bound set for the grid barriers
// (EBIT_OPT_BARRIER_SPIN) asks for the grid-barrier launch.
template <typename T, int NR>
static int cluster_plan(Solver& s, ClPlan& P, int& threads, size_t& smem) {
    const int nb = nbig_of<T>(s);
    if (!s.use_coop || s.barrier_spin > 0 || s.nz != 1 || nb < 2) return nb;
    if (!cluster_usable((const void*)k_coarse_cluster<T, NR>, PT<T>::prec * 2 + NR - 1)) return nb;
    const int ls = cluster_small<T>(s, nb), half = CL_THREADS / 2, need_s = small_threads<T, NR>(s, ls);
    P.S = small_plan<T>(s, ls);
    for (int l0 = 1; l0 < nb; ++l0) {
        if (ls - l0 > CL_MAX) continue;
        size_t off = 0;
        int need = need_s;
        P.nl = ls - l0;
        P.nt = nb - l0;
        for (int k = 0; k < P.nl; ++k) {
            const int l = l0 + k;
            P.nx[k] = s.lnx[l];
            P.ny[k] = s.lny[l];
            P.rp[k] = 2 * ((s.lny[l] / 2 + CL_BLOCKS - 1) / CL_BLOCKS);
            P.goff[k] = s.loff[l];
            P.off[k] = (int)off;
            if ((long long)P.rp[k] * P.nx[k] > 16 * CL_THREADS) {
                off = SMEM_MAX + 1;
                break;
            }
            off += ClMem<T, NR>::bytes(P.nx[k], P.rp[k]);
            // two blocks of cells per thread at most (one on the FP64 levels below the tiled ones)
            const int u = Blk<T, NR>::units(P.nx[k], P.rp[k]);
            if (u > (k < P.nt ? 2 : 1) * CL_THREADS) off = SMEM_MAX + 1;
            need = std::max(need, std::min(u, CL_THREADS));
        }
        P.soff = (int)off;
        smem = off + SmallMem<T, NR>::bytes(P.S);
        if (smem > SMEM_MAX || need_s > CL_THREADS) continue;
        threads = need > half ? CL_THREADS : half;
        return l0;
    }
    return nb;
}

// Plan of the whole-solve cluster kernel; false where the grid does not fit it (or the separate
// launches are asked for: EBIT_OPT_COOP 0, a barrier bound, smoother timing, a batch)
template <typename T, int NR>
static bool cg_plan(Solver& s, CgPlan& G, int& threads, size_t& smem) {
    const int nb = nbig_of<T>(s);
    if (!s.use_coop || s.barrier_spin > 0 || s.nz != 1 || !s.use_cgc || nb < 1) return false;
    const int nx = s.nx, ny = s.ny;
    // 16 blocks then have more work than launches cost: a 160x160 mixed step took 930 us separate, 940 whole
    if ((long long)nx * ny > 16384) return false;
    if (!cluster_usable((const void*)k_cg_cluster<T, NR>, 4 + PT<T>::prec * 2 + NR - 1)) return false;
    ClPlan& P = G.C;
    const int ls = cluster_small<T>(s, nb);
    if (ls > CL_MAX) return false;
    P.S = small_plan<T>(s, ls);
    P.nl = ls;
    P.nt = nb;
    G.unit = sizeof(T) == 8 ? 1 : NR == 2 ? 2 : nx % 4 == 0 ? 4 : 1;   // as cg_body chooses its kernels
    G.nslot = (nx * ny / G.unit + 255) / 256;
    G.ngrp = 8 * G.nslot;
    if (G.nslot > 64) return false;
    int need = small_threads<T, NR>(s, ls);
    size_t off = 0;
    for (int l = 0; l < ls; ++l) {
        P.nx[l] = s.lnx[l];
        P.ny[l] = s.lny[l];
        P.rp[l] = 2 * ((s.lny[l] / 2 + CL_BLOCKS - 1) / CL_BLOCKS);
        // level 0: a slab starts at a group of 32 units of the reductions
        while (l == 0 && (long long)P.rp[0] * nx % (32 * G.unit) != 0) P.rp[0] += 2;
        P.goff[l] = s.loff[l];
        P.off[l] = (int)off;
        off += ClMem<T, NR>::bytes(P.nx[l], P.rp[l]);
        need = std::max(need, Blk<T, NR>::units(P.nx[l], P.rp[l]));
        if (need > CL_THREADS || off > SMEM_MAX) return false;
    }
    threads = need > CL_THREADS / 2 ? CL_THREADS : CL_THREADS / 2;
    P.soff = (int)off;
    off += (SmallMem<T, NR>::bytes(P.S) + 127) & ~size_t(127);
    auto take = [&](size_t bytes) {
        const int o = (int)off;
        off += (bytes + 127) & ~size_t(127);
        return o;
    };
    G.tx = (nx + TX - 1) / TX;
    G.nt = G.tx * ((ny + TY - 1) / TY);
    if (G.nt > 64) return false;
    G.tslots = (G.nt + CL_BLOCKS - 1) / CL_BLOCKS;
    G.p_off = take(sizeof(T) * NR * ClMem<T, NR>::xn(nx, P.rp[0]));
    G.x_off = take(sizeof(T) * NR * Blk<T, NR>::CELLS * threads);
    // (these are cleared by the kernel as one range)
    G.pstride = (P.rp[0] * nx / G.unit / 32 + 1) * CG_GRP;
    G.prod_off = take(sizeof(double) * NR * G.pstride);
    G.w_off = take(sizeof(double) * 2 * NR * G.ngrp);
    G.tb_off = take(sizeof(T) * G.tslots * NR * 256);
    G.tw_off = take(sizeof(T) * G.tslots * NR * 16);
    G.ts_off = take(sizeof(double) * NR * 64);
    smem = off;
    return smem <= SMEM_MAX;
}
template <typename T, int NR>
static void launch_cg(Solver& s, const CgPlan& G, int threads, size_t smem, const T* r, T* x, cudaStream_t stm) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CL_BLOCKS);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stm;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL_BLOCKS;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_cg_cluster<T, NR>, G, (const T*)PT<T>::diag(s), (const T*)id_of<T>(s),
                       (const T*)PT<T>::wl(s), (const T*)PT<T>::wb(s), (const T*)PT<T>::inv(s), r, x, s.st);
}

// blocks of a persistent (TMA-staged) tile launch: one per tile, at most as many as are resident
// on the device at once (cached per kernel and shared-memory size)
static int persistent_blocks(const void* kern, int threads, size_t smem, int tiles) {
    struct Entry {
        const void* k;
        size_t smem;
        int dev, blocks;
    };
    thread_local std::vector<Entry> cache;
    int dev = 0;
    cudaGetDevice(&dev);
    int resident = 0;
    for (const Entry& e : cache)
        if (e.k == kern && e.smem == smem && e.dev == dev) resident = e.blocks;
    if (resident == 0) {
        int sms = 0, per = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, threads, smem);
        resident = per > 0 && sms > 0 ? per * sms : 1;
        cudaGetLastError();
        cache.push_back({kern, smem, dev, resident});
    }
    return tiles < resident ? tiles : resident;
}

// z = M r: r is the level-0 rhs, z the level-0 output (both NR-interleaved).
// k_pre of level l writes the pre-smoothed x into X2_l; k_post of level l reads X2_l and the
// coarse correction X_{l+1} (halo included) and writes the final x into X_l (z at level 0):
// no kernel writes an array that another of its blocks still reads.
template <typename T, int NR>
static void vcycle(Solver& s, const T* r, T* z, SolveState* st, cudaStream_t stm) {
    T* X = PT<T>::x(s);
    T* X2 = PT<T>::x2(s);
    T* B = PT<T>::b(s);
    const T* b = r;
    int nb = nbig_of<T>(s);
    ensure_tile_maps(s);
    const int pr = PT<T>::prec;
    ClPlan cp;
    int cthreads = 0;
    size_t csmem = 0;
    const int lc = cluster_plan<T, NR>(s, cp, cthreads, csmem);
    // tiled levels [l0, nb) go into the cluster or the cooperative launch
    const int l0 = lc < nb ? lc : coarse_start<T, NR>(s);
    for (int l = 0; l < l0; ++l) {
        Lev<T> L = lev<T>(s, l);
        dim3 grid((L.nx + TX - 1) / TX, (L.ny + TY - 1) / TY, s.nz);
        T* bc = B + 2 * s.loff[l + 1];
        size_t ix = tmap_index(pr, NR, l, 0);
        int tma = s.use_tma && s.nz == 1 && s.tma_ok[ix] && (l > 0 || r == PT<T>::r(s));
        using Rg = Region<T, NR, HPRE>;
        size_t smem = tma ? Rg::bytes() + 128 + Stage<T, NR, HPRE, false>::BYTES : Rg::bytes();
        if (tma)
            grid = dim3(persistent_blocks((const void*)k_pre<T, NR>, tile_block<HPRE>(), smem, grid.x * grid.y));
        k_pre<T, NR><<<grid, tile_block<HPRE>(), smem, stm>>>(L, b, X2 + 2 * s.loff[l], bc, st,
                                                              s.timing && l == 0 ? s.timer : nullptr,
                                                              s.tmaps[ix], tma,
                                                              l == 0 && l0 < nb && lc == nb ? s.tickets + 8 : nullptr);
        if (!s.use_graph) ++s.launches;
        b = bc;
    }
    SmallPlan P = small_plan<T>(s);
    if (lc < nb) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(CL_BLOCKS);
        cfg.blockDim = dim3(cthreads);
        cfg.dynamicSmemBytes = csmem;
        cfg.stream = stm;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = CL_BLOCKS;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cudaLaunchKernelEx(&cfg, k_coarse_cluster<T, NR>, cp, (const T*)PT<T>::diag(s), (const T*)id_of<T>(s),
                           (const T*)PT<T>::wl(s), (const T*)PT<T>::wb(s), (const T*)PT<T>::inv(s), b,
                           X + 2 * s.loff[l0], (const SolveState*)st);
        if (!s.use_graph) ++s.launches;
    } else if (l0 < nb) {
        CoarsePlan<T> C;
        C.l0 = l0;
        C.nb = nb;
        C.spin = s.barrier_spin > 0 ? s.barrier_spin : (1 << 22);
        for (int l = l0; l < nb; ++l) {
            C.L[l] = lev<T>(s, l);
            C.b[l] = l == 0 ? r : B + 2 * s.loff[l];
            C.x2[l] = X2 + 2 * s.loff[l];
            C.bc[l] = B + 2 * s.loff[l + 1];
            C.xo[l] = l == 0 ? z : X + 2 * s.loff[l];
            C.xc[l] = X + 2 * s.loff[l + 1];
        }
        C.xo[nb] = X + 2 * s.loff[nb];
        size_t smem = coarse_smem<T, NR>(P);
        int tiles = ((s.lnx[l0] + TX - 1) / TX) * ((s.lny[l0] + TY - 1) / TY);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(tiles);
        cfg.blockDim = dim3(CC_THREADS);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stm;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cudaLaunchKernelEx(&cfg, k_coarse_cycle<T, NR>, C, P, (const T*)PT<T>::diag(s), (const T*)id_of<T>(s), (const T*)PT<T>::wl(s),
                           (const T*)PT<T>::wb(s), (const T*)PT<T>::inv(s), st, s.tickets + 8);
        if (!s.use_graph) ++s.launches;
    } else {
        size_t smem = SmallMem<T, NR>::bytes(P);
        T* x = nb == 0 ? z : X + 2 * s.loff[nb];
        const T* inv = PT<T>::inv(s);
        if (nb == 0)
            k_small<T, NR, true><<<dim3(1, 1, s.nz), SMALL_THREADS, smem, stm>>>(P, PT<T>::diag(s), id_of<T>(s),
                                                                               PT<T>::wl(s), PT<T>::wb(s), inv, b, x,
                                                                               st);
        else
            k_small<T, NR, false><<<dim3(1, 1, s.nz), SMALL_THREADS, smem, stm>>>(P, PT<T>::diag(s), id_of<T>(s),
                                                                                PT<T>::wl(s), PT<T>::wb(s), inv, b, x,
                                                                                st);
        if (!s.use_graph) ++s.launches;
    }
    for (int l = l0 - 1; l >= 0; --l) {
        Lev<T> L = lev<T>(s, l);
        dim3 grid((L.nx + TX - 1) / TX, (L.ny + TY - 1) / TY, s.nz);
        const T* bl = l == 0 ? r : B + 2 * s.loff[l];
        const T* xin = X2 + 2 * s.loff[l];
        T* xout = l == 0 ? z : X + 2 * s.loff[l];
        const T* xc = X + 2 * s.loff[l + 1];
        size_t ix = tmap_index(pr, NR, l, 1);
        int tma = s.use_tma && s.nz == 1 && s.tma_ok[ix] && (l > 0 || r == PT<T>::r(s));
        using Rg = Region<T, NR, HPOST>;
        size_t smem = tma ? Rg::bytes() + 128 + Stage<T, NR, HPOST, true>::BYTES : Rg::bytes();
        KTimer* tm = s.timing && l == 0 ? s.timer + 1 : nullptr;
        if (tma) {
            const void* kern = l == 0 ? (const void*)k_post<T, NR, true> : (const void*)k_post<T, NR, false>;
            grid = dim3(persistent_blocks(kern, tile_block<HPOST>(), smem, grid.x * grid.y));
        }
        if (l == 0)
            k_post<T, NR, true><<<grid, tile_block<HPOST>(), smem, stm>>>(L, bl, xin, xout, xc, st, s.partial,
                                                                          s.tickets + 4, tm, s.tmaps[ix], tma);
        else
            k_post<T, NR, false><<<grid, tile_block<HPOST>(), smem, stm>>>(L, bl, xin, xout, xc, st, s.partial,
                                                                           s.tickets + 4, tm, s.tmaps[ix], tma);
        if (!s.use_graph) ++s.launches;
    }
}

// one CG iteration body: z = M r (+beta), p/q/alpha, x/r/test
template <typename T, int NR>
static void cg_body(Solver& s, T* x, T* r, T* z, T* p, T* q, SolveState* st, cudaGraphConditionalHandle h, int use_h,
                    cudaStream_t stm) {
    if (use_h == 2) k_cond_reset<<<1, 32, 0, stm>>>(h, h, 0);
    vcycle<T, NR>(s, r, z, st, stm);
    int N = s.nx * s.ny;
    Lev<T> L0 = lev<T>(s, 0);
    T* p1 = p + (size_t)N * NR;
    if constexpr (sizeof(T) == 4) {
        // four values per thread (four cells, or two cells of two right-hand sides) where the
        // rows and the arrays allow 16-byte accesses
        auto a16 = [](const void* ptr) { return ((uintptr_t)ptr & 15u) == 0; };
        constexpr int G = 4 / NR;   // cells per thread
        if (s.nx % G == 0 && s.zs % 16 == 0 && a16(x) && a16(r) && a16(z) && a16(p) && a16(q) && a16(L0.diag) &&
            a16(L0.wl) && a16(L0.wb)) {
            const int NQ = N / G;
            if constexpr (NR == 1)
                k_apply4<<<dim3(lblocks(NQ, s.nz), 1, s.nz), RB, 0, stm>>>(L0, z, p, p1, q, st, s.partial,
                                                                           s.tickets + 1, nblocks(NQ));
            else
                k_apply2<<<dim3(lblocks(NQ, s.nz), 1, s.nz), RB, 0, stm>>>(L0, z, p, p1, q, st, s.partial,
                                                                           s.tickets + 1, nblocks(NQ));
            k_update4<NR><<<dim3(lblocks(NQ, s.nz), 1, s.nz), RB, 0, stm>>>(N, s.zs, x, r, p, p1, q, st, s.partial,
                                                                            s.tickets + 2, h, use_h, nblocks(NQ));
            if (!s.use_graph) s.launches += 2;
            return;
        }
    }
    k_apply<T, NR><<<dim3(lblocks(N, s.nz), 1, s.nz), RB, 0, stm>>>(L0, z, p, p1, q, st, s.partial, s.tickets + 1,
                                                                   nblocks(N));
    k_update<T, NR><<<dim3(lblocks(N, s.nz), 1, s.nz), RB, 0, stm>>>(N, s.zs, x, r, p, p1, q, st, s.partial,
                                                                    s.tickets + 2, h, use_h, nblocks(N));
    if (!s.use_graph) s.launches += 2;
}

// capture helpers (graph mode): open a WHILE node at the current capture position
struct WhileScope {
    cudaStream_t outer, inner;
    cudaGraphConditionalHandle h;
    cudaGraphNode_t node;
    bool ok = false;
};

static cudaGraphConditionalHandle make_handle(cudaStream_t stm, cudaGraph_t* g_out) {
    cudaStreamCaptureStatus cs;
    unsigned long long id;
    cudaGraph_t g;
    const cudaGraphNode_t* deps;
    const cudaGraphEdgeData* ed;
    size_t nd;
    cudaStreamGetCaptureInfo(stm, &cs, &id, &g, &deps, &ed, &nd);
    cudaGraphConditionalHandle h;
    cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault);
    *g_out = g;
    return h;
}

static cudaStream_t begin_while(cudaStream_t stm, cudaStream_t bs, cudaGraphConditionalHandle h) {
    cudaStreamCaptureStatus cs;
    unsigned long long id;
    cudaGraph_t g;
    const cudaGraphNode_t* deps;
    const cudaGraphEdgeData* ed;
    size_t nd;
    cudaStreamGetCaptureInfo(stm, &cs, &id, &g, &deps, &ed, &nd);
    cudaGraphNodeParams cp = {};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = h;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t node;
    cudaGraphAddNode(&node, g, deps, ed, nd, &cp);
    cudaGraph_t body = cp.conditional.phGraph_out[0];
    cudaStreamUpdateCaptureDependencies(stm, &node, nullptr, 1, cudaStreamSetCaptureDependencies);
    cudaStreamBeginCaptureToGraph(bs, body, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed);
    return bs;
}

static void end_while(cudaStream_t bs) {
    cudaGraph_t g;
    cudaStreamEndCapture(bs, &g);
}

static void poll(Solver& s, cudaStream_t stm) {
    cudaMemcpyAsync(s.st_host + s.slot, s.st, sizeof(SolveState), cudaMemcpyDeviceToHost, stm);
    cudaStreamSynchronize(stm);
}

template <int NR>
static void solve_fp64(Solver& s, const double* b, double* x, double rtol, int max_iter, cudaStream_t stm) {
    int N = s.nx * s.ny;
    Lev<double> L0 = lev<double>(s, 0);
    double* z = s.d_x;   // level-0 slot of the per-level x is z
    CgPlan G;
    int cthreads = 0;
    size_t csmem = 0;
    if (cg_plan<double, NR>(s, G, cthreads, csmem)) {   // the whole solve in one launch
        k_init64<NR><<<dim3(lblocks(N, s.nz), 1, s.nz), RB, 0, stm>>>(L0, b, x, s.d_r, s.st, s.partial, s.tickets,
                                                                      rtol * rtol, max_iter, 0, 0, nblocks(N));
        launch_cg<double, NR>(s, G, cthreads, csmem, s.d_r, x, stm);
        s.launches += 2;
        return;
    }
    if (s.use_graph) {
        cudaGraph_t g;
        cudaGraphConditionalHandle h = make_handle(stm, &g);
        int mode = s.nz > 1 ? 2 : 1;
        k_init64<NR><<<dim3(lblocks(N, s.nz), 1, s.nz), RB, 0, stm>>>(L0, b, x, s.d_r, s.st, s.partial, s.tickets,
                                                                      rtol * rtol, max_iter, h, mode, nblocks(N));
        ++s.launches;
        cudaStream_t bs = begin_while(stm, s.aux[0], h);
        cg_body<double, NR>(s, x, s.d_r, z, s.d_p, s.d_q, s.st, h, mode, bs);
        end_while(bs);
        return;
    }
    k_init64<NR><<<dim3(lblocks(N, s.nz), 1, s.nz), RB, 0, stm>>>(L0, b, x, s.d_r, s.st, s.partial, s.tickets,
                                                                  rtol * rtol, max_iter, 0, 0, nblocks(N));
    ++s.launches;
    poll(s, stm);
    for (int it = 0; it < max_iter && !s.st_host[s.slot].done; ++it) {
        cg_body<double, NR>(s, x, s.d_r, z, s.d_p, s.d_q, s.st, 0, 0, stm);
        poll(s, stm);
    }
}

// The whole inner FP32 solve as one cooperative launch (use_coop == 2): single instances with
// at least one tiled level whose finest tiles and block slots fit the reduction buffer; the
// grid is min(finest tiles, co-resident blocks).  False: the solve runs as separate kernels.
template <int NR>
static bool persist_plan(Solver& s, CoarsePlan<float>& C, SmallPlan& P, int& G, size_t& smem) {
    if (s.use_coop != 2 || s.nz != 1) return false;
    int nb = nbig_of<float>(s);
    if (nb < 1) return false;
    P = small_plan<float>(s);
    smem = coarse_smem<float, NR>(P);
    struct Entry { size_t smem; int dev, res; };
    thread_local std::vector<Entry> cache[2];
    int dev = 0;
    cudaGetDevice(&dev);
    int res = -1;
    for (const Entry& e : cache[NR - 1])
        if (e.smem == smem && e.dev == dev) res = e.res;
    if (res < 0) {
        int sms = 0, per = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_cg_persist<float, NR>, CC_THREADS, smem);
        res = per * sms;
        cudaGetLastError();
        cache[NR - 1].push_back({smem, dev, res});
    }
    long long nt0 = (long long)tiles(s.nx, s.ny);
    G = (int)(nt0 < res ? nt0 : res);
    long long mb = nt0 > NRED ? nt0 : NRED;
    if (G < 1 || 2 * nt0 + 4LL * G > 4 * mb) return false;
    float* X = s.f_x;
    float* X2 = s.f_x2;
    float* B = s.f_b;
    C.l0 = 0;
    C.nb = nb;
    C.spin = s.barrier_spin > 0 ? s.barrier_spin : (1 << 22);
    for (int l = 0; l < nb; ++l) {
        C.L[l] = lev<float>(s, l);
        C.b[l] = l == 0 ? s.f_r : B + 2 * s.loff[l];
        C.x2[l] = X2 + 2 * s.loff[l];
        C.bc[l] = B + 2 * s.loff[l + 1];
        C.xo[l] = X + 2 * s.loff[l];
        C.xc[l] = X + 2 * s.loff[l + 1];
    }
    C.xo[nb] = X + 2 * s.loff[nb];
    return true;
}

template <int NR>
static void launch_persist(Solver& s, const CoarsePlan<float>& C, const SmallPlan& P, int G, size_t smem,
                           cudaStream_t stm) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(G);
    cfg.blockDim = dim3(CC_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stm;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_cg_persist<float, NR>, C, P, (const float*)s.f_diag, (const float*)s.f_wl,
                       (const float*)s.f_wb, (const float*)s.f_inv, s.f_e, s.f_r, s.f_p,
                       s.f_p + (size_t)s.nx * s.ny * NR, s.f_q, s.st, s.partial, s.tickets + 8);
    if (!s.use_graph) ++s.launches;
}

// two cells of a row per thread where rows and arrays allow 16-byte accesses, else one; rows per
// thread: eight (512 threads per SM from 2^20 cells on), two below (512^2: four take 5 % longer,
// most SMs then have one block)
template <int NR>
static void launch_ir_residual(Solver& s, const Lev<double>& L, const double* b, const double* x,
                               cudaGraphConditionalHandle ho, cudaGraphConditionalHandle hi, int mode, int set_hi,
                               unsigned* bar, cudaStream_t stm) {
    auto a16 = [](const void* p) { return ((uintptr_t)p & 15u) == 0; };
    const bool pair = s.nx % 2 == 0 && s.zs % 16 == 0 && a16(b) && a16(x) && a16(L.diag) && a16(L.wl) && a16(L.wb) &&
                      a16(s.f_r) && a16(s.f_e);
    // (16 keep the one-cell form's blocks within the reduction's slots)
    const int R = !pair ? 16 : (long long)s.nx * s.ny < (1 << 20) ? 2 : 8;
    const long long units = (long long)(pair ? s.nx / 2 : s.nx) * ((s.ny + R - 1) / R);
    const dim3 grid((unsigned)((units + IR_THREADS - 1) / IR_THREADS), 1, s.nz);
    auto k = pair ? k_ir_residual<NR, 2> : k_ir_residual<NR, 1>;
    k<<<grid, IR_THREADS, 0, stm>>>(L, b, x, s.f_r, s.f_e, s.st, s.partial, s.tickets + 5, ho, hi, mode, set_hi, bar, R);
}

template <int NR>
static void solve_mixed(Solver& s, const double* cd, const double* dd, const double* wl, const double* wb,
                        const double* b, double* x, double rtol, int max_iter, cudaStream_t stm) {
    int N = s.nx * s.ny;
    const int max_outer = 8;
    const double inner_rtol = s.inner_rtol;
    float* z = s.f_x;
    const int vb = nblocks(N), lb = lblocks(N, s.nz), lbu = lblocks((long long)N * NR, s.nz);
    // b.b and the outer tolerance do not need the hierarchy: in a captured graph they are a branch
    // beside its set-up (10-12 us behind 12-24 at 512^2)
    const bool fork = s.use_graph && s.aux[2] && s.ev[0];
    cudaStream_t si = fork ? s.aux[2] : stm;
    if (fork) {
        cudaEventRecord(s.ev[0], stm);
        cudaStreamWaitEvent(si, s.ev[0], 0);
    }
    // the FP32 hierarchy, plus D in FP64 for the refinement residual (whose face weights are the
    // caller's FP64 arrays)
    setup_levels<float>(s, cd, dd, wl, wb, s.d_diag, stm);
    Lev<double> L64{s.nx, s.ny, s.d_diag, wl, wb, s.zs, nullptr};
    k_ir_init<NR><<<dim3(lb, 1, s.nz), RB, 0, si>>>(N, s.zs, b, s.st, s.partial, s.tickets + 3, rtol * rtol,
                                                    inner_rtol, max_iter, max_outer, vb);
    ++s.launches;
    if (fork) {
        cudaEventRecord(s.ev[1], si);
        cudaStreamWaitEvent(stm, s.ev[1], 0);
    }
    CoarsePlan<float> PC;
    SmallPlan PS;
    int PG = 0;
    size_t psmem = 0;
    bool persist = persist_plan<NR>(s, PC, PS, PG, psmem);
    CgPlan G;
    int cthreads = 0;
    size_t csmem = 0;
    const bool whole = !persist && cg_plan<float, NR>(s, G, cthreads, csmem);   // each inner solve in one launch
    unsigned* pbar = persist ? s.tickets + 8 : nullptr;
    if (s.use_graph) {
        cudaGraph_t g;
        cudaGraphConditionalHandle ho = make_handle(stm, &g);
        cudaStream_t obs = begin_while(stm, s.aux[0], ho);
        int mode = s.nz > 1 ? 2 : 1;
        if (persist || whole) {
            launch_ir_residual<NR>(s, L64, b, x, ho, ho, mode, 0, pbar, obs);
            if (persist) launch_persist<NR>(s, PC, PS, PG, psmem, obs);
            else launch_cg<float, NR>(s, G, cthreads, csmem, s.f_r, s.f_e, obs);
        } else {
            cudaGraph_t og;
            cudaGraphConditionalHandle hi = make_handle(obs, &og);
            if (mode == 2) k_cond_reset<<<1, 32, 0, obs>>>(ho, hi, 1);
            launch_ir_residual<NR>(s, L64, b, x, ho, hi, mode, 1, nullptr, obs);
            cudaStream_t ibs = begin_while(obs, s.aux[1], hi);
            cg_body<float, NR>(s, s.f_e, s.f_r, z, s.f_p, s.f_q, s.st, hi, mode, ibs);
            end_while(ibs);
        }
        k_ir_update<NR><<<dim3(lbu, 1, s.nz), RB, 0, obs>>>(N, s.zs, x, s.f_e, s.st);
        end_while(obs);
        return;
    }
    for (int o = 0; o <= max_outer; ++o) {
        launch_ir_residual<NR>(s, L64, b, x, 0, 0, 0, 0, pbar, stm);
        ++s.launches;
        poll(s, stm);
        if (s.st_host[s.slot].odone) break;
        if (persist) {
            launch_persist<NR>(s, PC, PS, PG, psmem, stm);
        } else if (whole) {
            launch_cg<float, NR>(s, G, cthreads, csmem, s.f_r, s.f_e, stm);
            ++s.launches;
        } else {
            for (int it = 0; it < max_iter && !s.st_host[s.slot].done; ++it) {
                cg_body<float, NR>(s, s.f_e, s.f_r, z, s.f_p, s.f_q, s.st, 0, 0, stm);
                poll(s, stm);
            }
        }
        k_ir_update<NR><<<dim3(lbu, 1, s.nz), RB, 0, stm>>>(N, s.zs, x, s.f_e, s.st);
        ++s.launches;
    }
}

void Solver::solve(const double* cd, const double* dd, const double* wl, const double* wb, const double* b, double* x,
                   int nr, int precision, double rtol, int max_iter, cudaStream_t stm) {
    st = st_base + slot;
    // the FP64 level-0 operator is needed in both modes (outer residual of the refinement)
    if (precision == 0) {
        setup_levels<double>(*this, cd, dd, wl, wb, nullptr, stm);
        if (nr == 1) solve_fp64<1>(*this, b, x, rtol, max_iter, stm);
        else solve_fp64<2>(*this, b, x, rtol, max_iter, stm);
    } else {
        if (nr == 1) solve_mixed<1>(*this, cd, dd, wl, wb, b, x, rtol, max_iter, stm);
        else solve_mixed<2>(*this, cd, dd, wl, wb, b, x, rtol, max_iter, stm);
    }
}

bool Solver::set_schedule(int small_max, double inner) {
    if (small_max < 16 || small_max > SMALL_MAX_F_LIMIT || !(inner > 0 && inner < 1)) return false;
    small_max_f = small_max;
    inner_rtol = inner;
    int nb = 0;
    while (nb < nlev - 1 && (long long)lnx[nb] * lny[nb] > small_max_f) ++nb;
    nbig_f = nb;
    nbig = nbig_f;
    tma_ready = false;
    return true;
}

// whether the inner solves of a mixed solve are cooperative launches (EBIT_OPT_COOP 2)
template <typename T, int NR>
static bool persistent(Solver& s) {
    if constexpr (sizeof(T) == 4) {
        CoarsePlan<float> C;
        SmallPlan P;
        int g = 0;
        size_t m = 0;
        return persist_plan<NR>(s, C, P, g, m);
    }
    return false;
}

template <typename T, int NR>
static int loop_kernels(Solver& s, bool alone, bool* whole) {
    const int nb = nbig_of<T>(s);
    *whole = false;
    if (alone) {
        CgPlan G;
        ClPlan P;
        int t = 0;
        size_t m = 0;
        if (persistent<T, NR>(s) || cg_plan<T, NR>(s, G, t, m)) {
            *whole = true;
            return 0;
        }
        int l0 = cluster_plan<T, NR>(s, P, t, m);
        if (l0 == nb) l0 = coarse_start<T, NR>(s);
        return 2 * l0 + 1 + 2;
    }
    return 2 * nb + 1 + 2;
}
int Solver::body_size(int precision, int nr, bool alone, bool* whole) {
    if (precision == 0) return nr == 1 ? loop_kernels<double, 1>(*this, alone, whole) : loop_kernels<double, 2>(*this, alone, whole);
    return nr == 1 ? loop_kernels<float, 1>(*this, alone, whole) : loop_kernels<float, 2>(*this, alone, whole);
}

template <typename T, int NR>
static bool whole_if_allowed(Solver& s) {
    CgPlan G;
    int t = 0;
    size_t m = 0;
    return !persistent<T, NR>(s) && cg_plan<T, NR>(s, G, t, m);
}
bool Solver::whole_solves(int precision) {
    const int keep = use_cgc;
    use_cgc = 1;
    const bool w = precision == 0 ? whole_if_allowed<double, 1>(*this) || whole_if_allowed<double, 2>(*this)
                                  : whole_if_allowed<float, 1>(*this) || whole_if_allowed<float, 2>(*this);
    use_cgc = keep;
    return w;
}

bool Solver::supported(int nx, int ny) {
    Solver s;
    s.plan(nx, ny);
    return (long long)s.lnx[s.nlev - 1] * s.lny[s.nlev - 1] <= SMALL_MAX_D;
}

void Solver::fetch_states(cudaStream_t stm) {
    cudaMemcpyAsync(st_host, st_base, NSLOT * sizeof(SolveState), cudaMemcpyDeviceToHost, stm);
}

SolveResult Solver::read_result(int sl, int precision, cudaStream_t stm, cudaError_t* err) {
    cudaError_t e = cudaMemcpyAsync(st_host + sl, st_base + sl, sizeof(SolveState), cudaMemcpyDeviceToHost, stm);
    cudaError_t es = cudaStreamSynchronize(stm);
    if (e == cudaSuccess) e = es;
    if (err) *err = e;
    SolveResult r{};
    if (e != cudaSuccess) {   // the state was not read back: no valid result
        r.fault = true;
        return r;
    }
    return result_from_host(sl, precision);
}

SolveResult Solver::result_from_host(int sl, int precision) const {
    const SolveState& h = st_host[sl];
    SolveResult r{};
    double worst = 0.0;
    for (int k = 0; k < (h.nr > 0 ? h.nr : 1); ++k) {
        double num = precision == 0 ? h.rr[k] : h.orr[k];
        double den = precision == 0 ? h.bb[k] : h.obb[k];
        double q = sqrt(num / (den > 1e-300 ? den : 1e-300));
        if (q > worst) worst = q;
    }
    r.rel_res = worst;
    r.fault = h.fault != 0;
    r.nonfinite = h.nonfinite != 0;
    if (precision == 0) {
        r.iters = h.iters;
        r.converged = h.done != 0;
    } else {
        r.iters = h.itot;
        r.outer = h.oiters;
        bool ok = true;
        for (int k = 0; k < (h.nr > 0 ? h.nr : 1); ++k) ok = ok && h.orr[k] <= h.otol2[k];
        r.converged = ok;
    }
    return r;
}

}  // namespace ebit

// ---------------------------------------------------------------------------------------
// Allocation-free solve.  Some callers cannot allocate device memory when they call the
// solver: a host framework that owns the whole device memory through its own pool and
// forbids other allocations, or a long-running service loop that must not allocate per call
// (latency, fragmentation).  ebit_solve_system_noalloc takes the caller's device arrays for
// the operator, the right-hand side and the solution, and keeps every scratch array of the
// multigrid-preconditioned CG in the fixed array below.
//
// The array is a file-scope __device__ variable: every GPU that loads the library holds its
// 6 MiB until the process exits.  Its device address is looked up once per device, with that
// device current, by the first call on that device.  All calls share the array and it keeps
// the last call's contents; the per-call device state that must start at zero (reduction
// tickets, solver state, timers) is cleared at the start of each call.  Two calls whose work
// overlaps on the GPU (different streams, or different host threads) race on the array.
// ---------------------------------------------------------------------------------------
#include <atomic>

#include "../../include/ebit.h"
#include "status.h"

namespace ebit {
constexpr size_t NOALLOC_BYTES = (size_t)6 << 20;
constexpr int NOALLOC_MAX_CELLS = 128 * 128;
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_BYTES];
// device address of g_noalloc_scratch per device (host side); every writer stores the same
// address for a device, and the atomics make concurrent first calls well defined
static std::atomic<void*> g_noalloc_addr[64];
}  // namespace ebit

extern "C" ebit_status ebit_solve_system_noalloc(int nx, int ny, const double* D, const double* wl, const double* wb,
                                                 const double* b, double* x, int nr, int precision, double rtol,
                                                 int max_iter, void* stream, int* iters, double* rel_res) {
    using namespace ebit;
    if (nx < 2 || ny < 2 || !D || !wl || !wb || !b || !x || (nr != 1 && nr != 2) ||
        (precision != EBIT_FP64 && precision != EBIT_MIXED) || !(rtol > 0) || max_iter < 1)
        return EBIT_EINVAL;
    if ((long long)nx * ny > NOALLOC_MAX_CELLS || Solver::bytes(nx, ny) > NOALLOC_BYTES || !Solver::supported(nx, ny))
        return EBIT_EINVAL;   // larger than the fixed scratch array (at most 128 x 128 cells)
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return EBIT_ECUDA;
    void* base = g_noalloc_addr[dev].load(std::memory_order_acquire);
    if (!base) {
        if (cudaGetSymbolAddress(&base, g_noalloc_scratch) != cudaSuccess || !base) return EBIT_ECUDA;
        g_noalloc_addr[dev].store(base, std::memory_order_release);
    }
    // an error already pending from an earlier, unrelated runtime call is not this call's: it
    // is left in place, and only an error that appears during this call is taken (and cleared)
    const bool clean = cudaPeekAtLastError() == cudaSuccess;
    cudaStream_t st = (cudaStream_t)stream;
    Solver s;
    if (s.bind(base, nx, ny, false, st) != cudaSuccess) {
        if (clean) cudaGetLastError();
        return EBIT_ECUDA;
    }
    SolveState host[Solver::NSLOT];   // read_result synchronises before returning: the stack copy is safe
    s.st_host = host;
    s.slot = 0;
    s.use_graph = 0;
    s.solve(D, nullptr, wl, wb, b, x, nr, precision, rtol, max_iter, st);
    cudaError_t e = cudaSuccess;
    SolveResult r = s.read_result(0, precision, st, &e);
    if (e == cudaSuccess && clean) e = cudaGetLastError();   // launch errors of the solve
    if (e == cudaSuccess) {
        if (iters) *iters = r.iters;
        if (rel_res) *rel_res = r.rel_res;
    }
    return solve_status(e == cudaSuccess, r.fault, r.nonfinite, r.converged);
}
