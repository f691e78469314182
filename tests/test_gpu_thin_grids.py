"""Thin grids: the single-block levels at their largest shared memory.

A 4096 x 4 grid under a single-block size of 4096 cells, which the autotuner tries, starts them at
2048 x 2 cells: with two right-hand sides (the viscous solves) their arrays and borders take 204864
bytes.  No candidate may fail, and the tuned step solves the same systems.  (The mixed pressure solve
of 4096 x 4 cells stops at 1.1e-10 after its eight refinement passes, under every schedule.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_13677_gb300 import ebit as E
from paper_2402_13677_gb300 import workloads as w
from tests.test_gpu_batch import dev, make_ctx  # noqa: F401  (dev: the fixture)


@pytest.mark.parametrize("precision", [E.EBIT_FP64, E.EBIT_MIXED])
@pytest.mark.parametrize("rtol", [1e-10, 1e-8])
@pytest.mark.parametrize("nx, ny", [(4096, 4), (4, 4096)])
def test_thin_grids_are_tuned(dev, nx, ny, rtol, precision):  # noqa: F811
    pb = w.stefan(nx, ny, dt=1e-8, steps=0)
    out = []
    for tune in (True, False):
        ctx = make_ctx(dev, [pb], precision, rtol=rtol)
        try:
            if tune:
                E.ebit_autotune(ctx, 1)
            E.ebit_step(ctx, 1, allow_noconv=True)
            out.append(E.download(ctx, 0, nx, ny, ("T_l", "T_v", "vcol")))
        finally:
            E.ebit_destroy(ctx)
    assert np.array_equal(out[0]["vcol"], out[1]["vcol"])
    scale = max(np.max(np.abs(out[1][k])) for k in ("T_l", "T_v"))   # of the one system of both phases
    for k in ("T_l", "T_v"):   # both solved to the same relative residual
        assert np.max(np.abs(out[0][k] - out[1][k])) <= 1e-6 * scale, k
