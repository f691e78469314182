"""The coarse part of a V-cycle in one thread-block cluster against one launch per level.

Both forms run the same arithmetic on every cell, so a solve agrees bit for bit.  The sizes put the
slabs of the cluster's blocks at their edges: every block with rows, blocks without, a last slab of
fewer rows, two blocks of cells per thread, several FP64 levels kept by the cluster, one and two
right-hand sides, a coarsest level solved by sweeps (odd sides) and by its inverse."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_13677_gb300 import ebit as E
from paper_2402_13677_gb300 import workloads as w


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()
    torch.cuda.set_device(0)
    return E.TorchAllocator(), torch.cuda.Stream()


@pytest.mark.parametrize("nr", [1, 2])
@pytest.mark.parametrize("precision", [E.EBIT_FP64, E.EBIT_MIXED])
@pytest.mark.parametrize("nx, ny", [(512, 512), (512, 256), (256, 256), (128, 128), (208, 160), (120, 104), (80, 336),
                                    (336, 80)])
def test_cluster_coarse_cycle_equals_one_launch_per_level(dev, nx, ny, precision, nr):
    rng = np.random.default_rng(nx + 7 * ny + nr)
    wl = np.zeros((ny, nx)); wb = np.zeros((ny, nx))
    rho = np.where(rng.random((ny, nx)) < 0.5, 1.0, 20.0)
    wl[:, 1:] = 2.0 / (rho[:, 1:] + rho[:, :-1])
    wb[1:, :] = 2.0 / (rho[1:, :] + rho[:-1, :])
    D = np.zeros((ny, nx)); D[-1, :] = 0.2
    b = rng.normal(size=nx * ny * nr)
    out = []
    for coop in (1, 0):
        ctx = E.ebit_init([E.config_from_problem(w.Problem("system", nx, ny, 1.0 / nx))], dev[1].cuda_stream, dev[0])
        try:
            E.ebit_set_option(ctx, E.EBIT_OPT_COOP, coop)
            out.append(E.ebit_solve_system(ctx, 0, D, wl, wb, b, nr=nr, precision=precision, rtol=1e-10, max_iter=400))
        finally:
            E.ebit_destroy(ctx)
    assert out[0][1] == out[1][1] and out[0][2] == out[1][2]     # iterations, final residual
    assert np.array_equal(out[0][0], out[1][0])
