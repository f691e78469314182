"""A whole CG solve in one thread-block cluster against its separate launches.

The cluster form repeats the arithmetic and the order of every sum of the separate kernels, so
solutions, iteration counts and residuals agree bit for bit; status codes agree too.  The sizes put
it at its edges: the largest grid (16384 cells) and the first beyond it, sides that are no multiple
of a tile (32) or of a vector (4), slabs of fewer rows, blocks of the cluster without rows, long and
flat grids, one and two right-hand sides."""
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


def _both(dev, nx, ny, precision, nr, seed, poison=False, **kw):
    rng = np.random.default_rng(seed)
    wl = np.zeros((ny, nx)); wb = np.zeros((ny, nx))
    rho = np.where(rng.random((ny, nx)) < 0.5, 1.0, 20.0)
    wl[:, 1:] = 2.0 / (rho[:, 1:] + rho[:, :-1])
    wb[1:, :] = 2.0 / (rho[1:, :] + rho[:-1, :])
    D = np.zeros((ny, nx)); D[-1, :] = 0.2
    b = rng.normal(size=nx * ny * nr)
    x0 = rng.normal(size=nx * ny * nr)
    if poison:
        b[(nx * ny * nr) // 2] = np.nan
    out = []
    for coop in (1, 0):
        ctx = E.ebit_init([E.config_from_problem(w.Problem("system", nx, ny, 1.0 / nx))], dev[1].cuda_stream, dev[0])
        try:
            E.ebit_set_option(ctx, E.EBIT_OPT_COOP, coop)
            try:
                r = E.ebit_solve_system(ctx, 0, D, wl, wb, b, x0=x0, nr=nr, precision=precision, **kw)
                out.append((None, *r))
            except E.EbitError as e:
                out.append((e.status, None, None, None))
        finally:
            E.ebit_destroy(ctx)
    return out


@pytest.mark.parametrize("nr", [1, 2])
@pytest.mark.parametrize("precision", [E.EBIT_FP64, E.EBIT_MIXED])
@pytest.mark.parametrize("nx, ny", [(64, 64), (96, 80), (120, 104), (128, 128), (144, 128), (36, 44), (54, 40), (40, 54),
                                    (512, 32), (32, 512), (58, 68)])
def test_whole_solve_equals_separate_launches(dev, nx, ny, precision, nr):
    a, b = _both(dev, nx, ny, precision, nr, nx + 7 * ny + nr, rtol=1e-10, max_iter=400)
    assert a[0] == b[0] and a[2:] == b[2:]
    assert np.array_equal(a[1], b[1])


@pytest.mark.parametrize("precision", [E.EBIT_FP64, E.EBIT_MIXED])
@pytest.mark.parametrize("poison, max_iter", [(False, 2), (False, 1), (True, 50)])
def test_whole_solve_reports_as_separate_launches(dev, precision, poison, max_iter):
    a, b = _both(dev, 96, 80, precision, 1, 5, poison=poison, rtol=1e-12, max_iter=max_iter, allow_noconv=True)
    assert a[0] == b[0] == (E.EBIT_ENONFINITE if poison else None)
    if not poison:
        assert a[2:] == b[2:]
        assert np.array_equal(a[1], b[1])
