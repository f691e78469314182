"""The refinement residual (rows of cells walked by a thread) against FP64 NumPy.

A mixed solve is stopped at a loose tolerance and its reported relative residual is compared with
that of the returned solution.  The device sums squares of the FP32-rounded residual (2^-24 per
value) of FP64 differences (2^-52 of terms at most about 1e3 times b, against residuals above
1e-8 b): 1e-5 covers both.  Odd and even widths, odd heights, one and several rows per thread."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_13677_gb300 import ebit as E
from paper_2402_13677_gb300 import workloads as w


@pytest.mark.parametrize("nr", [1, 2])
@pytest.mark.parametrize("nx, ny", [(31, 33), (40, 25), (33, 30), (54, 40), (336, 80), (512, 512), (1024, 1088)])
def test_reported_residual_is_the_solutions(nx, ny, nr):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()
    rng = np.random.default_rng(nx + ny + nr)
    wl = np.zeros((ny, nx)); wb = np.zeros((ny, nx))
    wl[:, 1:] = rng.uniform(0.1, 1.0, (ny, nx - 1))
    wb[1:, :] = rng.uniform(0.1, 1.0, (ny - 1, nx))
    D = np.where(rng.random((ny, nx)) < 0.5, 0.0, 0.05)
    b = rng.normal(size=(ny, nx, nr))
    stream = torch.cuda.Stream()
    ctx = E.ebit_init([E.config_from_problem(w.Problem("system", nx, ny, 1.0 / nx))], stream.cuda_stream,
                      E.TorchAllocator())
    try:
        x, _, rel = E.ebit_solve_system(ctx, 0, D, wl, wb, b, nr=nr, precision=E.EBIT_MIXED, rtol=1e-6, max_iter=400)
    finally:
        E.ebit_destroy(ctx)
    x = np.asarray(x).reshape(ny, nx, nr)
    Ax = D[..., None] * x
    f = wl[:, 1:, None] * (x[:, 1:] - x[:, :-1])
    Ax[:, 1:] += f; Ax[:, :-1] -= f
    f = wb[1:, :, None] * (x[1:] - x[:-1])
    Ax[1:] += f; Ax[:-1] -= f
    want = max(np.linalg.norm(b[..., k] - Ax[..., k]) / np.linalg.norm(b[..., k]) for k in range(nr))
    assert rel <= 1e-6
    assert abs(rel - want) <= 1e-5 * want
