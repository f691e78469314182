"""Timing sessions (ebit_timing_begin .. ebit_timing_end) and what they leave behind."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_13677_gb300 import ebit as E
from paper_2402_13677_gb300 import workloads as w
from tests.test_gpu_batch import NAMES, dev, make_ctx  # noqa: F401  (dev: the fixture)


def bubble(n):
    return w.bubble(n, R0=0.2, rho_ratio=5.0, k_ratio=1.0, St=0.2, dt=1e-5, steps=0)


@pytest.mark.parametrize("graph", [1, 0])
@pytest.mark.parametrize("sides", [(64,), (160,), (48, 48, 64)])
def test_launches_after_the_session_are_not_timed(dev, sides, graph):  # noqa: F811
    """The second end reports the first one's figures although a step ran in between; a new session
    starts from zero."""
    ctx = make_ctx(dev, [bubble(n) for n in sides], E.EBIT_MIXED)
    try:
        E.ebit_set_option(ctx, E.EBIT_OPT_GRAPH, graph)
        E.ebit_timing_begin(ctx)
        E.ebit_step(ctx, 1)
        first = E.ebit_timing_end(ctx)
        E.ebit_step(ctx, 1)
        assert E.ebit_timing_end(ctx) == first
        assert first[0] > 0 and first[1] > 0
        E.ebit_timing_begin(ctx)
        assert E.ebit_timing_end(ctx)[:2] == (0.0, 0)
    finally:
        E.ebit_destroy(ctx)


def test_a_session_keeps_the_step_graphs_it_can_use(dev):  # noqa: F811
    """Above 16384 cells a timed step launches what an untimed one does: its graph is not captured
    again.  The first step of a session is compared with a later one of it and with a step that does
    capture (an option was set, which drops the graphs): it is the nearer to the former."""
    ctx = make_ctx(dev, [bubble(160)], E.EBIT_MIXED)

    def step():
        torch.cuda.synchronize()
        t = time.perf_counter()
        E.ebit_step(ctx, 1)
        return time.perf_counter() - t
    try:
        capture, first, later = [], [], []
        for _ in range(9):
            E.ebit_set_option(ctx, E.EBIT_OPT_TMA, 1)
            step(), step()              # both sweep orders
            E.ebit_timing_begin(ctx)
            E.ebit_set_option(ctx, E.EBIT_OPT_TMA, 1)
            capture.append(step())
            step()
            later.append(step())
            E.ebit_timing_end(ctx)
            E.ebit_timing_begin(ctx)
            first.append(step())
            E.ebit_timing_end(ctx)
        assert 2 * min(first) < min(later) + min(capture), (min(first), min(later), min(capture))
    finally:
        E.ebit_destroy(ctx)


@pytest.mark.parametrize("nr", [1, 2])
@pytest.mark.parametrize("precision", [E.EBIT_FP64, E.EBIT_MIXED])
@pytest.mark.parametrize("nx, ny", [(128, 128), (120, 104), (96, 80), (512, 32), (32, 512), (72, 88)])
def test_solves_of_a_session_equal_whole_and_separate_ones(dev, nx, ny, precision, nr):  # noqa: F811
    """Grids whose solve is one launch run it as separate ones in a session, their coarse levels in a
    cluster: bit for bit the whole solve outside it and the solve of one launch per level."""
    rng = np.random.default_rng(nx + 7 * ny + nr)
    wl = np.zeros((ny, nx)); wb = np.zeros((ny, nx))
    rho = np.where(rng.random((ny, nx)) < 0.5, 1.0, 20.0)
    wl[:, 1:] = 2.0 / (rho[:, 1:] + rho[:, :-1])
    wb[1:, :] = 2.0 / (rho[1:, :] + rho[:-1, :])
    D = np.zeros((ny, nx)); D[-1, :] = 0.2
    b = rng.normal(size=nx * ny * nr)
    ctx = E.ebit_init([E.config_from_problem(w.Problem("system", nx, ny, 1.0 / nx))], dev[1].cuda_stream, dev[0])

    def solve():
        return E.ebit_solve_system(ctx, 0, D, wl, wb, b, nr=nr, precision=precision, rtol=1e-10, max_iter=400)
    try:
        whole = solve()
        E.ebit_timing_begin(ctx)
        timed = solve()
        _, launches, _ = E.ebit_timing_end(ctx)
        E.ebit_set_option(ctx, E.EBIT_OPT_COOP, 0)
        separate = solve()
    finally:
        E.ebit_destroy(ctx)
    assert launches > 0
    for other in (timed, separate):
        assert other[1:] == whole[1:]
        assert np.array_equal(other[0], whole[0])


@pytest.mark.parametrize("precision", [E.EBIT_FP64, E.EBIT_MIXED])
def test_steps_of_a_session_equal_untimed_ones(dev, precision):  # noqa: F811
    out = []
    for timed in (True, False):
        ctx = make_ctx(dev, [bubble(64)], precision)
        try:
            if timed:
                E.ebit_timing_begin(ctx)
            E.ebit_step(ctx, 2)
            if timed:
                E.ebit_timing_end(ctx)
            E.ebit_step(ctx, 2)
            out.append(E.download(ctx, 0, 64, 64, NAMES))
        finally:
            E.ebit_destroy(ctx)
    for k in NAMES:
        assert np.array_equal(out[0][k], out[1][k], equal_nan=True), k
