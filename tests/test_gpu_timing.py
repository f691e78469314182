"""Timing sessions (ebit_timing_begin .. ebit_timing_end) and what they leave behind."""
import time

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_13677_gb300 import ebit as E
from paper_2402_13677_gb300 import workloads as w
from tests.test_gpu_batch import dev, make_ctx  # noqa: F401  (dev: the fixture)


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
