"""Solver statistics of batched instances are read back to their own instance.

Two interleaved batches and an instance alone: a graph step reads each batch's slots in one strided
copy, host-driven stages (one instance solved at a time) read them one by one.  Both must report what
each instance reports when it is stepped alone."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_13677_gb300 import ebit as E
from paper_2402_13677_gb300 import workloads as w
from tests.test_gpu_batch import dev, make_ctx  # noqa: F401  (dev: the fixture)


@pytest.mark.parametrize("graph", [1, 0])
def test_statistics_reach_their_instance(dev, graph):  # noqa: F811
    def bubble(n, ratio):
        return w.bubble(n, R0=0.2, rho_ratio=ratio, k_ratio=1.0, St=0.2, dt=1e-4, steps=0)
    pbs = [bubble(32, 5.0), bubble(48, 5.0), bubble(32, 50.0), bubble(40, 5.0), bubble(48, 50.0), bubble(32, 2.0)]
    ctx = make_ctx(dev, pbs)
    try:
        E.ebit_set_option(ctx, E.EBIT_OPT_GRAPH, graph)
        E.ebit_step(ctx, 1)
        got = [E.ebit_get_diagnostics(ctx, b) for b in range(len(pbs))]
    finally:
        E.ebit_destroy(ctx)
    for b, pb in enumerate(pbs):
        ctx = make_ctx(dev, [pb])
        try:
            E.ebit_step(ctx, 1)
            assert np.array_equal(got[b], E.ebit_get_diagnostics(ctx, 0), equal_nan=True), b
        finally:
            E.ebit_destroy(ctx)
