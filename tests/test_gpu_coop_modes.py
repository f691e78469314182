"""EBIT_OPT_COOP 2 where it has no form of its own, and its launch counts.

2 replaces the inner FP32 solves of the mixed mode; FP64 solves run as with 1: the same launches and
the same values.  A graph step counts the kernels that the same step launched from the host counts."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_13677_gb300 import ebit as E
from paper_2402_13677_gb300 import workloads as w
from tests.test_gpu_batch import NAMES, dev, make_ctx  # noqa: F401  (dev: the fixture)


def one_step(dev, n, precision, coop, graph=1):  # noqa: F811
    pb = w.bubble(n, R0=0.2, rho_ratio=5.0, k_ratio=1.0, St=0.2, dt=1e-5, steps=0)
    ctx = make_ctx(dev, [pb], precision, rtol=1e-10)
    try:
        E.ebit_set_option(ctx, E.EBIT_OPT_GRAPH, graph)
        E.ebit_set_option(ctx, E.EBIT_OPT_COOP, coop)
        n0 = E.ebit_launch_count(ctx)
        E.ebit_step(ctx, 1)
        return E.ebit_launch_count(ctx) - n0, E.download(ctx, 0, n, n, NAMES)
    finally:
        E.ebit_destroy(ctx)


@pytest.mark.parametrize("n", [64, 160, 256])
def test_fp64_runs_as_with_one_launch_per_coarse_cycle(dev, n):  # noqa: F811
    (n0, f0), (n1, f1), (n2, f2) = (one_step(dev, n, E.EBIT_FP64, coop) for coop in (0, 1, 2))
    assert n2 == n1 < n0
    for k in NAMES:
        assert np.array_equal(f1[k], f2[k], equal_nan=True) and np.array_equal(f0[k], f2[k], equal_nan=True), k


@pytest.mark.parametrize("n", [64, 160, 256])
@pytest.mark.parametrize("precision", [E.EBIT_FP64, E.EBIT_MIXED])
def test_graph_step_counts_the_kernels_of_a_host_driven_one(dev, n, precision):  # noqa: F811
    assert one_step(dev, n, precision, 2, 1)[0] == one_step(dev, n, precision, 2, 0)[0]
