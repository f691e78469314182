"""ebit_launch_count of a graph step against the same step launched from the host."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_13677_gb300 import ebit as E
from paper_2402_13677_gb300 import workloads as w
from tests.test_gpu_batch import dev, make_ctx  # noqa: F401  (dev: the fixture)


def launches(dev, pb, precision, coop, graph):  # noqa: F811
    ctx = make_ctx(dev, [pb], precision, rtol=1e-10)
    try:
        E.ebit_set_option(ctx, E.EBIT_OPT_GRAPH, graph)
        E.ebit_set_option(ctx, E.EBIT_OPT_COOP, coop)
        n0 = E.ebit_launch_count(ctx)
        E.ebit_step(ctx, 1)
        return E.ebit_launch_count(ctx) - n0
    finally:
        E.ebit_destroy(ctx)


@pytest.mark.parametrize("one_fluid", [False, True])
@pytest.mark.parametrize("precision", [E.EBIT_FP64, E.EBIT_MIXED])
@pytest.mark.parametrize("coop", [0, 1])
@pytest.mark.parametrize("n", [64, 160, 256])
def test_graph_step_counts_the_kernels_of_a_host_driven_one(dev, n, coop, precision, one_fluid):  # noqa: F811
    pb = w.bubble(n, R0=0.2, rho_ratio=5.0, k_ratio=1.0, St=0.2, dt=1e-5, steps=0)
    if one_fluid:
        pb = w.one_fluid(pb)
    assert launches(dev, pb, precision, coop, 1) == launches(dev, pb, precision, coop, 0)
