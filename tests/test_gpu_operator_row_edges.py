"""Operator kernels with several rows per thread, at remainders, walls and unequal phases.

A batch takes four rows of a column per thread from 2^17 cells on and eight (the energy operator four)
from 2^21; an instance alone of this size takes one.  The step must come out bit for bit the same.
Sides of 54 leave two rows of four and six of eight, sides of 92 four of eight; viscosities and
conductivities differ between the phases; the film has a no-slip wall of fixed temperature, symmetry
sides and outflow, the bubble outflow all around."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_13677_gb300 import ebit as E
from paper_2402_13677_gb300 import workloads as w
from tests.test_gpu_batch import NAMES, dev, make_ctx  # noqa: F401  (dev: the fixture)


def film(n):
    return w.film(n, n, mean=0.3, amp=0.05, modes=2, dt=0.01 / n)


def bubble(n):
    pb = w.bubble(n, R0=0.2, rho_ratio=5.0, k_ratio=5.0, St=0.2, dt=1e-4, steps=0)
    pb.mu_l, pb.mu_v = 0.02, 0.005
    return pb


@pytest.mark.parametrize("problem", [film, bubble, lambda n: w.one_fluid(bubble(n))], ids=["film", "bubble", "one_fluid"])
@pytest.mark.parametrize("n, count", [(54, 60), (92, 260), (54, 730)])
def test_step_of_a_batch_equals_the_instance_alone(dev, n, count, problem):  # noqa: F811
    pb = problem(n)
    assert pb.mu_l != pb.mu_v and pb.lam_l != pb.lam_v
    assert n * n < 2 ** 17 <= n * n * count
    out = []
    for pbs in ([pb] * count, [pb]):
        ctx = make_ctx(dev, pbs, E.EBIT_MIXED)
        try:
            E.ebit_step(ctx, 1)
            out.append([E.download(ctx, b, n, n, NAMES) for b in {0, len(pbs) - 1}])
        finally:
            E.ebit_destroy(ctx)
    for got in out[0]:
        for k in NAMES:
            assert np.array_equal(got[k], out[1][0][k], equal_nan=True), k
