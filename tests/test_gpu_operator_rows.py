"""Operator kernels with one row per thread against several rows that share coefficients.

A batch of equal grids takes more rows per thread than one of its instances alone (one below 2^17
cells, four from there, eight from 2^21 on); every row must come out bit for bit the same.  Sides that
are no multiple of the rows or of a warp, an interface inside the rows, walls and outflow."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_13677_gb300 import ebit as E
from paper_2402_13677_gb300 import workloads as w
from tests.test_gpu_batch import NAMES, dev, make_ctx  # noqa: F401  (dev: the fixture)


@pytest.mark.parametrize("nx, count, one_fluid", [(92, 20, False), (92, 20, True), (52, 60, False), (128, 130, False)])
def test_rows_per_thread_do_not_change_a_step(dev, nx, count, one_fluid):  # noqa: F811
    pb = w.bubble(nx, R0=0.2, rho_ratio=5.0, k_ratio=1.0, St=0.2, dt=1e-4, steps=0)
    if one_fluid:
        pb = w.one_fluid(pb)
    out = []
    for pbs in ([pb] * count, [pb]):
        ctx = make_ctx(dev, pbs, E.EBIT_MIXED)
        try:
            E.ebit_step(ctx, 2)
            out.append(E.download(ctx, len(pbs) - 1, nx, pb.ny, NAMES))
        finally:
            E.ebit_destroy(ctx)
    for k in NAMES:
        assert np.array_equal(out[0][k], out[1][k], equal_nan=True), k
