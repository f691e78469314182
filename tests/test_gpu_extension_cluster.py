"""The narrow-band extension of an instance stepped alone (one cluster of blocks) against one launch
per Jacobi sweep, on bands of a few cells and of more cells than the cluster has threads."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2402_13677_gb300 import ebit as E
from paper_2402_13677_gb300 import workloads as w


@pytest.mark.parametrize("iters", [2, 5])
@pytest.mark.parametrize("n, waves", [(16, 1), (96, 3), (384, 40)])
def test_cluster_extension_equals_launch_per_sweep(n, waves, iters):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()
    pb = w.const_mdot_levelset(
        lambda x, y: np.cos(np.pi * waves * x) * np.cos(np.pi * waves * y) + 0.1, n=n, steps=1)
    pb.energy, pb.extend_iters = True, iters
    rng = np.random.default_rng(n)
    stream, alloc, out = torch.cuda.Stream(), E.TorchAllocator(), []
    T_l, T_v = rng.normal(size=(n, n)), rng.normal(size=(n, n))
    for ext in (1, 0):
        ctx = E.ebit_init([E.config_from_problem(pb)], stream.cuda_stream, alloc)
        try:
            E.ebit_set_option(ctx, E.EBIT_OPT_EXT_BLOCK, ext)
            E.upload_state(ctx, 0, pb, pb.vcol, np.where(pb.hx_cut > 0, pb.hx_pos, 0.0),
                           np.where(pb.vy_cut > 0, pb.vy_pos, 0.0), {"T_l": T_l, "T_v": T_v}, 0.0)
            E.ebit_run_stage(ctx, E.STAGE_PREPARE)     # T_l, T_v and mdot are extended
            out.append(E.download(ctx, 0, n, n, ["T_l", "T_v", "mdot", "band"]))
        finally:
            E.ebit_destroy(ctx)
    assert out[0]["band"].sum() > (4096 if waves == 40 else 0)
    for k in ("T_l", "T_v", "mdot"):
        assert np.array_equal(out[0][k], out[1][k]), k
