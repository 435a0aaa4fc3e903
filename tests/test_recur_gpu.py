"""The token-by-token kernel (fp32 calls, bf16 calls of a few tokens) at the edges of its passes and stages."""
import pytest

from pf_synth import Workload
from tests import util

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("mode,step", [("sum", "euler"), ("product", "exact")])
@pytest.mark.parametrize("r,d_k,d_v", [(1, 64, 128), (2, 128, 64), (3, 128, 128), (4, 64, 64)])
@pytest.mark.parametrize("L", [1, 3, 4, 15, 17, 24, 50])
def test_pass_and_stage_edges(dtype, mode, step, r, d_k, d_v, L):
    w = Workload(f"recur_{L}", B=2, H=1, L=L, d_k=d_k, d_v=d_v, r=r, chunk=64, dtype=dtype, beta_scale=2.0,
                 s0_std=0.1, seed=80 + L)
    assert util.kernels_of(lambda: util.check_parity(w, impl="simt", mode=mode, step=step, tol=util.TOL_F32)) == ["recur"]
    if dtype == "bf16" and L <= 24:
        (kernel,) = util.kernels_of(lambda: util.check_parity(w, impl="auto", mode=mode, step=step))
        assert kernel == "recur" or (kernel == "chain" and L > 4)      # (the line between the two lies at 8 to 30 tokens)


@pytest.mark.parametrize("d_k,d_v,r,H,L,mode", [
    (64, 64, 2, 2, 1000, "sum"), (64, 128, 1, 1, 2049, "sum"), (128, 64, 3, 1, 1111, "product"), (128, 128, 1, 2, 1777, "sum"),
    (64, 64, 4, 5, 640, "product"), (64, 64, 2, 1, 200, "sum"), (128, 128, 1, 1, 300, "sum"), (128, 128, 1, 8, 1000, "sum"),
])
def test_few_long_sequences_are_walked_in_segments(d_k, d_v, r, H, L, mode):
    """The walk, the composition of the start states, their contribution to O; step sizes to 1 and to 2."""
    import paper_2504_00492_b200 as pf
    for s0_std, beta_scale in ((0.0, 1.0), (0.1, 1.0), (0.1, 2.0)):
        w = Workload(f"recur_seg_{L}", B=1, H=H, L=L, d_k=d_k, d_v=d_v, r=r, chunk=64, dtype="f32", s0_std=s0_std, beta_scale=beta_scale,
                     seed=500 + r)
        assert util.kernels_of(lambda: util.check_parity(w, mode=mode)) == ["recur", "recur_compose", "recur_apply"]
        assert pf.pf_last_launch_count() == 3
