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
    util.check_parity(w, impl="simt", mode=mode, step=step, tol=util.TOL_F32)
    if dtype == "bf16" and L <= 24:
        util.check_parity(w, impl="auto", mode=mode, step=step, tol=util.TOL_F32)
