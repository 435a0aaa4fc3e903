"""The one-kernel chunk form (bf16 calls that the library chooses the kernels for) at the edges of its blocks of 64 rows and
with each way of spreading a sequence's columns over CTAs (2, 40 and 160 sequences)."""
import pytest

from pf_synth import Workload
from tests import util

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,step", [("sum", "euler"), ("product", "exact")])
@pytest.mark.parametrize("d_k,d_v", [(128, 128), (64, 128), (128, 64), (64, 64)])
@pytest.mark.parametrize("r,L", [(1, 64), (1, 65), (1, 449), (2, 32), (2, 33), (2, 225), (3, 25), (3, 42), (3, 148), (4, 31), (4, 113)])
def test_block_edges(mode, step, d_k, d_v, r, L):
    w = Workload(f"chain_{L}", B=1, H=2, L=L, d_k=d_k, d_v=d_v, r=r, chunk=64, beta_scale=2.0, s0_std=0.1, seed=200 + L)
    util.check_parity(w, mode=mode, step=step)


@pytest.mark.parametrize("d_k,d_v", [(128, 128), (64, 128), (128, 64), (64, 64)])
@pytest.mark.parametrize("r", [1, 2, 3, 4])
@pytest.mark.parametrize("H", [40, 160])
def test_column_spreads(d_k, d_v, r, H):
    w = Workload(f"chain_h{H}", B=1, H=H, L=131, d_k=d_k, d_v=d_v, r=r, chunk=64, s0_std=0.1, seed=300 + r)
    util.check_parity(w)
