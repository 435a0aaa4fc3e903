"""The one-kernel chunk form (bf16 calls that the library chooses the kernels for) at the edges of its blocks of 64 rows and
with each way of spreading a sequence's columns over CTAs (2, 40 and 160 sequences)."""
import pytest

import pf_synth
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


@pytest.mark.parametrize("d_k,d_v,r,H,L,mode", [
    (128, 128, 1, 1, 3001, "sum"), (128, 128, 2, 3, 2500, "sum"), (64, 64, 1, 2, 4097, "sum"), (64, 128, 3, 1, 2111, "product"),
    (128, 64, 4, 2, 1500, "sum"), (64, 64, 2, 10, 3000, "product"),
    (64, 64, 2, 4, 200, "sum"), (64, 128, 4, 1, 230, "sum"), (128, 128, 2, 2, 600, "sum"),
])
def test_few_long_sequences_are_walked_in_segments(d_k, d_v, r, H, L, mode):
    """Told apart by the number of kernels: the walk, the composition of the start states, their contribution to O."""
    import paper_2504_00492_b200 as pf
    for s0_std in (0.0, 0.1):
        w = Workload(f"chain_seg_{L}", B=1, H=H, L=L, d_k=d_k, d_v=d_v, r=r, chunk=64, s0_std=s0_std, seed=400 + r)
        util.check_parity(w, mode=mode)
        assert pf.pf_last_launch_count() == 3


@pytest.mark.parametrize("d_k,d_v,r,H,L,mode", [(128, 128, 1, 4, 8000, "sum"), (64, 64, 1, 2, 4097, "sum"), (128, 128, 2, 3, 2500, "product"),
                                                (64, 128, 3, 1, 2111, "sum")])
def test_segments_of_a_state_that_changes_slowly(d_k, d_v, r, H, L, mode):
    """Step sizes of about 0.01: a segment changes little of its start state, and only the change may be rounded to fp16 (2^-11 of
    it; the whole sequence changes less than half of the state here), not the state once per segment."""
    import paper_2504_00492_b200 as pf
    w = Workload(f"slow_{L}", B=1, H=H, L=L, d_k=d_k, d_v=d_v, r=r, chunk=64, s0_std=0.1, beta_scale=0.02, seed=500 + r)
    inp = pf_synth.make_inputs(w)
    O, S = util.run_gpu(w, inp, mode=mode)
    assert pf.pf_last_launch_count() == 3
    O_ref, S_ref = util.run_oracle(inp, mode=mode)
    util.check_per_sequence(O, O_ref, util.TOL_BF16, "O")
    assert util.rel_l2(S, S_ref) <= 2 ** -12, util.rel_l2(S, S_ref)
