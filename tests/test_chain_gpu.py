"""The one-kernel chunk form (bf16 calls that the library chooses the kernels for) at the edges of its blocks of 64 rows and
with fewer and more sequences than SMs (2, 40 and 160).  Which kernels ran is part of each test: the
library chooses by estimates, and a change of one must not move these calls elsewhere unnoticed."""
import numpy as np
import pytest
import torch

import pf_synth
from pf_synth import Workload
from tests import util

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,step", [("sum", "euler"), ("product", "exact")])
@pytest.mark.parametrize("d_k,d_v", [(128, 128), (64, 128), (128, 64), (64, 64)])
@pytest.mark.parametrize("r,L", [(1, 64), (1, 65), (1, 449), (2, 32), (2, 33), (2, 225), (3, 25), (3, 42), (3, 148), (4, 31), (4, 113)])
def test_block_edges(mode, step, d_k, d_v, r, L):
    w = Workload(f"chain_{L}", B=1, H=2, L=L, d_k=d_k, d_v=d_v, r=r, chunk=64, beta_scale=2.0, s0_std=0.1, seed=200 + L)
    assert util.kernels_of(lambda: util.check_parity(w, mode=mode, step=step))[0] == "chain"


@pytest.mark.parametrize("d_k,d_v", [(128, 128), (64, 128), (128, 64), (64, 64)])
@pytest.mark.parametrize("r", [1, 2, 3, 4])
@pytest.mark.parametrize("H", [40, 160])
def test_column_spreads(d_k, d_v, r, H):
    """A CTA per sequence, in one wave and in two."""
    w = Workload(f"chain_h{H}", B=1, H=H, L=131, d_k=d_k, d_v=d_v, r=r, chunk=64, s0_std=0.1, seed=300 + r)
    assert util.kernels_of(lambda: util.check_parity(w)) == ["chain"]


@pytest.mark.parametrize("d_k,d_v,r,H,L,mode", [
    (128, 128, 1, 1, 3001, "sum"), (128, 128, 2, 3, 2500, "sum"), (64, 64, 1, 2, 4097, "sum"), (64, 128, 3, 1, 2111, "product"),
    (128, 64, 4, 2, 1500, "sum"), (64, 64, 2, 10, 3000, "product"),
    (64, 64, 2, 4, 200, "sum"), (64, 128, 4, 1, 230, "sum"), (128, 128, 2, 2, 600, "sum"),
])
def test_few_long_sequences_are_walked_in_segments(d_k, d_v, r, H, L, mode):
    """The walk, the composition of the start states, their contribution to O; step sizes to 1 and to 2."""
    import paper_2504_00492_b200 as pf
    for s0_std, beta_scale in ((0.0, 1.0), (0.1, 1.0), (0.1, 2.0)):
        w = Workload(f"chain_seg_{L}", B=1, H=H, L=L, d_k=d_k, d_v=d_v, r=r, chunk=64, s0_std=s0_std, beta_scale=beta_scale, seed=400 + r)
        assert util.kernels_of(lambda: util.check_parity(w, mode=mode)) == ["chain", "chain_compose", "chain_apply"]
        assert pf.pf_last_launch_count() == 3


# (few and many sequences, with and without segments, and, with 32 x 2048 at d = 128, the single launch)
RANGE_CASES = [
    (128, 128, 1, 2, 225, "sum", "chain"), (128, 128, 2, 2, 200, "product", "chain"), (128, 64, 3, 2, 148, "sum", "chain"),
    (128, 128, 4, 2, 113, "sum", "chain"), (64, 64, 2, 40, 131, "sum", "chain"), (64, 128, 3, 160, 131, "product", "chain"),
    (128, 128, 2, 160, 131, "sum", "chain"), (64, 64, 4, 160, 70, "sum", "chain"), (128, 128, 1, 70, 300, "sum", "chain"),
    (128, 128, 2, 3, 2500, "sum", "chain"), (64, 64, 1, 2, 4097, "sum", "chain"), (128, 128, 2, 32, 2048, "sum", "fused"),
]


@pytest.mark.parametrize("token", [0, 60])
@pytest.mark.parametrize("d_k,d_v,r,H,L,mode,kernel", RANGE_CASES)
def test_a_state_that_fp16_holds_but_its_products_with_keys_exceed(d_k, d_v, r, H, L, mode, kernel, token):
    """Two columns of the start state have entries of 2e4, all aligned with the key of one token, so that the product S k there is
    2e4 sqrt(d_k) = 1.6e5 or 2.3e5, past what fp16 holds; beta is 2 there (the state is reflected, its size stays) or 1/4 (U'
    stays below, V - K S^T does not).  In those columns everything else is small beside the state, and the other columns
    must not notice."""
    import paper_2504_00492_b200 as pf
    w = Workload("range_keys", B=1, H=H, L=L, d_k=d_k, d_v=d_v, r=r, chunk=64, s0_std=0.1, seed=600 + r)
    inp = pf_synth.make_inputs(w)
    sign = torch.where(torch.randn(d_k, generator=torch.Generator().manual_seed(7)) < 0, -1.0, 1.0)
    big = [5, d_v - 1]
    # the tokens before it leave these columns alone: their keys are orthogonal to the state (neighbouring entries cancel)
    for t in range(token):
        x = inp.k[:, :, t].float() * sign
        x = (x[..., 0::2] - x[..., 1::2]).repeat_interleave(2, -1) * torch.tensor([1.0, -1.0]).repeat(d_k // 2)
        inp.k[:, :, t] = (x / x.norm(dim=-1, keepdim=True) * sign).to(inp.k.dtype)
    inp.k[:, :, token, 0] = (sign / d_k ** 0.5).to(inp.k.dtype)
    # (each factor takes about beta / d_k of the state away: step sizes with which what S_final keeps of the start state is still large)
    inp.beta *= min(1.0, 2.0 * d_k / (L * r))
    inp.beta[:, 0::2, token, 0], inp.beta[:, 1::2, token, 0] = 2.0, 0.25
    inp.S0[:, :, :, big] = (2e4 * sign)[:, None]
    d = inp.to("cuda")
    out = []
    assert kernel in util.kernels_of(lambda: out.append(pf.pf_deltanet_fwd_ex(d.q, d.k, d.v, d.beta, d.S0, w.chunk, mode=mode)))
    assert pf.pf_read_status() == 0
    rest = [j for j in range(d_v) if j not in big]
    for x, ref, what in zip(out[0], util.run_oracle(inp, mode=mode), ("O", "S_final")):
        x = x.cpu().numpy()
        assert np.isfinite(x).all(), what
        # (a step's rounding error is relative to the state at that step, so the bound is TOL_BF16 of the largest entries there have been)
        err, top = np.abs(x - ref)[..., big].max(axis=(-1, -2)), np.abs(ref[..., big]).max(axis=(-1, -2))
        assert (err <= util.TOL_BF16 * np.maximum(top, 2e4)).all(), (what, (err / np.maximum(top, 2e4)).max())
        util.check_per_sequence(x[..., rest], ref[..., rest], util.TOL_BF16, what + ", other columns")


def test_a_call_whose_end_state_replaces_its_start_state():
    """S_final written over S0, also where rows of the state have to be walked a second time."""
    import paper_2504_00492_b200 as pf
    w = Workload("in_place", B=1, H=2, L=96, d_k=128, d_v=128, r=2, chunk=64, s0_std=0.1, seed=611)
    inp = pf_synth.make_inputs(w)
    inp.S0[:, 1, :, 3] = 2e4
    inp.k[:, :, 0, 0] = 128 ** -0.5
    d = inp.to("cuda")
    O, S = pf.pf_deltanet_fwd(d.q, d.k, d.v, d.beta, d.S0, w.chunk)
    O2, S2 = pf.pf_deltanet_fwd(d.q, d.k, d.v, d.beta, d.S0, w.chunk, S_final=d.S0)
    assert torch.isfinite(O).all() and torch.isfinite(S).all()
    assert torch.equal(O, O2) and torch.equal(S, S2) and S2.data_ptr() == d.S0.data_ptr()


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


@pytest.mark.parametrize("d_k,d_v", [(128, 128), (64, 64), (128, 64)])
@pytest.mark.parametrize("r", [1, 2, 3, 4])
@pytest.mark.parametrize("blocks", [2, 3, 4, 5, 6, 7, 13])
def test_the_ring_of_stages_wraps(d_k, d_v, r, blocks):
    """As many blocks as there are stages of shared memory (3 to 6), one more, one fewer, and several times round."""
    L = blocks * (64 // r) - (blocks % 2)
    w = Workload(f"ring_{blocks}", B=1, H=70, L=L, d_k=d_k, d_v=d_v, r=r, chunk=64, beta_scale=2.0, s0_std=0.1, seed=700 + r)
    assert util.kernels_of(lambda: util.check_parity(w))[0] == "chain"


@pytest.mark.parametrize("d_k,d_v,r,H,L,impl", [(128, 128, 1, 148, 320, "auto"), (128, 128, 2, 148, 200, "auto"), (64, 64, 3, 148, 150, "auto"),
                                                (64, 128, 4, 148, 100, "auto"), (128, 128, 1, 3, 2500, "auto"), (128, 128, 2, 32, 1024, "tc"),
                                                (128, 128, 2, 160, 300, "auto"), (64, 64, 4, 32, 3001, "auto")])
def test_repeated_calls_agree_to_the_bit(d_k, d_v, r, H, L, impl):
    """Which products of an accumulator run one after another must not be a matter of timing: the same call, many times in a row."""
    import paper_2504_00492_b200 as pf
    w = Workload("again", B=1, H=H, L=L, d_k=d_k, d_v=d_v, r=r, chunk=64, beta_scale=2.0, s0_std=0.1, seed=800 + r)
    d = pf_synth.make_inputs(w).to("cuda")
    first = pf.pf_deltanet_fwd_ex(d.q, d.k, d.v, d.beta, d.S0, w.chunk, impl=impl)
    for _ in range(200):
        O, S = pf.pf_deltanet_fwd_ex(d.q, d.k, d.v, d.beta, d.S0, w.chunk, impl=impl)
        assert torch.equal(O, first[0]) and torch.equal(S, first[1])


@pytest.mark.parametrize("where", ["response", "readout"])
@pytest.mark.parametrize("in_place", [False, True])
def test_responses_that_leave_the_range_of_fp16(where, in_place):
    """32 sequences of 8192, which are walked in segments for speed.  In every third sequence 18 tokens of the second segment double and negate what the state
    holds along one key: the response to the segment's start state reaches 2^18 while the state itself, 1e-3 there, stays small.  Or one query of
    the segment is as long as 3e5, so that only a token's response leaves the range.  Neither may cost more than time."""
    import paper_2504_00492_b200 as pf
    w = Workload("amplified", B=1, H=32, L=8192, d_k=128, d_v=128, r=2, chunk=64, beta_scale=0.5, s0_std=0.1, seed=990)
    inp = pf_synth.make_inputs(w)
    seqs = slice(0, w.H, 3)
    k = inp.k.float()
    k[..., 0] = 0.0                                               # (nothing else touches the first entry)
    inp.k = (k / k.norm(dim=-1, keepdim=True)).to(inp.k.dtype)
    inp.S0[:, :, 0] *= 1e-2
    if where == "response":
        for t in range(5700, 5700 + 18 * 64, 64):
            inp.k[:, seqs, t] = torch.eye(128)[0].to(inp.k.dtype)
            inp.v[:, seqs, t] = 0.0
            inp.beta[:, seqs, t] = 1.5
    else:
        inp.q[:, seqs, 6000] = (3e5 * torch.eye(128)[0]).to(inp.q.dtype)
        inp.S0[:, seqs, 0] *= 1e-2
    d = inp.to("cuda")
    out = []
    names = util.kernels_of(lambda: out.append(pf.pf_deltanet_fwd(d.q, d.k, d.v, d.beta, d.S0, w.chunk, S_final=d.S0 if in_place else None)))
    assert names == ["chain", "chain_compose", "chain_apply"] and pf.pf_read_status() == 0
    O_ref, S_ref = util.run_oracle(inp)
    for x, ref, what in zip(out[0], (O_ref, S_ref), ("O", "S_final")):
        assert torch.isfinite(x).all(), what
        util.check_per_sequence(x.cpu().numpy(), ref, util.TOL_BF16, what)


@pytest.mark.parametrize("d,r,most", [(128, 2, 35), (64, 2, 25)])
def test_the_second_walk_of_lost_rows_takes_a_bounded_multiple_of_the_call(d, r, most):
    """Every row lost (a start state beyond fp16): 20 and 14 times the call without, 63 and 34 where eight warps walk 16 rows each."""
    import paper_2504_00492_b200 as pf
    w = Workload("lost", B=1, H=70, L=400, d_k=d, d_v=d, r=r, chunk=64, s0_std=0.1, seed=901)
    c = pf_synth.make_inputs(w).to("cuda")
    times = []
    for S0 in (c.S0, torch.full_like(c.S0, 1e5)):
        for _ in range(3):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            for _ in range(4):
                O, S = pf.pf_deltanet_fwd(c.q, c.k, c.v, c.beta, S0, w.chunk)
            e1.record()
            e1.synchronize()
            times.append(e0.elapsed_time(e1))
        assert torch.isfinite(O).all() and torch.isfinite(S).all()
    assert min(times[3:]) <= most * min(times[:3]), times


@pytest.mark.parametrize("r,L,mode,beta_scale,most", [(4, 600, "sum", 2.0, 3.1e-4), (2, 1200, "product", 2.0, 3.1e-4), (1, 2400, "sum", 1.0, 2.35e-4), (3, 801, "sum", 1.0, 2.35e-4)])
def test_values_that_the_state_predicts(r, L, mode, beta_scale, most):
    """v = S* k, what the delta rule is for: once S is near S*, v - S k is small, and no more than the rounding of k and of S may be left in it.
    Relative L2 error of O: 2.7e-4 for step sizes to 2 and 2.2e-4 for step sizes to 1; 3.7e-4 and 2.5e-4 where the inverse is applied to
    v and to k apart.  The bounds lie between the two."""
    w = Workload("predicted", B=1, H=100, L=L, d_k=64, d_v=64, r=r, chunk=64, beta_scale=beta_scale, seed=920 + r)
    inp = pf_synth.make_inputs(w)
    S = torch.randn(1, w.H, 64, 64, generator=torch.Generator().manual_seed(11)) / 8
    inp.v = torch.einsum("bhji,bhtri->bhtrj", S, inp.k.float()).to(inp.v.dtype)
    O, S_end = util.run_gpu(w, inp, mode=mode)
    O_ref, S_ref = util.run_oracle(inp, mode=mode)
    assert util.rel_l2(O, O_ref) <= most and util.rel_l2(S_end, S_ref) <= most, (util.rel_l2(O, O_ref), util.rel_l2(S_end, S_ref))


def _workspaces(w):
    """Bytes of workspace with which the call's walks may be shared out among all SMs, and what a call of one walk to a CTA has."""
    import paper_2504_00492_b200 as pf
    step_sizes = (w.B * w.H * w.L * w.r * 4 + 255) // 256 * 256
    return pf.pf_workspace_bytes(w.B, w.H, w.L, w.d_k, w.d_v, w.r, w.chunk), 1024 + step_sizes


@pytest.mark.parametrize("lost", [False, True])
@pytest.mark.parametrize("d_k,d_v,r,H,L,mode,step", [(128, 128, 2, 160, 300, "sum", "euler"), (128, 64, 3, 150, 200, "product", "exact"), (64, 128, 1, 200, 1000, "sum", "euler"),
                                                     (128, 128, 1, 190, 1000, "sum", "exact"), (128, 128, 4, 180, 701, "product", "euler"), (64, 64, 1, 200, 2000, "sum", "euler")])
def test_walks_shared_out_match_whole_ones_to_the_bit(d_k, d_v, r, H, L, mode, step, lost):
    """More sequences than SMs: a walk that is cut goes on in another CTA from the very state it had.  Without workspace for that every walk is whole.
    lost: columns that leave fp16's range in some sequences are walked again, all of the walk by the CTA that has its end."""
    import paper_2504_00492_b200 as pf
    w = Workload("shared", B=1, H=H, L=L, d_k=d_k, d_v=d_v, r=r, chunk=64, s0_std=0.1, seed=950 + r)
    inp = pf_synth.make_inputs(w)
    if lost:
        inp.S0[:, ::3, :, 5] = 1e5
    need, small = _workspaces(w)
    assert need >= small + torch.cuda.get_device_properties(0).multi_processor_count // 2 * 4 * d_k * d_v, "not shared out"
    d = inp.to("cuda")
    whole = pf.pf_deltanet_fwd_ex(d.q, d.k, d.v, d.beta, d.S0, w.chunk, mode=mode, step=step, workspace=torch.empty(small, dtype=torch.uint8, device="cuda"))
    for workspace in (None, torch.full((need,), 255, dtype=torch.uint8, device="cuda")):
        O, S = pf.pf_deltanet_fwd_ex(d.q, d.k, d.v, d.beta, d.S0, w.chunk, mode=mode, step=step, workspace=workspace)
        assert pf.pf_read_status(workspace) == 0 and torch.isfinite(O).all() and torch.isfinite(S).all()
        assert torch.equal(O, whole[0]) and torch.equal(S, whole[1])
    if not lost:
        O_ref, S_ref = util.run_oracle(inp, mode=mode, step=step)
        util.check_per_sequence(O.cpu().numpy(), O_ref, util.TOL_BF16, "O")
        util.check_per_sequence(S.cpu().numpy(), S_ref, util.TOL_BF16, "S_final")


@pytest.mark.parametrize("d,r,H,L,beta_scale,mode,step", [(64, 2, 32, 5000, 1.0, "sum", "euler"), (128, 4, 32, 2100, 1.0, "sum", "euler"), (64, 4, 32, 3001, 2.0, "product", "exact"),
                                                          (128, 4, 32, 2100, 0.02, "sum", "euler")])
def test_segments_shared_out(d, r, H, L, beta_scale, mode, step):
    """Few sequences in segments of two lengths, cut and shared out among all SMs."""
    w = Workload("shared_seg", B=1, H=H, L=L, d_k=d, d_v=d, r=r, chunk=64, s0_std=0.1, beta_scale=beta_scale, seed=970 + r)
    need, _ = _workspaces(w)
    assert util.kernels_of(lambda: util.check_parity(w, mode=mode, step=step)) == ["chain", "chain_compose", "chain_apply"]
    # (a byte less is not enough for that, and the call takes the segments it has without: it would be refused if it did not share)
    less = torch.empty(need - 1, dtype=torch.uint8, device="cuda")
    assert util.kernels_of(lambda: util.check_parity(w, mode=mode, step=step, workspace=less)) == ["chain", "chain_compose", "chain_apply"]


@pytest.mark.parametrize("d,r,L", [(128, 4, 2100), (64, 4, 3001)])
def test_segments_shared_out_whose_end_state_replaces_the_start_state(d, r, L):
    """One CTA reads S0 and another writes S_final; in every third sequence a column's products with keys leave fp16's range, so that the first segment's walk is walked again."""
    import paper_2504_00492_b200 as pf
    w = Workload("shared_in_place", B=1, H=32, L=L, d_k=d, d_v=d, r=r, chunk=64, s0_std=0.1, seed=980 + r)
    inp = pf_synth.make_inputs(w)
    inp.S0[:, ::3, :, 3] = 2e4
    inp.k[:, :, 0, 0] = d ** -0.5
    c = inp.to("cuda")
    O, S = pf.pf_deltanet_fwd(c.q, c.k, c.v, c.beta, c.S0, w.chunk)
    O2, S2 = pf.pf_deltanet_fwd(c.q, c.k, c.v, c.beta, c.S0, w.chunk, S_final=c.S0)
    assert pf.pf_last_launch_count() == 3 and pf.pf_read_status() == 0
    assert torch.equal(O, O2) and torch.equal(S, S2) and S2.data_ptr() == c.S0.data_ptr()
    for x, ref, what in zip((O, S), util.run_oracle(inp), ("O", "S_final")):
        assert torch.isfinite(x).all(), what
        util.check_per_sequence(x.cpu().numpy(), ref, util.TOL_BF16, what)


@pytest.mark.parametrize("d,r,H,L", [(128, 2, 160, 300), (128, 4, 32, 2100)])
def test_shared_out_calls_on_two_streams(d, r, H, L):
    """States that go from one CTA to another through memory, of two calls at a time, each many times."""
    import paper_2504_00492_b200 as pf
    w = Workload("streams", B=1, H=H, L=L, d_k=d, d_v=d, r=r, chunk=64, beta_scale=1.0, s0_std=0.1, seed=985 + r)
    inputs = [pf_synth.make_inputs(w, seed).to("cuda") for seed in (1, 2)]
    want = [pf.pf_deltanet_fwd(c.q, c.k, c.v, c.beta, c.S0, w.chunk) for c in inputs]
    streams = [torch.cuda.Stream() for _ in inputs]
    torch.cuda.synchronize()
    got = [[], []]
    for _ in range(20):
        for x, (c, stream) in enumerate(zip(inputs, streams)):
            with torch.cuda.stream(stream):
                got[x].append(pf.pf_deltanet_fwd(c.q, c.k, c.v, c.beta, c.S0, w.chunk))
    torch.cuda.synchronize()
    for x, first in enumerate(want):
        for O, S in got[x]:
            assert torch.equal(O, first[0]) and torch.equal(S, first[1])


def test_shared_out_segments_need_no_more_workspace_than_the_library_keeps():
    """What the pool does not keep is mapped anew at every call of a caller who synchronises in between: 2.7 ms instead of 0.3 at 9600 tokens."""
    shared = 0
    for L in range(4096, 20000, 400):
        need, small = _workspaces(Workload("keep", B=1, H=32, L=L, d_k=128, d_v=128, r=2, chunk=64))
        assert need - (small - 1024) <= 96 << 20, (L, need)
        shared = max(shared, need)
    assert shared > 90 << 20, "not shared out"


def test_segments_of_an_option_take_less_workspace_than_sharing_walks_out_would():
    """160 walks of the option `segments` are shared out for speed where there is workspace for that, and are a CTA's each where not."""
    import paper_2504_00492_b200 as pf
    w = Workload("option", B=1, H=20, L=8000, d_k=128, d_v=128, r=2, chunk=64, s0_std=0.1, seed=995)
    need = pf.pf_workspace_bytes_ex(w.B, w.H, w.L, w.d_k, w.d_v, w.r, w.chunk, segments=8)
    states = torch.cuda.get_device_properties(0).multi_processor_count // 2 * 4 * w.d_k * w.d_v
    for workspace in (None, need, need - states):
        util.check_parity(w, segments=8, workspace=workspace and torch.empty(workspace, dtype=torch.uint8, device="cuda"))
