"""The library's own workspaces: calls on two streams and from two threads share the pool, and it is given back on request."""
import threading

import pytest
import torch

import pf_synth
from pf_synth import Workload

pytestmark = pytest.mark.gpu

# calls in segments, which take their intermediate results from the pool
CASES = [
    Workload("pool_bf16", B=1, H=2, L=4097, d_k=64, d_v=64, r=1, chunk=64, s0_std=0.1, seed=71),
    Workload("pool_bf16_r2", B=1, H=3, L=2500, d_k=128, d_v=128, r=2, chunk=64, s0_std=0.1, seed=72),
    Workload("pool_f32", B=1, H=2, L=1000, d_k=64, d_v=64, r=2, chunk=64, dtype="f32", s0_std=0.1, seed=73),
]


def _call(w, d):
    import paper_2504_00492_b200 as pf
    return (pf.pf_deltanet_fwd_f32 if w.dtype == "f32" else pf.pf_deltanet_fwd)(d.q, d.k, d.v, d.beta, d.S0, w.chunk)


def test_calls_on_two_streams_share_the_pool():
    import paper_2504_00492_b200 as pf
    inputs = [pf_synth.make_inputs(w).to("cuda") for w in CASES]
    want = [_call(w, d) for w, d in zip(CASES, inputs)]
    assert pf.pf_last_launch_count() == 3
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    got = []
    for i in range(40):
        with torch.cuda.stream(streams[i % 2]):
            n = (i // 2 + i) % len(CASES)
            got.append((n, _call(CASES[n], inputs[n])))
    torch.cuda.synchronize()
    for n, (O, S) in got:
        assert torch.equal(O, want[n][0]) and torch.equal(S, want[n][1]), CASES[n].name


def test_calls_from_two_threads_share_the_pool():
    inputs = [pf_synth.make_inputs(w).to("cuda") for w in CASES]
    want = [_call(w, d) for w, d in zip(CASES, inputs)]
    torch.cuda.synchronize()
    bad = []

    def work(first):
        with torch.cuda.stream(torch.cuda.Stream()):
            for i in range(20):
                n = (first + i) % len(CASES)
                O, S = _call(CASES[n], inputs[n])
                torch.cuda.current_stream().synchronize()
                if not (torch.equal(O, want[n][0]) and torch.equal(S, want[n][1])):
                    bad.append(CASES[n].name)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_the_pool_gives_its_pages_back():
    """A pass whose workspace is tens of MB; its pages stay with the pool until they are asked back, and the next call works."""
    import paper_2504_00492_b200 as pf
    w = Workload("pool_big", B=1, H=4, L=32768, d_k=64, d_v=64, r=1, chunk=64, s0_std=0.1, seed=74)
    d = pf_synth.make_inputs(w).to("cuda")
    O, S = _call(w, d)
    assert pf.pf_last_launch_count() == 3
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    pf.pf_release_workspaces()
    after = torch.cuda.mem_get_info()[0]
    responses = w.B * w.H * w.L * w.d_k * 2                  # (fp16 responses, the largest part)
    assert after - before >= responses, (before, after)
    pf.pf_release_workspaces()                               # nothing left: no error
    O2, S2 = _call(w, d)
    assert torch.equal(O, O2) and torch.equal(S, S2)
