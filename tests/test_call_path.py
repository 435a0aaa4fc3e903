"""The native call path of the Python entry points: what goes wrong on it arrives as a Python exception."""
import os
import subprocess
import sys

import pytest
import torch

import pf_synth
from pf_synth import Workload

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = """
import torch
from torch._subclasses.fake_tensor import FakeTensorMode
import paper_2504_00492_b200 as pf
with FakeTensorMode():
    e = lambda *s: torch.empty(*s, dtype=torch.bfloat16, device="cuda:0")
    try:
        pf.pf_deltanet_fwd(e(1, 2, 70, 64), e(1, 2, 70, 2, 64), e(1, 2, 70, 2, 64), e(1, 2, 70, 2), None, 64)
    except RuntimeError as x:
        print("raised", x)
"""


def test_tensors_without_storage_raise():
    """(In a process of its own: a C++ exception that leaves the extension ends the interpreter.)"""
    p = subprocess.run([sys.executable, "-c", FAKE], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert p.returncode == 0 and p.stdout.startswith("raised"), (p.returncode, p.stdout, p.stderr[-2000:])


@pytest.mark.gpu
def test_no_memory_for_the_outputs_raises():
    import paper_2504_00492_b200 as pf
    w = Workload("no_memory", B=1, H=4, L=8192, d_k=64, d_v=128, r=1, chunk=64, s0_std=0.1, seed=91)
    d = pf_synth.make_inputs(w).to("cuda")
    O, S = pf.pf_deltanet_fwd(d.q, d.k, d.v, d.beta, d.S0, w.chunk)
    torch.cuda.synchronize()
    keep = O.clone()
    del O
    torch.cuda.empty_cache()
    total = torch.cuda.get_device_properties(0).total_memory
    torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + (2 << 20)) / total)      # (O takes 16 MB)
    try:
        with pytest.raises(torch.OutOfMemoryError):
            pf.pf_deltanet_fwd(d.q, d.k, d.v, d.beta, d.S0, w.chunk)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    O, S2 = pf.pf_deltanet_fwd(d.q, d.k, d.v, d.beta, d.S0, w.chunk)
    assert torch.equal(O, keep) and torch.equal(S2, S)


@pytest.mark.gpu
@pytest.mark.parametrize("entry", ["plain", "ex", "ex, own workspace"])
def test_the_stream_is_the_tensors_devices(entry):
    """The current stream of the tensors' device is used, also while another device is current; with one device, that it
    is the current stream and not the default one: work queued on it before the call is seen by the call."""
    import paper_2504_00492_b200 as pf
    here = torch.device("cuda", torch.cuda.device_count() - 1)
    w = Workload("stream", B=1, H=2, L=300, d_k=128, d_v=128, r=2, chunk=64, s0_std=0.1, seed=92)
    d = pf_synth.make_inputs(w).to(here)
    ref, _ = pf.pf_deltanet_fwd(d.q, d.k, d.v, d.beta, d.S0, w.chunk)
    torch.cuda.synchronize(here)
    filled = torch.zeros_like(d.v)
    s = torch.cuda.Stream(device=here)
    ws = torch.empty(pf.pf_workspace_bytes(w.B, w.H, w.L, w.d_k, w.d_v, w.r, w.chunk), dtype=torch.uint8, device=here)
    torch.cuda.synchronize(here)
    with torch.cuda.stream(s):
        torch.cuda._sleep(20_000_000)                  # (about 10 ms: a call on another stream would be through before)
        filled.copy_(d.v, non_blocking=True)
        with torch.cuda.device(0):
            args = (d.q, d.k, filled, d.beta, d.S0, w.chunk)
            if entry == "plain":
                O, _ = pf.pf_deltanet_fwd(*args)
            else:
                O, _ = pf.pf_deltanet_fwd_ex(*args, workspace=ws if "own" in entry else None)
    s.synchronize()
    assert torch.equal(O, ref)
