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
