"""bench.py's account of what the kernel it timed has done: the form, the chunk length and the peak are that kernel's own."""
import pytest

import bench
import pf_synth

PEAKS = {"hbm_gbs": 6500.0, "bf16_tflops": 1600.0, "sm_max_mhz": 1965.0}


def test_token_by_token_kernel_is_bound_by_ffma():
    w = pf_synth.CONFIGS["c0"]                               # fp32, 256 tokens, d = 64, r = 1
    r = bench.kernel_roofline({"recur": 0.02, "recur_compose": 0.001, "recur_apply": 0.001}, w, 64, PEAKS, "measured")
    flops = 256 * 6 * 64 * 64
    assert r["kernel"] == "recur" and r["bound"] == "alu" and r["unit"] == "TFLOP/s"
    assert r["peak"] == pytest.approx(148 * 128 * 2 * 1965e6 / 1e12)
    assert r["achieved"] == pytest.approx(flops / 20e-6 / 1e12)
    assert bench.chunk_of("recur", w, 64) == 1
    assert "bf16" not in r and "tensor" not in r


def test_chain_kernel_is_counted_in_its_own_blocks():
    w = pf_synth.CONFIGS["c3"]                               # 128 sequences of 4096, d = 64, r = 4
    assert bench.chunk_of("chain", w, 32) == 16
    n, d, C = 64, 64, 16
    per_block = 2 * n * n * d * 2 + 2 * C * n * d * 2 + 2 * n * d * d * 2 + 2 * C * d * d
    assert bench.pass_flops("chain", w, 32, tri=False, solve=False) == 128 * 4096 / 16 * per_block
    r = bench.kernel_roofline({"chain": 0.35}, w, 32, PEAKS, "measured")
    nbytes = w.token_heads * bench.alg_bytes_per_token_head(w)
    assert r["bound"] == "hbm" and r["achieved"] == pytest.approx(nbytes / 0.35e-3 / 1e9)
    assert r["tensor"]["tflops_dense"] == pytest.approx(128 * 256 * per_block / 0.35e-3 / 1e12)
    assert r["tensor"]["pipe_active_pct"] is None            # (no capture of this kernel at this size)


def test_kernels_that_follow_in_segments_are_part_of_the_pass():
    w = pf_synth.CONFIGS["c2"]
    r = bench.kernel_roofline({"chain": 0.18, "chain_compose": 0.01, "chain_apply": 0.06}, w, 64, PEAKS, "measured")
    nbytes = w.token_heads * bench.alg_bytes_per_token_head(w)
    assert r["kernel"] == "chain" and r["bound"] == "hbm" and r["achieved"] == pytest.approx(nbytes / 0.25e-3 / 1e9)
    assert r["frac"] == pytest.approx(r["achieved"] / PEAKS["hbm_gbs"])


def test_single_launch_keeps_the_chunk_form():
    w = pf_synth.CONFIGS["c2"]
    assert bench.chunk_of("fused", w, 64) == 64
    fl = bench.flops_per_chunk(w, tri=False)
    want = 32 * 128 * (sum(fl.values()) - fl["solve"])
    r = bench.kernel_roofline({"fused": 0.25}, w, 64, PEAKS, "measured")
    assert r["bound"] == "hbm" and r["tensor"]["tflops_dense"] == pytest.approx(want / 0.25e-3 / 1e12)


def test_kernels_of_a_part_of_the_chunk_form():
    w = pf_synth.CONFIGS["c2"]
    for kernel, bound in (("simt_wu", "alu"), ("tc_flow", "tensor")):
        r = bench.kernel_roofline({kernel: 0.4, "other": 0.1}, w, 64, PEAKS, "measured")
        assert r["kernel"] == kernel and r["bound"] == bound and r["unit"] == "TFLOP/s"


def test_the_l2_note_says_what_is_so():
    assert "larger than L2" in bench.l2_note(471_000_000)
    assert "larger" not in bench.l2_note(86_000_000)
