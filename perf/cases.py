"""Performance cases of the delta-rule forward pass: the calls a user of this library makes, through its public entry
points, from a single decoded token to a long-context prefill.

A case is a dict of plain values:
    dtype            "bf16" (pf_deltanet_fwd) or "f32" (pf_deltanet_fwd_f32): the type of q, k, v and beta
    B, H, L          batch, heads, tokens per sequence
    d_k, d_v, r      head dimensions and rank (factors per token)
    chunk            the chunk length the caller asks for
    s0               whether the call starts from a state (a continued sequence) or from zero
    beta_scale       beta = beta_scale * sigmoid(N(0, 1)): 1 as in the delta rule, 2 where negative eigenvalues are wanted
    mode, step       options of pf_deltanet_fwd_ex; with both at their defaults the plain entry point is called
"""
import math

import torch

import paper_2504_00492_b200 as pf


def _case(name, B, H, L, d_k, d_v, r, chunk, dtype="bf16", s0=True, beta_scale=1.0, mode="sum", step="euler"):
    return {"name": name, "dtype": dtype, "B": B, "H": H, "L": L, "d_k": d_k, "d_v": d_v, "r": r, "chunk": chunk,
            "s0": s0, "beta_scale": beta_scale, "mode": mode, "step": step}


def listed():
    return [
        # one short fp32 sequence of one head: a unit check or a small research model; latency and launches count
        _case("f32_one_head", 1, 1, 256, 64, 64, 1, 64, dtype="f32", s0=False),
        # one decoded token for a batch of running sequences: state in, state out
        _case("decode_one_token", 8, 16, 1, 128, 128, 2, 64),
        # a prompt of a few hundred tokens, not a multiple of the chunk
        _case("prefill_short_ragged", 1, 16, 333, 128, 128, 2, 64),
        # rank 1 (plain DeltaNet), training-like batch of ordinary length
        _case("rank1_2k", 4, 8, 2048, 128, 128, 1, 64),
        # many sequences of ordinary length: a training micro-batch or a full serving batch
        _case("many_sequences_1k", 16, 16, 1024, 128, 128, 2, 64),
        # rank 3 with the factors of a token applied one after another, mixed head dimensions, ragged length
        _case("rank3_product_ragged", 4, 12, 1999, 64, 128, 3, 32, beta_scale=2.0, mode="product"),
        # one long document, few heads
        _case("few_heads_16k", 1, 4, 16384, 128, 128, 1, 64, s0=False),
        # the benchmark's workload: rank 2, 8192 tokens
        _case("rank2_8k", 2, 16, 8192, 128, 128, 2, 64, s0=False),
        # rank 4 at head dimension 64, beta in (0, 2)
        _case("rank4_d64_4k", 8, 16, 4096, 64, 64, 4, 64, s0=False, beta_scale=2.0),
        # long context: 65536 tokens, state carried in and out
        _case("rank2_64k", 1, 32, 65536, 128, 128, 2, 64),
        # fp32 throughout: a run that a bf16 model is validated against
        _case("f32_rank2_2k", 4, 8, 2048, 128, 128, 2, 64, dtype="f32"),
        # fp32, head dimension 64, ragged length, shorter chunk
        _case("f32_d64_ragged", 2, 8, 1000, 64, 64, 2, 32, dtype="f32"),
    ]


# What a call may cost at most, in elements of q, k, v and O per call: the largest listed case of its type.
_MOST = {"bf16": 32 * 65536 * (128 + 4 * 128 + 128), "f32": 32 * 2048 * (128 + 4 * 128 + 128)}


def draw(rng):
    def log_int(lo, hi):
        return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    dtype = "f32" if rng.random() < 0.25 else "bf16"
    H = log_int(1, 32)
    B = log_int(1, 16)
    d_k, d_v = rng.choice(((128, 128), (128, 128), (64, 64), (64, 128), (128, 64)))
    r = rng.choice((1, 1, 2, 2, 3, 4))
    L = 1 if rng.random() < 0.15 else log_int(2, 65536)
    most = _MOST[dtype] // (B * H * (d_k + r * (d_k + d_v) + d_v))
    if L > most:
        L = max(1, int(most * rng.uniform(0.3, 1.0)))
    mode = "product" if r > 1 and rng.random() < 0.3 else "sum"
    step = "exact" if (r == 1 or mode == "product") and rng.random() < 0.2 else "euler"
    case = _case("", B, H, L, d_k, d_v, r, rng.choice((16, 32, 64, 64)), dtype=dtype, s0=L == 1 or rng.random() < 0.6,
                 beta_scale=rng.choice((1.0, 2.0)), mode=mode, step=step)
    del case["name"]
    return case


def prepare(case, seed):
    """Inputs on the GPU: q, v ~ N(0, 1/d), keys L2-normalised one by one, beta = beta_scale * sigmoid(N(0, 1)), a start
    state of entries N(0, 0.01) as an earlier part of the sequence leaves behind."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    B, H, L, r, d_k, d_v = case["B"], case["H"], case["L"], case["r"], case["d_k"], case["d_v"]
    dtype = torch.float32 if case["dtype"] == "f32" else torch.bfloat16

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32)

    q = normal(B, H, L, d_k).mul_(d_k ** -0.5).to(dtype)
    k = normal(B, H, L, r, d_k)
    k = k.div_(k.norm(dim=-1, keepdim=True)).to(dtype)
    v = normal(B, H, L, r, d_v).mul_(d_v ** -0.5).to(dtype)
    beta = torch.sigmoid(normal(B, H, L, r)).mul_(case["beta_scale"]).to(dtype)
    S0 = normal(B, H, d_k, d_v).mul_(0.1) if case["s0"] else None
    return {"case": case, "args": (q, k, v, beta, S0, case["chunk"])}


def run(state):
    """One forward pass: (O [B,H,L,d_v], S_final [B,H,d_k,d_v])."""
    case = state["case"]
    if case["mode"] != "sum" or case["step"] != "euler":
        return pf.pf_deltanet_fwd_ex(*state["args"], mode=case["mode"], step=case["step"])
    if case["dtype"] == "f32":
        return pf.pf_deltanet_fwd_f32(*state["args"])
    return pf.pf_deltanet_fwd(*state["args"])


def work(case):
    """One read of q, k, v, beta and S0, one write of O and S_final; the operations of the recurrence itself: per token
    and head, r products S k and r rank-1 updates of S, and the readout S q."""
    token_heads = case["B"] * case["H"] * case["L"]
    d_k, d_v, r = case["d_k"], case["d_v"], case["r"]
    size = 4 if case["dtype"] == "f32" else 2
    states = case["B"] * case["H"] * d_k * d_v * 4 * (2 if case["s0"] else 1)
    return {"bytes": token_heads * (size * (d_k + r * (d_k + d_v + 1)) + 4 * d_v) + states,
            "flops": token_heads * (4 * r + 2) * d_k * d_v}


def tolerance(case):
    """bf16 inputs are multiplied as 16-bit operands (one rounding of 2^-11 each for the inverse, W, U, the state ...)
    with fp32 sums; fp32 calls keep fp32 throughout."""
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-4}
    return {"rel": 2e-3, "max": 2e-2}
