"""Performance cases of darkattn: what a program that uses the library has it do, through the public entry points.

A case is one of three kinds of call:
  "forward"  darkattn_forward without a stash: a prompt (causal) or an encoder layer (not causal) at inference
  "train"    darkattn_forward with its stash, then darkattn_backward (and darkattn_backward_dw where "dw" is set: the
             projections are trained too)
  "decode"   darkattn_decode_step: one token per sequence added to the running state
Queries and keys are anisotropic Gaussians (covariance spectrum lambda_i ~ rho^i of trace d in a random basis, as in the
library's synthetic workloads), values and output gradients standard normal, M near the identity, W standard normal.
"""
import math

import torch

from paper_2603_04127_b200 import binding

# Every case states all of these.
_FIELDS = ("kind", "dtype", "causal", "B", "H", "H_kv", "N", "d", "r", "dv", "m", "dw")


def _case(kind, dtype, causal, B, H, N, d, m, H_kv=0, r=0, dv=0, dw=False, name=None):
    c = dict(zip(_FIELDS, (kind, dtype, causal, B, H, H_kv or H, N, d, r or d, dv or d, m, dw)))
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # serving, one decode step of a few sequences: one short launch, the caller waits for it at every token
        _case("decode", "bf16", True, 4, 16, 1, 128, 256, name="decode_small"),
        # serving with many sequences at once: the running state (134 MB) is read and written at every token
        _case("decode", "bf16", True, 64, 16, 1, 128, 256, name="decode_large"),
        # the smallest configuration: one head of 256 tokens in single precision (launch latencies)
        _case("forward", "f32", False, 1, 1, 256, 64, 64, name="f32_one_head"),
        # a short prompt of a single request; prompt lengths are whatever the user typed
        _case("forward", "bf16", True, 1, 12, 333, 64, 256, name="prompt_short_odd"),
        # an ordinary batch of prompts of odd length, keys and values shared by groups of four heads
        _case("forward", "bf16", True, 2, 16, 2001, 128, 256, H_kv=4, name="prompt_odd_grouped"),
        # encoder layer, no mask (8 x 12 heads of 4096 tokens)
        _case("forward", "bf16", False, 8, 12, 4096, 64, 256, name="encoder"),
        # prefill of long prompts (4 x 16 heads of 8192 tokens, width 128)
        _case("forward", "bf16", True, 4, 16, 8192, 128, 256, name="prefill_8k"),
        # prefill of one very long document: few heads, 65536 tokens, 512 features
        _case("forward", "bf16", True, 1, 8, 65536, 64, 512, name="prefill_64k"),
        # training step of a small model (8 x 12 heads of 2048 tokens)
        _case("train", "bf16", True, 8, 12, 2048, 64, 256, name="train_2k"),
        # training step of the benchmark's headline shape, causal and without the mask
        _case("train", "bf16", True, 4, 16, 8192, 128, 256, name="train_8k"),
        _case("train", "bf16", False, 4, 16, 8192, 128, 256, name="train_8k_no_mask"),
        # single-precision training at an odd length, the projections trained as well
        _case("train", "f32", True, 2, 8, 1000, 64, 128, dw=True, name="f32_train_dw"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("decode", "forward", "forward", "train", "train", "exact"))
    H = rng.choice((8, 12, 16))
    d = rng.choice((64, 128))
    m = rng.choice((128, 256, 512))
    dv = rng.choice((d, d, d, 64, 128))
    r = rng.choice((d, d, d, 32, 64))
    H_kv = rng.choice((H, H, H, H // 4, H // 2))
    if kind == "decode":
        B = _log_int(rng, 1, min(64, 64 * 16 * 256 * 128 // (H * m * dv)))
        return _case("decode", rng.choice(("bf16", "bf16", "bf16", "f32")), True, B, H, 1, d, m, H_kv=H_kv, r=r, dv=dv)
    if kind == "exact":         # single precision: any length, whole step or forward pass; smaller problems
        N = _log_int(rng, 64, 4096)
        B = max(1, min(_log_int(rng, 1, 8), 2 * 16 * 2001 * 256 // (H * N * max(m, 256))))
        what = rng.choice(("forward", "train"))
        return _case(what, "f32", rng.random() < 0.7, B, H, N, d, m, H_kv=H_kv, r=r, dv=dv, dw=what == "train" and rng.random() < 0.5)
    causal = rng.random() < 0.7
    if rng.random() < 0.4:      # lengths as they come
        N = _log_int(rng, 64, 8192)
        N += N % 128 == 0
        most = 2 * 16 * 2001 * 256
    else:                       # sequences packed or padded to the chunk length
        N = 128 * _log_int(rng, 1, 512 if kind == "forward" and causal else 64)
        most = 4 * 16 * 8192 * 256
    B = max(1, min(_log_int(rng, 1, 16), most // (H * N * max(m, 256))))
    while B * H * N * m > most and m > 128:
        m //= 2
    while B * H * N * max(m, 256) > most:
        H, H_kv = H // 2, max(1, H_kv // 2)
    return _case(kind, "bf16", causal, B, H, N, d, m, H_kv=H_kv if H % H_kv == 0 else H, r=r, dv=dv, dw=kind == "train" and rng.random() < 0.2)


def _dtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.bfloat16


def prepare(case, seed):
    B, H, Hkv, N, d, r, dv, m = (case[k] for k in ("B", "H", "H_kv", "N", "d", "r", "dv", "m"))
    dt = _dtype(case)
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device="cuda")

    basis = torch.linalg.qr(normal(d, d))[0]
    rho = 0.95 if d > 64 else 0.9
    lam = rho ** torch.arange(d, device="cuda", dtype=torch.float32)
    root = (lam * (d / lam.sum())).sqrt()[:, None] * basis.T

    def rows(*shape):                           # anisotropic queries and keys
        return (normal(*shape, d) @ root).to(dt)

    plan = binding.darkattn_plan(B, H, N, d, m, r=r, dv=dv, dtype=binding.F32 if case["dtype"] == "f32" else binding.BF16,
                                 causal=case["causal"], H_kv=0 if Hkv == H else Hkv)
    s = {"kind": case["kind"], "plan": plan,
         "M": (torch.eye(r, d, device="cuda") + 0.1 / math.sqrt(d) * normal(H, r, d)).to(dt), "W": normal(m, r).to(dt)}
    if case["kind"] == "decode":
        s.update(q=rows(B, H), k=rows(B, Hkv), v=normal(B, Hkv, dv).to(dt), o=torch.empty(B, H, dv, dtype=dt, device="cuda"))
        # a state some hundred tokens old: sums of positive features, and of the same times the tokens' values
        z = 1e-3 * torch.exp(2 * normal(B, H, m))
        s.update(z=z, S=0.2 * z[..., None] * normal(B, H, m, dv))
        return s
    s.update(Q=rows(B, H, N), K=rows(B, Hkv, N), V=normal(B, Hkv, N, dv).to(dt), O=torch.empty(B, H, N, dv, dtype=dt, device="cuda"),
             workspace=plan.alloc_workspace(), saved=None)
    if case["kind"] == "train":
        if plan.saved_bytes:
            s["saved"] = torch.empty(plan.saved_bytes, dtype=torch.uint8, device="cuda")
        s.update(dO=normal(B, H, N, dv).to(dt), dQ=torch.empty_like(s["Q"]), dK=torch.empty_like(s["K"]), dV=torch.empty_like(s["V"]),
                 dM=torch.empty(H, r, d, dtype=torch.float32, device="cuda"),
                 dW=torch.empty(m, r, dtype=torch.float32, device="cuda") if case["dw"] else None)
    return s


def run(s):
    if s["kind"] == "decode":
        binding.darkattn_decode_step(s["plan"], s["q"], s["k"], s["v"], s["M"], s["W"], s["S"], s["z"], s["o"])
        return s["o"], s["S"], s["z"]
    binding.darkattn_forward(s["plan"], s["Q"], s["K"], s["V"], s["M"], s["W"], s["O"], s["workspace"], saved=s["saved"])
    if s["kind"] == "forward":
        return s["O"]
    binding.darkattn_backward(s["plan"], s["Q"], s["K"], s["V"], s["M"], s["W"], s["O"], s["dO"], s["dQ"], s["dK"], s["dV"], s["dM"],
                              s["workspace"], saved=s["saved"])
    if s["dW"] is not None:
        binding.darkattn_backward_dw(s["plan"], s["M"], s["dW"], s["workspace"])
    return s["O"], s["dQ"], s["dK"], s["dV"], s["dM"], s["dW"]


def work(case):
    """Bytes: every input read once, every output written once. Operations: the method's own products. The feature map
    of one row takes 2 d r + 2 r m (x -> Mx -> W Mx); the contraction 4 m dv per token and head; a causal chunk of C =
    128 tokens the lower triangle of its kernel values, (C + 1)(m + dv) per token. The backward pass has each product of
    the forward pass twice, once for each factor's gradient."""
    B, H, Hkv, N, d, r, dv, m = (case[k] for k in ("B", "H", "H_kv", "N", "d", "r", "dv", "m"))
    e = 4 if case["dtype"] == "f32" else 2
    features = 2 * (2 * d * r + 2 * r * m)
    params = (H * r * d + m * r) * e
    if case["kind"] == "decode":
        state = 4 * B * H * m * (dv + 1)
        return {"bytes": 2 * state + params + e * B * (H * (d + dv) + Hkv * (d + dv)), "flops": B * H * (features + 4 * m * dv)}
    flops = features + 4 * m * dv + ((min(128, N) + 1) * (m + dv) if case["causal"] else 0)
    nbytes = params + e * B * N * (H * (d + dv) + Hkv * (d + dv))
    if case["kind"] == "train":
        flops *= 3
        # dO in; dQ, dK, dV in the storage type and dM (dW) in single precision out
        nbytes += e * B * N * (H * (d + dv) + Hkv * (d + dv)) + 4 * (H * r * d + (m * r if case["dw"] else 0))
    return {"bytes": nbytes, "flops": B * H * N * flops}


def tolerance(case):
    # single precision: sums of 32-bit products behind an exponential whose argument is such a sum
    if case["dtype"] == "f32":
        return {"rel": 1e-5}
    # decode: the state is kept in single precision; the output row is rounded to bf16 once (2^-8 of its value at most)
    if case["kind"] == "decode":
        return {"rel": 1e-3, "max": 0.01}
    return {"rel": 1e-2}
