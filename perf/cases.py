"""The calls a user of this library makes, as timed cases: prefill, training steps and decode through the public entry points.

A case names its path and its sizes:

    path   "forward"  prefill / evaluation: entmax_attn_fwd (or _fwd_ex with ALiBi slopes) with a workspace the program keeps
           "train"    a training step through torch autograd (entmax_attention): O and every gradient
           "layer"    a training step of a layer with the content-dependent scale: projection, attention, both backwards
           "decode"   new query rows against a key/value cache, sequences of different lengths
    keys   "gauss"    Q, K ~ N(0, 1)
           "planted"  N(0, 1) with `plant` matching keys per planted query (associative recall)
           "needle"   a faint background (sigma 0.25) with `plant` matching keys per planted query
           "init"     logits of a freshly initialised model (sigma 0.03): every row's support has thousands of keys
    scale  "none"     c = 1
           "length"   ASEntmax, c_i = delta + beta (ln n_i)^gamma with beta, gamma, delta ~ U[0.5, 1.5] per head
           "paper"    the values the paper's learned scale settles at: beta = 1, gamma = -0.5, delta = 1
           "rows"     a table c[b, h, i] that the scale projection computes ("layer")
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2506_16640_b200 import binding
from paper_2506_16640_b200.autograd import entmax_attention


def _case(name, path, B, H, N, d, dtype="bf16", causal=True, alpha=1.5, keys="gauss", plant=0, scale="length", nape=False,
          keep=False, d_model=0, q_len=0, ragged=False):
    c = dict(path=path, B=B, H=H, N=N, d=d, dtype=dtype, causal=causal, alpha=alpha, keys=keys, plant=plant, scale=scale,
             nape=nape, keep=keep, d_model=d_model, q_len=q_len, ragged=ragged)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one short fp32 call, as in a unit test or a numerics comparison: latency
        _case("fp32_fwd_n128", "forward", 1, 2, 128, 64, dtype="fp32", scale="none"),
        # an fp32 training step at a ragged length: debugging a model at full precision
        _case("fp32_train_n777", "train", 2, 4, 777, 64, dtype="fp32"),
        # a training step of the 12-head, 1024-token learned-scale study
        _case("train_8x12x1024_d64", "train", 8, 12, 1024, 64, keys="planted", plant=4),
        # a training step of a 64-wide-head language model at 8192 tokens, supports kept for the backward pass
        _case("train_4x16x8192_d64", "train", 4, 16, 8192, 64, keep=True),
        # a training step at 32768 tokens, the length the library is quoted at
        _case("train_16x32768_d128", "train", 1, 16, 32768, 128, keys="planted", plant=8),
        # a ragged prefill with a denser map (alpha = 1.25)
        _case("prefill_16x20011_d128_a125", "forward", 1, 16, 20011, 128, alpha=1.25, keys="planted", plant=8),
        # a non-causal retrieval model trained at 65536 tokens
        _case("train_retrieval_8x65536_d64", "train", 1, 8, 65536, 64, causal=False, keys="needle", plant=4),
        # the first steps of a training run: near-uniform attention, supports in the thousands
        _case("train_init_16x8192_d128", "train", 1, 16, 8192, 128, keys="init"),
        # one layer of the full method: beta and gamma projected from the layer input, ragged length
        _case("layer_2x12x3001_d64", "layer", 2, 12, 3001, 64, scale="rows", d_model=768),
        # NAPE (ALiBi slopes on half of the heads) at the temperature the paper's learned scale settles at, sparsemax
        _case("train_nape_12x6000_d64_a2", "train", 1, 12, 6000, 64, alpha=2.0, scale="paper", nape=True),
        # generating one token of one long sequence
        _case("decode_1x16x32768_d128_q1", "decode", 1, 16, 32768, 128, keys="planted", plant=8, q_len=1),
        # a serving batch: eight sequences of different lengths, four new rows each, token-major cache
        _case("decode_8x16x16384_d128_q4", "decode", 8, 16, 16384, 128, q_len=4, ragged=True),
    ]


def _log_int(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]; half of them multiples of 64 where the range allows.  Lengths of
    1921 ... 2047 are rounded up to 2048: the dense-tile forward kernel first measured with this file could not take them."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    n = max(64, n // 64 * 64) if n >= 128 and rng.random() < 0.5 else n
    return 2048 if 1920 < n < 2048 else n


# visible (query, key) pairs x head_dim a drawn case may have: the 32768-token training step's, and what the paths that
# cost more per pair may take of it
_PAIRS = 16 * 32768 * 32769 // 2 * 128


def _heads(rng, N, d, causal, share=1.0):
    """Batch and heads from the configurations in use, as many as keep the case below the largest listed one."""
    per = N * (N + 1) // 2 if causal else N * N
    room = max(1, int(share * _PAIRS / (per * d)))
    fits = [(B, H) for B in (1, 2, 4, 8) for H in (1, 2, 4, 8, 12, 16) if B * H <= min(room, 128)]
    return rng.choice(fits[len(fits) // 2:])


def draw(rng):
    path = rng.choice(["fp32", "forward", "forward", "train", "train", "train", "init", "layer", "decode", "decode"])
    d = rng.choice([64, 128])
    alpha = rng.choice([1.25, 1.5, 1.5, 1.5, 1.7, 2.0])
    if path == "fp32":
        N = _log_int(rng, 64, 1500)
        return _case(None, rng.choice(["forward", "train"]), rng.choice([1, 2]), rng.choice([1, 2, 4]), N, d, dtype="fp32",
                     causal=rng.random() < 0.7, alpha=alpha, scale=rng.choice(["none", "length"]))
    if path == "decode":
        N = _log_int(rng, 512, 65536)
        B = rng.choice([b for b in (1, 2, 4, 8, 16) if b * N <= 1 << 18])
        return _case(None, "decode", B, rng.choice([8, 12, 16]), N, d, alpha=alpha, keys=rng.choice(["gauss", "planted"]),
                     plant=8, q_len=rng.randint(1, 8), ragged=B > 1)
    if path == "layer":
        N = _log_int(rng, 512, 8192)
        B, H = _heads(rng, N, d, True, 0.1)
        return _case(None, "layer", B, H, N, d, alpha=alpha, scale="rows", d_model=H * d)
    if path == "init":
        N = _log_int(rng, 512, 8192)
        B, H = _heads(rng, N, d, True, 0.05)
        return _case(None, rng.choice(["forward", "train"]), B, H, N, d, alpha=alpha, keys="init")
    causal = rng.random() < 0.8
    keys = rng.choice(["gauss", "planted", "planted"] if causal else ["planted", "needle"])
    # the denser maps cost more per pair: shorter problems there
    N = _log_int(rng, 256, 32768 if alpha >= 1.5 and keys != "gauss" else 12000)
    B, H = _heads(rng, N, d, causal, 0.5)
    nape = causal and keys == "gauss" and rng.random() < 0.4
    return _case(None, path, B, H, N, d, causal=causal, alpha=alpha, keys=keys, plant=0 if keys == "gauss" else rng.choice([4, 8]),
                 scale="paper" if nape and alpha >= 1.5 else "length", nape=nape, keep=path == "train" and rng.random() < 0.5)


# ------------------------------------------------------------------------------------------------------------ inputs
def _planted_slots(n_heads, N, p, causal, rng):
    """Key slots [n_heads, R, p] of the planted queries i = p, 2p+1, ...: each takes p slots uniformly from the still free
    ones it can see."""
    rows = np.arange(p, N, p + 1)
    u = rng.random((len(rows) * p, n_heads))
    free = np.zeros((n_heads, N + p + 1), dtype=np.int64)
    slots = np.empty((n_heads, len(rows) * p), dtype=np.int64)
    every = np.arange(n_heads)
    if not causal:
        free[:, :N] = np.arange(N)
    m, seen = (0, 0) if causal else (N, N)
    for r, i in enumerate(rows):
        if seen <= i:
            free[:, m:m + i + 1 - seen] = np.arange(seen, i + 1)
            m, seen = m + i + 1 - seen, i + 1
        for t in range(r * p, r * p + p):
            x = (u[t] * m).astype(np.int64)
            slots[:, t] = free[every, x]
            m -= 1
            free[every, x] = free[:, m]
    return rows, slots.reshape(n_heads, len(rows), p)


def _qkv(case, seed):
    B, H, N, d = case["B"], case["H"], case["N"], case["d"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    sigma = {"gauss": 1.0, "planted": 1.0, "needle": 0.25, "init": 0.03}[case["keys"]]
    draw_one = lambda s: (torch.randn((B, H, N, d), generator=gen, device="cuda") * s).to(dt)
    q, k, v, d_o = draw_one(sigma), draw_one(sigma), draw_one(1.0), draw_one(1.0)
    if case["keys"] in ("planted", "needle") and case["plant"] > 0:
        rows, slots = _planted_slots(B * H, N, case["plant"], case["causal"], np.random.default_rng(seed))
        qi = q.view(B * H, N, d)[:, torch.from_numpy(rows).cuda()].float()                        # [BH, R, d]
        dirs = qi / qi.norm(dim=-1, keepdim=True).clamp_min(1e-20)
        noise = torch.randn((B * H, len(rows), case["plant"], d), generator=gen, device="cuda") * 0.1
        planted = (3.0 * math.sqrt(d) * dirs[:, :, None] + noise).to(dt).reshape(B * H, -1, d)
        at = torch.from_numpy(slots.reshape(B * H, -1)).cuda()[:, :, None].expand(-1, -1, d)
        k.view(B * H, N, d).scatter_(1, at, planted)
    u = lambda: torch.rand((H,), generator=gen, device="cuda") + 0.5
    if case["scale"] == "length":
        scale = (u(), u(), u())
    elif case["scale"] == "paper":
        scale = tuple(torch.full((H,), x, device="cuda") for x in (1.0, -0.5, 1.0))
    else:
        scale = (None, None, None)
    slopes = None
    if case["nape"]:      # half of the heads, geometric slopes
        half = max(1, H // 2)
        slopes = torch.tensor([2.0 ** (-8.0 * (h + 1) / half) if h < half else 0.0 for h in range(H)], device="cuda")
    return gen, q, k, v, d_o, scale, slopes


def prepare(case, seed):
    gen, q, k, v, d_o, scale, slopes = _qkv(case, seed)
    B, H, N, d = case["B"], case["H"], case["N"], case["d"]
    st = dict(case=case, q=q, k=k, v=v, scale=scale, slopes=slopes)
    if case["path"] == "forward":
        st["workspace"] = binding.alloc_workspace(binding.make_params(q, case["alpha"], case["causal"]), False, q.device)
    elif case["path"] == "train":
        st["d_o"] = d_o
        st["params"] = [t.requires_grad_() for t in (q, k, v) + scale if t is not None]
    elif case["path"] == "layer":
        st["d_o"] = d_o
        st["x"] = torch.randn((B, N, case["d_model"]), generator=gen, device="cuda").to(q.dtype)
        s = 1.0 / math.sqrt(case["d_model"])
        st["w_beta"] = torch.randn((H, case["d_model"]), generator=gen, device="cuda") * s
        st["w_gamma"] = torch.randn((H, case["d_model"]), generator=gen, device="cuda") * s
        st["delta"] = torch.rand((H,), generator=gen, device="cuda") + 0.5
    else:
        # the cache is token-major [B, capacity, H, d]; the new rows are the last q_len tokens of each sequence
        token_major = lambda t: t.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)
        lens = torch.full((B,), N, dtype=torch.int64)
        if case["ragged"]:
            lens = torch.from_numpy(np.random.default_rng(seed).integers(max(8, N // 4), N + 1, size=B))
            lens[0] = N
        at = (lens[:, None] - case["q_len"] + torch.arange(case["q_len"])).cuda()                # [B, q_len]
        st["q"] = q.gather(2, at[:, None, :, None].expand(-1, H, -1, d)).contiguous()
        st["k"], st["v"] = token_major(k), token_major(v)
        st["kv_len"] = lens.to(torch.int32).cuda()
    return st


def run(st):
    c = st["case"]
    q, k, v, alpha, causal = st["q"], st["k"], st["v"], c["alpha"], c["causal"]
    beta, gamma, delta = st["scale"]
    if c["path"] == "forward":
        if st["slopes"] is None:
            return binding.entmax_attn_fwd(q, k, v, alpha, causal, beta, gamma, delta, workspace=st["workspace"])
        return binding.entmax_attn_fwd_ex(q, k, v, alpha, causal, beta, gamma, delta, alibi_slopes=st["slopes"],
                                          workspace=st["workspace"])
    if c["path"] == "train":
        o, tau = entmax_attention(q, k, v, beta, gamma, delta, alibi_slopes=st["slopes"], alpha=alpha, causal=causal,
                                  keep_supports=c["keep"], return_tau=True)
        return (o.detach(), tau) + torch.autograd.grad(o, st["params"], st["d_o"])
    if c["path"] == "layer":
        x, wb, wg = st["x"], st["w_beta"], st["w_gamma"]
        c_rows = binding.entmax_attn_scale_proj_fwd(x, wb, wg, st["delta"], 1.0, causal)
        o, tau = binding.entmax_attn_fwd_rowscale(q, k, v, c_rows, alpha, causal)
        dq, dk, dv, dc = binding.entmax_attn_bwd_rowscale(q, k, v, c_rows, tau, st["d_o"], alpha, causal)
        return (c_rows, o, tau, dq, dk, dv, dc) + binding.entmax_attn_scale_proj_bwd(x, wb, wg, dc, 1.0, causal)
    return binding.entmax_attn_decode_fwd(q, k, v, alpha, st["kv_len"], beta, gamma, delta)


def work(case):
    """One contraction of scores is what sparse rows cannot do without (the supports it finds are a few keys per row); rows
    with supports in the thousands need P V and the five contractions of the backward pass too."""
    B, H, N, d = case["B"], case["H"], case["N"], case["d"]
    el = 2 if case["dtype"] == "bf16" else 4
    if case["path"] == "decode":
        keys = H * N * (1 + 0.625 * (B - 1) if case["ragged"] else B)     # mean length of a ragged batch
        return {"bytes": keys * d * el, "flops": 2.0 * d * keys * case["q_len"]}
    pairs = N * (N + 1) // 2 if case["causal"] else N * N
    heads = B * (H - max(1, H // 2)) if case["nape"] else B * H        # the window leaves the ALiBi heads little
    step = case["path"] != "forward"
    per_pair = 2 * d if case["keys"] != "init" else (14 * d if step else 4 * d)
    tensors = 8 if step else 4
    nbytes = B * H * N * (d * el * tensors + 4) + (2 * B * N * case["d_model"] * el if case["path"] == "layer" else 0)
    flops = per_pair * heads * pairs + (12 * B * N * H * case["d_model"] if case["path"] == "layer" else 0)
    return {"bytes": float(nbytes), "flops": float(flops)}


def tolerance(case):
    """About four times what the outputs differ by from a float64 evaluation of the same inputs (N up to 1800, every alpha and
    kind of keys): float32 1.2e-5 and at most 1.1e-3 of an entry; bfloat16 2.3e-3 (one rounding of the result is 1.7e-3, P is
    rounded too on dense rows) and at most 1.6e-2 there, more in problems with more entries.  At alpha = 2 the Jacobian jumps
    when a key crosses the threshold, so single entries of the gradients may be off."""
    if case["dtype"] == "fp32":
        return {"rel": 5e-5, "max": 5e-3, "differ": 0.0}
    return {"rel": 1e-2, "max": 0.9 if case["alpha"] >= 2.0 else 0.2, "differ": 0.01}
