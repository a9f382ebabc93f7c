"""The work a user of this library has it do, as cases that can be timed and checked.

`listed()` names them, `draw(rng)` gives more of the same ranges, `prepare` makes what a user's
program holds before the call (inputs on the GPU), `run` is one call through the package's public
functions, `work` the bytes and operations the call cannot do without, and `exact` the same
outputs in 64-bit arithmetic by plain torch.

Kinds of case and their ranges (B*H: independent heads; every size may be odd):

    fwd     attn_fwd, the inference forward      bf16 and fp32
    lse     attn_fwd_lse, the training forward   bf16 and fp32
    split   attn_fwd_splitkv with the library's own split: decoding, chunks over a long cache; bf16
    bwd     attn_bwd, reproducible gradients     bf16 and fp32
    fused   attn_bwd(fused=True)                 bf16, d_k = d_v = 64
    qkv     qkv_proj, the input projections      bf16

    bf16    d_k, d_v in {64, 128}; 1..128 heads; 48..32768 queries and keys (split: 1..256 queries
            over 512..65536 keys; qkv: 1..16384 tokens, d_model 256..4096)
    fp32    d_k, d_v multiples of 4 up to 128; 1..32 heads; 32..2048 queries and keys
"""
from __future__ import annotations

import math

import torch

import paper_2606_07713_gb300 as moa


def _attn(name, kind, B, H, Nq, Nk, dk, dv, dtype="bf16", sigma=1.0, plants=0):
    return {"name": name, "kind": kind, "B": B, "H": H, "Nq": Nq, "Nk": Nk, "dk": dk, "dv": dv,
            "dtype": dtype, "sigma": sigma, "plants": plants}


def _qkv(name, B, N, d_model, H, dk, dv):
    return {"name": name, "kind": "qkv", "B": B, "N": N, "d_model": d_model, "H": H, "dk": dk,
            "dv": dv}


def listed():
    return [
        # The smallest call: one head of 128 rows in fp32 (bench.py's workload 1); latency.
        _attn("fwd_f32_small", "fwd", 1, 1, 128, 128, 64, 64, "fp32"),
        # Reference-precision attention over ragged lengths, queries and keys of different lengths.
        _attn("fwd_f32", "fwd", 2, 8, 1000, 1500, 64, 64, "fp32"),
        # Reference-precision training: the fp32 gradients.
        _attn("bwd_f32", "bwd", 1, 8, 1024, 1024, 64, 64, "fp32"),
        # Many short odd-length sequences, as an encoder over patches or sentences has them.
        _attn("fwd_short", "fwd", 16, 12, 197, 197, 64, 64),
        # The training forward (output and log-sum-exp) at d = 64 (bench.py's workload 2).
        _attn("lse_d64", "lse", 4, 16, 2048, 2048, 64, 64),
        # Cross-attention with a narrow value head (bench.py's workload 4).
        _attn("fwd_cross", "fwd", 8, 8, 1024, 4096, 128, 64),
        # The longest prefill, with spread-out scores and dominant keys (bench.py's workload 5).
        _attn("fwd_long", "fwd", 1, 16, 32768, 32768, 128, 128, sigma=8.0, plants=8),
        # Decoding: one query row per head over an odd-length cache.
        _attn("decode", "split", 8, 16, 1, 8191, 128, 128),
        # A chunk of 256 query rows over a long cache (prefill in chunks).
        _attn("chunk", "split", 1, 16, 256, 32768, 128, 128),
        # Training gradients at d = 64 from one kernel (bench.py --pass bwd's workload).
        _attn("bwd_d64", "fused", 4, 16, 2048, 2048, 64, 64),
        # Reproducible training gradients at d = 128.
        _attn("bwd_d128", "bwd", 2, 16, 4096, 4096, 128, 128),
        # The input projections of a wide layer (bench.py --pass qkv --workload 3).
        _qkv("qkv", 2, 8192, 4096, 32, 128, 128),
    ]


def _log_int(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def _heads(rng, most):
    bh = _log_int(rng, 1, most)
    b = rng.choice([x for x in range(1, min(bh, 16) + 1) if bh % x == 0])
    return b, bh // b


# Bounds of a drawn case, so that none costs more than the largest listed one.
_MAX_FLOPS = {("fwd", "bf16"): 4.0e12, ("lse", "bf16"): 2.0e12, ("bwd", "bf16"): 2.0e12,
              ("fused", "bf16"): 1.5e12, ("fwd", "fp32"): 1.2e10, ("lse", "fp32"): 1.2e10,
              ("bwd", "fp32"): 8.0e9, ("split", "bf16"): 1.0e12}
_MAX_BYTES = 1.2e9


def draw(rng):
    kind = rng.choice(["fwd", "fwd", "lse", "split", "split", "bwd", "fused", "qkv", "f32", "f32"])
    while True:
        if kind == "qkv":
            H = rng.choice([4, 8, 12, 16, 20, 32])
            dk, dv = rng.choice([(64, 64), (128, 128), (128, 128), (128, 64), (64, 128)])
            N = _log_int(rng, 1, 8192)
            case = _qkv(None, rng.choice([1, 2]), N, 8 * _log_int(rng, 32, 512), H, dk, dv)
            limit = 1.7e12
        else:
            k, dtype = kind, "bf16"
            sigma = rng.choice([1.0, 1.0, 1.0, 4.0])
            if kind == "f32":
                k, dtype, sigma = rng.choice(["fwd", "lse", "bwd"]), "fp32", 1.0
                B, H = _heads(rng, 32)
                Nq, Nk = _log_int(rng, 32, 2048), _log_int(rng, 32, 2048)
                dk = 4 * rng.randint(4, 32) if rng.random() < 0.4 else rng.choice([32, 64, 128])
                dv = dk if rng.random() < 0.7 else 4 * rng.randint(4, 32)
            elif kind == "split":
                B, H = _heads(rng, 128)
                Nq, Nk = _log_int(rng, 1, 256), _log_int(rng, 512, 65536)
                dk, dv = rng.choice([(64, 64), (128, 128), (128, 128), (128, 64), (64, 128)])
            else:
                B, H = _heads(rng, 128)
                Nk = _log_int(rng, 48, 32768 if kind in ("fwd", "lse") else 8192)
                Nq = Nk if rng.random() < 0.5 else _log_int(
                    rng, 48, 32768 if kind in ("fwd", "lse") else 8192)
                dk, dv = rng.choice([(64, 64), (64, 64), (128, 128), (128, 128), (128, 64), (64, 128)])
                if kind == "fused":
                    dk = dv = 64
            case = _attn(None, k, B, H, Nq, Nk, dk, dv, dtype, sigma)
            limit = _MAX_FLOPS[(k, dtype)]
        del case["name"]
        w = work(case)
        if w["flops"] <= limit and w["bytes"] <= _MAX_BYTES:
            return case


def _normal(gen, shape, dtype, sigma=1.0):
    t = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)
    return t.mul_(sigma).to(dtype)


def _inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if case["kind"] == "qkv":
        d = case["d_model"]
        x = _normal(gen, (case["B"], case["N"], d), torch.bfloat16)
        w = _normal(gen, (d, case["H"] * (2 * case["dk"] + case["dv"])), torch.bfloat16,
                    1.0 / math.sqrt(d))
        return {"x": x, "w": w}
    dt = torch.float32 if case["dtype"] == "fp32" else torch.bfloat16
    B, H, Nq, Nk, dk, dv = (case[n] for n in ("B", "H", "Nq", "Nk", "dk", "dv"))
    q = _normal(gen, (B, H, Nq, dk), dt, case["sigma"])
    k = _normal(gen, (B, H, Nk, dk), dt, case["sigma"])
    v = _normal(gen, (B, H, Nk, dv), dt)
    if case["plants"]:
        # dominant keys: these query rows repeat a key, so one weight is nearly 1
        rows = torch.randint(0, Nq, (case["plants"],), generator=gen, device="cuda")
        keys = torch.randint(0, Nk, (case["plants"],), generator=gen, device="cuda")
        q[:, :, rows] = k[:, :, keys]
    t = {"q": q, "k": k, "v": v}
    if case["kind"] in ("bwd", "fused"):
        t["do"] = _normal(gen, (B, H, Nq, dv), dt)
    return t


def prepare(case, seed):
    state = _inputs(case, seed)
    state["case"] = case
    if case["kind"] in ("bwd", "fused"):
        # what a training step has kept from its forward pass
        state["o"], state["lse"] = moa.attn_fwd_lse(state["q"], state["k"], state["v"])
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "qkv":
        return moa.qkv_proj(state["x"], state["w"], case["H"], case["dk"], case["dv"])
    q, k, v = state["q"], state["k"], state["v"]
    if kind == "fwd":
        return moa.attn_fwd(q, k, v)
    if kind == "lse":
        return moa.attn_fwd_lse(q, k, v)
    if kind == "split":
        return moa.attn_fwd_splitkv(q, k, v)
    return moa.attn_bwd(q, k, v, state["o"], state["lse"], state["do"], fused=kind == "fused")


def work(case):
    if case["kind"] == "qkv":
        tokens, d = case["B"] * case["N"], case["d_model"]
        cols = case["H"] * (2 * case["dk"] + case["dv"])
        return {"bytes": 2 * (tokens * d + d * cols + tokens * cols), "flops": 2 * tokens * d * cols}
    elt = 4 if case["dtype"] == "fp32" else 2
    bh, Nq, Nk, dk, dv = case["B"] * case["H"], case["Nq"], case["Nk"], case["dk"], case["dv"]
    once = elt * bh * (Nq * dk + Nk * dk + Nk * dv + Nq * dv)  # q, k, v, o
    if case["kind"] in ("bwd", "fused"):
        # reads q, k, v, o, do, lse; writes dq, dk, dv; scores, dP, dV, dQ and dK products
        return {"bytes": 2 * once + 4 * bh * Nq, "flops": 2 * bh * Nq * Nk * (3 * dk + 2 * dv)}
    if case["kind"] == "lse":
        once += 4 * bh * Nq
    return {"bytes": once, "flops": 2 * bh * Nq * Nk * (dk + dv)}


def exact(case, seed):
    t = _inputs(case, seed)
    if case["kind"] == "qkv":
        if work(case)["flops"] > 2e13:
            return None
        x, w = t["x"].double(), t["w"].double()
        B, N, H, dk, dv = (case[n] for n in ("B", "N", "H", "dk", "dv"))
        out, c0 = [], 0
        for d in (dk, dk, dv):
            y = x.reshape(B * N, -1) @ w[:, c0:c0 + H * d]
            out.append(y.reshape(B, N, H, d).permute(0, 2, 1, 3).contiguous())
            c0 += H * d
        return tuple(out)
    B, H, Nq, Nk, dk, dv = (case[n] for n in ("B", "H", "Nq", "Nk", "dk", "dv"))
    if work(case)["flops"] > 1e13:
        return None
    scale = 1.0 / math.sqrt(dk)
    bwd = case["kind"] in ("bwd", "fused")
    dev = {"dtype": torch.float64, "device": "cuda"}
    q, k, v = (t[n].flatten(0, 1) for n in ("q", "k", "v"))
    if bwd:
        do = t["do"].flatten(0, 1)
        dq, gk, gv = torch.empty(q.shape, **dev), torch.zeros(k.shape, **dev), torch.zeros(v.shape, **dev)
    else:
        o, lse = torch.empty((B * H, Nq, dv), **dev), torch.empty((B * H, Nq), **dev)
    # heads together while their score blocks stay below about 1 GB, rows of one head otherwise
    rows = max(1, min(Nq, (1 << 27) // Nk))
    heads = max(1, min(B * H, (1 << 27) // (rows * Nk)))
    for h in range(0, B * H, heads):
        hs = slice(h, h + heads)
        k64, v64 = k[hs].double(), v[hs].double()
        for r in range(0, Nq, rows):
            rs = slice(r, r + rows)
            q64 = q[hs, rs].double()
            s = (q64 * scale) @ k64.transpose(1, 2)
            m = s.amax(dim=2, keepdim=True)
            w = s.sub_(m).exp_()
            z = w.sum(dim=2, keepdim=True)
            if not bwd:
                o[hs, rs] = (w @ v64) / z
                lse[hs, rs] = (m + z.log()).squeeze(2)
                continue
            w.div_(z)
            g64 = do[hs, rs].double()
            gv[hs] += w.transpose(1, 2) @ g64
            dp = g64 @ v64.transpose(1, 2)
            d = (w * dp).sum(dim=2, keepdim=True)
            ds = dp.sub_(d).mul_(w)
            dq[hs, rs] = (ds @ k64) * scale
            gk[hs] += (ds.transpose(1, 2) @ q64) * scale
    if bwd:
        return tuple(x.reshape(B, H, *x.shape[1:]) for x in (dq, gk, gv))
    o, lse = o.reshape(B, H, Nq, dv), lse.reshape(B, H, Nq)
    return (o, lse) if case["kind"] == "lse" else o
