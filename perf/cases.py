"""Measured cases of the budget-routed decode library: what a serving program
calls, through the package's public entry points.

A case is a dict of plain values:
  op       "decode" (buddy_decode_step), "decode_host" (buddy_decode_step_host),
           "prefill" (buddy_prefill), "append" (buddy_kv_append on every layer)
           or "route" (buddy_route)
  shape    per-layer sizes of a model family (SHAPES)
  layers   decoder layers of the model
  batch    sequences
  lo, hi   cached positions per sequence before the call, evenly spread over
           [lo, hi] (which sequence has which is drawn)
  tok_lo, tok_hi   prefill / append: new tokens per sequence, spread likewise
           (append: tok_lo for every sequence, as the call takes one count)
  k_lo, k_hi   budgets, evenly spread over [k_lo, k_hi]; 0: the Budget
           Predictor chooses
  graph    decode steps replayed as a CUDA graph
  prior, feature, ctx_layer, skip, predictor   router options
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2606_09514_gb300 as pkg

# d_model, query heads, KV heads, head dim, FFN width, DM hidden, dtype, eps, theta, qkv bias
SHAPES = {
    "llama3-8b": (4096, 32, 8, 128, 14336, 256, "bf16", 1e-5, 5e5, False),
    "llama2-13b": (5120, 40, 40, 128, 13824, 256, "bf16", 1e-5, 1e4, False),
    "qwen2.5-7b": (3584, 28, 4, 128, 18944, 256, "bf16", 1e-6, 1e6, True),
    "small-gqa": (576, 9, 3, 64, 1472, 64, "bf16", 1e-5, 1e4, False),
    "tiny-f32": (256, 4, 4, 64, 688, 128, "f32", 1e-5, 1e4, False),
}
REWIND = 32   # decode passes on one state before the program starts its next request
OMEGA = 0.1   # weight of the prior where a case has one


def _case(name, op, shape, layers, batch, lo=0, hi=None, tok_lo=0, tok_hi=None, k_lo=1, k_hi=None, graph=True,
          prior=False, feature="v", ctx_layer=0, skip="zero", predictor=0):
    c = {"op": op, "shape": shape, "layers": layers, "batch": batch, "lo": lo, "hi": lo if hi is None else hi,
         "tok_lo": tok_lo, "tok_hi": tok_lo if tok_hi is None else tok_hi, "k_lo": k_lo,
         "k_hi": k_lo if k_hi is None else k_hi, "graph": graph, "prior": prior, "feature": feature,
         "ctx_layer": ctx_layer, "skip": skip, "predictor": predictor}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the router by itself for a few requests: the smallest call a program makes
        _case("route-b3", "route", "llama3-8b", 32, 3, 100, 3000, k_lo=8, k_hi=30),
        # re-routing a full server batch
        _case("route-b250", "route", "qwen2.5-7b", 28, 250, 512, 8000, k_lo=6, k_hi=26),
        # a small fp32 model, as in unit-scale experiments: latency and launches only
        _case("decode-tiny-f32-b4", "decode", "tiny-f32", 8, 4, 128, k_lo=3),
        # one user's generation on a whole 8B model at the 50% budget (the headline)
        _case("decode-llama3-b1", "decode", "llama3-8b", 32, 1, 2048, k_lo=15),
        # a few interactive requests with host buffers, masked skips, a later context layer,
        # the K + V feature and predicted budgets; launched directly
        _case("decode-host-llama3-b7", "decode_host", "llama3-8b", 6, 7, 37, 1900, k_lo=0, k_hi=3, graph=False,
              feature="kv", ctx_layer=1, skip="masked", predictor=128),
        # an ordinary mixed serving batch with a prior
        _case("decode-llama3-b64", "decode", "llama3-8b", 6, 64, 512, 4096, k_lo=1, k_hi=4, prior=True),
        # multi-head attention (no KV sharing) at a long context: KV bandwidth
        _case("decode-llama2-13b-b32", "decode", "llama2-13b", 4, 32, 4096, k_lo=1),
        # the largest decode batch, ragged contexts
        _case("decode-qwen-b256", "decode", "qwen2.5-7b", 5, 256, 512, 4300, k_lo=1, k_hi=3),
        # loading the cache of a few saved prompts behind a shared prefix
        _case("append-llama3-6x1000", "append", "llama3-8b", 3, 6, 100, tok_lo=1000),
        # time to first token of one short prompt
        _case("prefill-llama3-1x61", "prefill", "llama3-8b", 4, 1, 0, tok_lo=61),
        # an ordinary admission batch of ragged prompts, two budgets
        _case("prefill-llama3-5x128-1024", "prefill", "llama3-8b", 4, 5, 0, tok_lo=128, tok_hi=1023, k_lo=1, k_hi=2),
        # long documents, one behind a cached prefix
        _case("prefill-qwen-2x3000-5000", "prefill", "qwen2.5-7b", 3, 2, 0, 512, tok_lo=2999, tok_hi=5000),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["route", "append", "decode", "decode", "decode", "decode_host", "prefill", "prefill"])
    shape = rng.choice(["llama3-8b", "llama3-8b", "llama2-13b", "qwen2.5-7b", "small-gqa", "tiny-f32"])
    if op == "prefill" and shape == "tiny-f32":   # prefill is a bf16 entry
        shape = "small-gqa"
    nkv, hd = SHAPES[shape][2], SHAPES[shape][3]
    layers = rng.randint(3, 5)
    if op == "route":
        lo = _log(rng, 1, 4000)
        k = rng.randint(1, layers + 20)
        return _case(None, op, shape, layers + 22, _log(rng, 1, 256), lo, lo + _log(rng, 1, 4000), k_lo=1, k_hi=k)
    if op == "append":
        n = _log(rng, 1, 4000)
        most = max(1, min(32, 16000 // n))
        return _case(None, op, shape, 3, rng.randint(1, most), _log(rng, 1, 500), tok_lo=n)
    if op == "prefill":
        layers = 3
        total = _log(rng, 9, 7000)
        B = rng.randint(1, max(1, min(8, total // 9)))
        tok = max(1, total // B)
        return _case(None, op, shape, layers, B, 0, rng.choice([0, 0, 300]), tok_lo=max(1, tok // 2), tok_hi=tok,
                     skip=rng.choice(["zero", "zero", "masked"]))
    B = _log(rng, 1, 256)
    # the caches of one state stay within those of the largest listed case
    ctx = _log(rng, 64, max(65, min(8000, int(1.2e9 // (B * nkv * hd * 4)))))
    n_cand = layers - 2
    return _case(None, op, shape, layers, B, max(1, ctx // 4), ctx, k_lo=1, k_hi=n_cand, graph=rng.random() < 0.7,
                 prior=rng.random() < 0.3, feature=rng.choice(["v", "v", "k"]),
                 skip=rng.choice(["zero", "zero", "zero", "masked"]))


# --------------------------------------------------------------------------
# Inputs: everything from the seed, as plain tensors
# --------------------------------------------------------------------------
class _Spec:
    def __init__(self, case):
        (self.d, self.nq, self.nkv, self.hd, self.F, self.r, dt, self.eps, self.theta, self.bias) = SHAPES[case["shape"]]
        self.bf16 = dt == "bf16"
        self.dtype = torch.bfloat16 if self.bf16 else torch.float32
        self.esz = 2 if self.bf16 else 4
        self.L, self.B, self.c = case["layers"], case["batch"], case["ctx_layer"]
        self.n_cand = self.L - 2 - self.c
        self.kvd, self.qd = self.nkv * self.hd, self.nq * self.hd
        self.op = case["op"]
        self.masked = case["skip"] == "masked"
        spread = lambda a, b, n: np.rint(np.linspace(a, b, n)).astype(np.int64) if n > 1 else np.array([b], np.int64)
        self.lens = spread(case["lo"], case["hi"], self.B)   # before the shuffle
        self.toks = spread(case["tok_lo"], case["tok_hi"], self.B)
        self.ks = np.clip(spread(case["k_lo"], case["k_hi"], self.B), 0 if case["predictor"] else 1, self.n_cand)
        self.layer_params = self.d * (self.qd + 2 * self.kvd) + self.qd * self.d + 3 * self.F * self.d


def _inputs(case, seed):
    s = _Spec(case)
    perm = np.random.default_rng([int(seed), 7])
    g = torch.Generator(device="cuda").manual_seed(int(seed) * 1009 + 17)
    N = lambda shape, sd, dt=torch.float32: torch.empty(shape, dtype=dt, device="cuda").normal_(0.0, sd, generator=g)
    x = {"s": s, "lens": s.lens[perm.permutation(s.B)], "toks": s.toks[perm.permutation(s.B)],
         "ks": s.ks[perm.permutation(s.B)]}
    x["dm"] = {"w1": N((s.r, 2 * s.d), 0.02), "b1": N((s.r,), 0.02), "w2": N((s.n_cand, s.r), 0.02),
               "b2": N((s.n_cand,), 0.02)}
    x["prior"] = N((s.n_cand,), 1.0) if case["prior"] else None
    p = case["predictor"]
    x["pred"] = ({"w1": N((p, 2 * s.d), 0.02), "b1": N((p,), 0.02), "w2": N((s.n_cand, p), 0.5),
                  "b2": N((s.n_cand,), 0.5)} if p else None)
    x["h"] = N((s.B if s.op != "prefill" else int(x["toks"].sum()), s.d), 1.0)
    x["layers"] = []
    if s.op == "route":
        x["pool"] = N((s.B, s.kvd), 1.0) * torch.tensor(x["lens"], device="cuda").float().sqrt()[:, None]
        return x
    if s.op != "append":   # the append call reads no layer weights
        for _ in range(s.L):
            w = {"w_qkv": N((s.qd + 2 * s.kvd, s.d), 0.02, s.dtype), "w_o": N((s.d, s.qd), 0.02, s.dtype),
                 "w_gate_up": N((2 * s.F, s.d), 0.02, s.dtype), "w_down": N((s.d, s.F), 0.02, s.dtype),
                 "attn_norm": 1.0 + N((s.d,), 0.1), "ffn_norm": 1.0 + N((s.d,), 0.1)}
            if s.bias:
                w["b_qkv"] = N((s.qd + 2 * s.kvd,), 0.02)
            x["layers"].append(w)
    grow = x["toks"] if s.op in ("prefill", "append") else np.full(s.B, REWIND, np.int64)
    x["caps"] = x["lens"] + grow
    n = int(x["caps"].sum()) * s.kvd
    x["kc"] = [N((n,), 1.0, s.dtype) for _ in range(s.L)]
    x["vc"] = [N((n,), 1.0, s.dtype) for _ in range(s.L)]
    if s.masked:   # positions each layer holds: some earlier tokens skipped it
        ll = np.array([[int(v) if l <= s.c or l == s.L - 1 else int(v) * (1 + (i + l) % 3) // 3
                        for i, v in enumerate(x["lens"])] for l in range(s.L)], np.int32)
    else:
        ll = np.tile(x["lens"].astype(np.int32), (s.L, 1))
    x["layer_len"] = ll
    if s.op == "append":
        n = int(s.toks[0])
        x["new"] = [(N((s.B, n, s.nkv, s.hd), 1.0, s.dtype), N((s.B, n, s.nkv, s.hd), 1.0, s.dtype))
                    for _ in range(s.L)]
    return x


def _rows(x, buf, i):
    """Sequence i's block of a cache buffer: [n_kv, cap_i, hd]."""
    s = x["s"]
    a = int(x["caps"][:i].sum()) * s.kvd
    return buf[a:a + int(x["caps"][i]) * s.kvd].view(s.nkv, int(x["caps"][i]), s.hd)


def _feature(case, k, v):
    return {"v": lambda: v, "k": lambda: k, "kv": lambda: k + v}[case["feature"]]()


# --------------------------------------------------------------------------
# One pass through the library
# --------------------------------------------------------------------------
def prepare(case, seed):
    x = _inputs(case, seed)
    s = x["s"]
    T = int(x["toks"].sum())
    max_pos = int(x["caps"].max()) if "caps" in x else int(x["lens"].max())
    ctx = pkg.Context(n_layers=s.L, d_model=s.d, n_q_heads=s.nq, n_kv_heads=s.nkv, head_dim=s.hd, ffn_dim=s.F,
                      dm_hidden=s.r, dtype="bf16" if s.bf16 else "f32", max_batch=s.B, max_pos=max_pos,
                      qkv_bias=s.bias, rms_eps=s.eps, rope_theta=s.theta, feature=case["feature"],
                      ctx_layer=s.c, skip_kv=case["skip"], max_prefill_tokens=T if s.op == "prefill" else 0)
    if s.op in ("route", "append"):   # a router-only or cache-only process: one layer's storage stands for all
        one = {"w_qkv": (s.qd + 2 * s.kvd, s.d), "w_o": (s.d, s.qd), "w_gate_up": (2 * s.F, s.d),
               "w_down": (s.d, s.F)}
        w = {k: torch.zeros(v, dtype=s.dtype, device="cuda") for k, v in one.items()}
        w["attn_norm"] = w["ffn_norm"] = torch.ones(s.d, device="cuda")
        if s.bias:
            w["b_qkv"] = torch.zeros(s.qd + 2 * s.kvd, device="cuda")
        layers = [w] * s.L
    else:
        layers = x["layers"]
    ctx.buddy_set_weights(layers, x["dm"], prior=x["prior"], omega=OMEGA if case["prior"] else 0.0)
    if x["pred"]:
        ctx.buddy_set_budget_predictor(x["pred"])
    ctx.buddy_set_options(case["graph"])
    if s.op == "route":   # the router reads lengths and pooled sums only
        kv = pkg.KVCache(s.L, s.nkv, s.hd, [1] * s.B, s.dtype, "cuda")
        kv.cap.copy_(torch.tensor(x["lens"], dtype=torch.int32))
        kv.len.copy_(torch.tensor(x["lens"], dtype=torch.int32))
        kv.pool_sum.copy_(x["pool"])
    else:
        kv = pkg.KVCache(s.L, s.nkv, s.hd, x["caps"].tolist(), s.dtype, "cuda", masked=s.masked)
        for l in range(s.L):
            kv.k[l].copy_(x["kc"][l])
            kv.v[l].copy_(x["vc"][l])
            x["kc"][l] = x["vc"][l] = None
        kv.len.copy_(torch.tensor(x["lens"], dtype=torch.int32))
        if s.masked:
            kv.layer_len.copy_(torch.tensor(x["layer_len"]))
        for i in range(s.B):
            n = int(x["layer_len"][s.c, i])
            kv.pool_sum[i] = _feature(case, kv.view("k", s.c, i)[:, :n].float(),
                                      kv.view("v", s.c, i)[:, :n].float()).sum(1).reshape(-1)
    st = {"case": case, "s": s, "ctx": ctx, "kv": kv, "n": 0, "toks": [int(t) for t in x["toks"]],
          "k": torch.tensor(x["ks"], dtype=torch.int32, device="cuda"), "h": x["h"], "new": x.get("new"),
          "ids": torch.arange(s.B, dtype=torch.int32, device="cuda"),
          "len0": kv.len.clone(), "pool0": kv.pool_sum.clone(),
          "ll0": kv.layer_len.clone() if s.masked and s.op != "route" else None,
          "mask": torch.zeros(s.B, s.L, dtype=torch.uint8, device="cuda"),
          "count": torch.zeros(s.L, dtype=torch.int32, device="cuda"),
          "scores": torch.zeros(s.B, s.n_cand, device="cuda"),
          "sel": torch.zeros(s.B, s.n_cand, dtype=torch.int32, device="cuda"),
          "out": torch.zeros_like(x["h"])}
    if s.op == "decode_host":
        st["h"], st["k"], st["out"] = st["h"].cpu().pin_memory(), st["k"].cpu().pin_memory(), st["out"].cpu().pin_memory()
        st["mask"] = st["mask"].cpu().pin_memory()
    return st


def _rewind(st):
    """The program's next request on the same slots: positions and pooled sums as before the generation."""
    st["kv"].len.copy_(st["len0"])
    if st["s"].op not in ("append", "prefill"):   # those recompute the pooled sums themselves
        st["kv"].pool_sum.copy_(st["pool0"])
    if st["ll0"] is not None:
        st["kv"].layer_len.copy_(st["ll0"])


def run(st):
    s, ctx, kv = st["s"], st["ctx"], st["kv"]
    if s.op == "route":
        ctx.buddy_route(kv, st["h"], st["k"], st["sel"], st["mask"], st["scores"])
        return {"sel": st["sel"], "mask": st["mask"], "scores": st["scores"]}
    if s.op == "append":
        if st["n"]:
            _rewind(st)
        for l in range(s.L):
            ctx.buddy_kv_append(kv, l, st["ids"], st["new"][l][0], st["new"][l][1], advance=l == s.L - 1)
    elif s.op == "prefill":
        if st["n"]:
            _rewind(st)
        ctx.buddy_prefill(kv, st["toks"], st["h"], st["k"], st["out"], st["mask"], st["scores"])
    else:
        if st["n"] == REWIND:
            _rewind(st)
            st["n"] = 0
        if s.op == "decode_host":
            ctx.buddy_decode_step_host(kv, st["h"], st["k"], st["out"], st["mask"])
        else:
            ctx.buddy_decode_step(kv, st["h"], st["k"], st["out"], st["mask"], None, st["count"], st["scores"])
    st["n"] += 1
    out = {"len": kv.len, "pool": kv.pool_sum}
    if s.op != "append":
        out.update(h=st["out"], mask=st["mask"])
    if s.op in ("prefill", "decode"):
        out["scores"] = st["scores"]
    if s.op == "decode":
        out["count"] = st["count"]
    if kv.layer_len is not None:
        out["layer_len"] = kv.layer_len
    ls = range(s.L) if s.L <= 8 else (0, s.L - 1)   # at most 64 outputs: the always-executed layers of a deep model
    out["k_cache"], out["v_cache"] = [kv.k[l] for l in ls], [kv.v[l] for l in ls]
    return out


# --------------------------------------------------------------------------
# What a pass cannot do without
# --------------------------------------------------------------------------
def work(case):
    s = _Spec(case)
    dm = 4 * (s.r + case["predictor"]) * (2 * s.d + s.n_cand)
    rows = s.B * (4 * s.kvd + 4 * s.d)
    route_flops = 2 * s.B * (s.r + case["predictor"]) * (2 * s.d + s.n_cand)
    if s.op == "route":
        return {"bytes": dm + rows + s.B * (s.L + 8 * s.n_cand), "flops": route_flops}
    if s.op == "append":
        T = int(s.toks.sum())
        # new entries read and written in every layer; the context layer's prefix read once for its pooled sum
        return {"bytes": s.L * T * s.kvd * s.esz * 4 + int(s.lens.sum()) * s.kvd * s.esz + 4 * s.B * s.kvd,
                "flops": int(s.lens.sum() + T) * s.kvd}
    ks = np.where(s.ks == 0, (s.n_cand + 1) / 2, s.ks)        # a predicted budget: the middle of its range
    always = s.c + 2
    touched = always + min(s.n_cand, int(math.ceil(ks.sum())))   # layers whose weights some sequence needs
    pairs = float(ks.sum() + always * s.B)                       # executed (sequence, layer) pairs
    skipped = s.L * s.B - pairs
    depth = 2.0 / 3.0 if s.masked else 1.0                       # a masked layer holds about that share of the positions
    if s.op == "prefill":
        T = float(s.toks.sum())
        share = pairs / s.B
        att = sum(4.0 * s.qd * (t * n + t * (t + 1) / 2) for t, n in zip(s.toks, s.lens))
        b = (touched * s.layer_params * s.esz + share * T * 2 * s.kvd * s.esz + 2 * T * s.d * 4 + dm
             + share * float(s.lens.sum()) * 2 * s.kvd * s.esz
             + (0 if s.masked else (s.L - share) * T * 2 * s.kvd * s.esz))
        return {"bytes": b, "flops": share * (2 * s.layer_params * T + att) + route_flops}
    mean_len = float(s.lens.mean())
    kv = (s.B * always + float(ks.sum()) * depth) * (mean_len + 1) * 2 * s.kvd * s.esz
    b = touched * s.layer_params * s.esz + kv + dm + 2 * s.B * s.d * 4
    if not s.masked:
        b += skipped * 2 * s.kvd * s.esz
    return {"bytes": b, "flops": pairs * (2 * s.layer_params + 4 * s.qd * (mean_len + 1) * depth) + route_flops}


def tolerance(case):
    s = _Spec(case)
    if s.op in ("route", "append") or not s.bf16:
        return {"rel": 2e-6}       # fp32 sums: 2e-8 to 2e-7 from their 64-bit values
    # bf16 operands between the GEMMs of each block, fp32 sums: the hidden states lie 3e-3 to 4e-3
    # (3 to 6 layers) and 9e-3 (32 layers) from their 64-bit values
    return {"rel": 1.2e-2 if s.L <= 8 else 2.5e-2, "max": 0.2}


# --------------------------------------------------------------------------
# The same pass in 64 bits, in plain torch.  New K and V are not rounded to the
# cache's type, so that an output's distance holds that rounding whole instead
# of the few values that round the other way.
# --------------------------------------------------------------------------
def _rms(h, g, eps):
    return h * torch.rsqrt(h.square().mean(-1, keepdim=True) + eps) * g.double()


def _rope(s, t, pos):
    """t [n, heads, hd] at positions pos [n], rotate-half."""
    half = s.hd // 2
    th = torch.tensor(float(s.theta), dtype=torch.float64, device="cuda") ** (
        -2.0 * torch.arange(half, dtype=torch.float64, device="cuda") / s.hd)
    a = pos.double()[:, None] * th[None]
    co, si = a.cos()[:, None], a.sin()[:, None]
    u, v = t[..., :half], t[..., half:]
    return torch.cat([u * co - v * si, v * co + u * si], -1)


def _attend(s, q, K, V, first):
    """q [t, nq, hd], the tokens at cache positions first ..; K, V [nkv, n, hd]; causal."""
    G, n = s.nq // s.nkv, K.shape[1]
    out = torch.empty_like(q)
    for a in range(0, q.shape[0], 512):
        qa = q[a:a + 512]
        t = qa.shape[0]
        last = min(n, first + a + t)
        qg = qa.reshape(t, s.nkv, G, s.hd).permute(1, 2, 0, 3).reshape(s.nkv, G * t, s.hd)
        z = (qg @ K[:, :last].double().transpose(1, 2)) / math.sqrt(s.hd)
        z = z.view(s.nkv, G, t, last)
        vis = torch.arange(last, device="cuda")[None] <= first + a + torch.arange(t, device="cuda")[:, None]
        z = z.masked_fill(~vis, -math.inf).softmax(-1).view(s.nkv, G * t, last)
        o = (z @ V[:, :last].double()).view(s.nkv, G, t, s.hd)
        out[a:a + t] = o.permute(2, 0, 1, 3).reshape(t, s.nq, s.hd)
    return out


def _block(x, l, H, seqs, off, toks):
    """Runs layer l on the tokens of `seqs` (rows off[i] .. of H), storing their K/V."""
    s, w = x["s"], x["layers"][l]
    rows = torch.cat([torch.arange(off[i], off[i] + toks[i], device="cuda") for i in seqs])
    pos = torch.cat([int(x["lens"][i]) + torch.arange(toks[i], device="cuda") for i in seqs])
    h = H[rows]
    qkv = _rms(h, w["attn_norm"], s.eps) @ w["w_qkv"].double().T
    if s.bias:
        qkv = qkv + w["b_qkv"].double()
    q, k, v = qkv.split([s.qd, s.kvd, s.kvd], -1)
    q = _rope(s, q.reshape(-1, s.nq, s.hd), pos)
    k = _rope(s, k.reshape(-1, s.nkv, s.hd), pos)
    v = v.reshape(-1, s.nkv, s.hd)
    o = torch.empty_like(q)
    a = 0
    for i in seqs:
        t, n = toks[i], int(x["layer_len"][l, i])
        K, V = _rows(x, x["kc"][l], i), _rows(x, x["vc"][l], i)
        K[:, n:n + t] = k[a:a + t].transpose(0, 1).to(K.dtype)
        V[:, n:n + t] = v[a:a + t].transpose(0, 1).to(V.dtype)
        o[a:a + t] = _attend(s, q[a:a + t], K[:, :n + t], V[:, :n + t], n)
        a += t
    h = h + o.reshape(-1, s.qd) @ w["w_o"].double().T
    y = _rms(h, w["ffn_norm"], s.eps)
    gu = w["w_gate_up"]
    act = torch.nn.functional.silu(y @ gu[:s.F].double().T) * (y @ gu[s.F:].double().T)
    H[rows] = h + act @ w["w_down"].double().T


def _mlp(w, x):
    w = {k: v.double() for k, v in w.items()}
    return torch.nn.functional.silu(x @ w["w1"].T + w["b1"]) @ w["w2"].T + w["b2"]


def _router(case, x, pool, n, h):
    """Scores [B, n_cand], the chosen layers per sequence."""
    s = x["s"]
    p = (pool.double() / n[:, None]).view(s.B, s.nkv, 1, s.hd).expand(-1, -1, s.nq // s.nkv, -1).reshape(s.B, s.qd)
    f = torch.cat([p, h.double()], -1)
    sc = _mlp(x["dm"], f)
    if x["prior"] is not None:
        sc = sc + float(np.float32(OMEGA)) * x["prior"].double()
    ks = [int(k) for k in x["ks"]]
    if x["pred"]:
        best = _mlp(x["pred"], f).argmax(-1)
        ks = [k or int(best[i]) + 1 for i, k in enumerate(ks)]
    order = torch.sort(sc, dim=-1, descending=True, stable=True).indices.tolist()
    return sc, [sorted(s.c + 1 + j for j in order[i][:ks[i]]) for i in range(s.B)]


def exact(case, seed):
    w = work(case)
    if w["flops"] > 1.5e13:
        return None
    x = _inputs(case, seed)
    s = x["s"]
    lens = torch.tensor(x["lens"], device="cuda")
    if s.op == "route":
        sc, sel = _router(case, x, x["pool"], lens.double(), x["h"])
        return {"sel": _sel(s, sel), "mask": _mask(s, sel), "scores": sc}
    wide = torch.float32 if s.bf16 else torch.float64
    for which in ("kc", "vc"):
        for l in range(s.L):
            x[which][l] = x[which][l].to(wide)
    toks = [int(t) for t in x["toks"]] if s.op in ("prefill", "append") else [1] * s.B
    if s.op == "append":
        for l in range(s.L):
            for i in range(s.B):
                n = int(x["lens"][i])
                _rows(x, x["kc"][l], i)[:, n:n + toks[i]] = x["new"][l][0][i].transpose(0, 1)
                _rows(x, x["vc"][l], i)[:, n:n + toks[i]] = x["new"][l][1][i].transpose(0, 1)
        sel = None
        out = {}
    else:
        off = np.concatenate([[0], np.cumsum(toks)[:-1]]).tolist()
        H = x["h"].double()
        every = list(range(s.B))
        for l in range(s.c + 1):
            _block(x, l, H, every, off, toks)
    new_len = lens + torch.tensor(toks, device="cuda")
    pool = torch.empty(s.B, s.kvd, dtype=torch.float64, device="cuda")
    for i in range(s.B):
        n = int(x["layer_len"][s.c, i]) + toks[i]
        pool[i] = _feature(case, _rows(x, x["kc"][s.c], i)[:, :n].double(),
                           _rows(x, x["vc"][s.c], i)[:, :n].double()).sum(1).reshape(-1)
    if s.op != "append":
        last = torch.tensor([off[i] + toks[i] - 1 for i in every], device="cuda")
        sc, sel = _router(case, x, pool, new_len.double(), H[last])
        for l in range(s.c + 1, s.L - 1):
            seqs = [i for i in every if l in sel[i]]
            if seqs:
                _block(x, l, H, seqs, off, toks)
            if not s.masked:
                for i in every:
                    if l not in sel[i]:
                        n = int(x["lens"][i])
                        _rows(x, x["kc"][l], i)[:, n:n + toks[i]] = 0
                        _rows(x, x["vc"][l], i)[:, n:n + toks[i]] = 0
        _block(x, s.L - 1, H, every, off, toks)
        m = _mask(s, sel)
        out = {"h": H, "mask": m}
        if s.op in ("prefill", "decode"):
            out["scores"] = sc
        if s.op == "decode":
            out["count"] = m.sum(0, dtype=torch.int32)
        if s.masked:
            out["layer_len"] = torch.tensor(x["layer_len"], device="cuda") + (
                m.T.int() * torch.tensor(toks, dtype=torch.int32, device="cuda")[None])
    out.update(len=new_len.int(), pool=pool)
    ls = range(s.L) if s.L <= 8 else (0, s.L - 1)
    out["k_cache"], out["v_cache"] = [x["kc"][l] for l in ls], [x["vc"][l] for l in ls]
    return out


def _mask(s, sel):
    m = torch.zeros(s.B, s.L, dtype=torch.uint8)
    m[:, :s.c + 1] = 1
    m[:, s.L - 1] = 1
    for i, ls in enumerate(sel):
        m[i, ls] = 1
    return m.cuda()


def _sel(s, sel):
    out = torch.full((s.B, s.n_cand), -1, dtype=torch.int32)
    for i, ls in enumerate(sel):
        out[i, :len(ls)] = torch.tensor(ls, dtype=torch.int32)
    return out.cuda()
