"""GPU test of the prefill GEMM's schedule: launches in which a pair of SMs takes several
units, units cut along K whose shares span two units, both in one launch, and more M-tiles
than one group walks, in every epilogue, against 64-bit results of the whole call.
"""
import dataclasses

import pytest
import torch

import paper_2606_09514_gb300 as pkg
from workloads import configs as C
from workloads import synth

pytestmark = pytest.mark.gpu

# K = 4096 in all four projections; 24, 16, 32 and 16 weight tiles
SHAPE = dataclasses.replace(C.LLAMA3_8B, name="units", n_layers=3, ffn_dim=4096)
LENGTHS = [[290, 10], [450, 239], [1000], [1300, 1061]]


def launches(tokens):
    """(projection, hi + lo, units computed whole, units cut, granularity of the cuts, M-tiles) by the rule of
    launch_gemm_pf, of the blocks of a prompt batch."""
    s = SHAPE
    P = torch.cuda.get_device_properties(0).multi_processor_count // 2
    mt = -(-tokens // 256)
    kb = s.d_model // 64
    tiles = {"qkv": -(-s.qkv_dim // 256), "o": s.d_model // 256, "gate_up": s.ffn_dim // 128, "down": s.d_model // 256}
    for name, t in tiles.items():
        for split in (True, False):
            units = t * mt
            R = units % P
            cut = R if R > 0 and (P - R) * kb * (52 if split else 26) > 800 * P else 0
            yield name, split, units - cut, cut, max(4, 4 if P <= 4 * R else (kb + 3) // 4), mt, P


def test_schedules_are_reached():
    every = [x for n in LENGTHS for x in launches(sum(n))]
    # every epilogue, with and without hi + lo, cut where shares span two units (R / P of a unit's K blocks each)
    assert {(n, sp) for n, sp, _, cut, gran, _, P in every if cut and gran == 4 and P % cut} == {
        (n, sp) for n in ("qkv", "o", "gate_up", "down") for sp in (True, False)}
    # whole and cut units in one launch; several whole units per pair; two groups of M-tiles, the second short
    for n in ("qkv", "o", "gate_up", "down"):
        assert any(x[0] == n and x[2] >= x[6] and x[3] for x in every)
        assert any(x[0] == n and x[2] >= 2 * x[6] and x[5] > 8 and x[5] % 8 for x in every)


def rms(h, g, eps):
    return h * torch.rsqrt(h.square().mean(1, keepdim=True) + eps) * g.double()


def rope(t, pos, theta):
    half = t.shape[-1] // 2
    f = theta ** (-torch.arange(half, dtype=torch.float64, device="cuda") / half)
    a = pos.double()[:, None, None] * f
    u, v = t[..., :half], t[..., half:]
    return torch.cat([u * a.cos() - v * a.sin(), v * a.cos() + u * a.sin()], -1)


def block64(w, h, lengths):
    """One block on prompts that start empty caches: new hidden states, K, V."""
    s = SHAPE
    pos = torch.cat([torch.arange(n, device="cuda") for n in lengths])
    q, k, v = (rms(h, w["attn_norm"], s.rms_eps) @ w["w_qkv"].double().T).split([s.q_dim, s.kv_dim, s.kv_dim], 1)
    q = rope(q.view(-1, s.n_q_heads, s.head_dim), pos, s.rope_theta)
    k, v = rope(k.view(-1, s.n_kv_heads, s.head_dim), pos, s.rope_theta), v.view(-1, s.n_kv_heads, s.head_dim)
    o, at = [], 0
    for n in lengths:
        kk, vv = (t[at:at + n].transpose(0, 1).repeat_interleave(s.group, 0) for t in (k, v))
        z = q[at:at + n].transpose(0, 1) @ kk.transpose(1, 2) / s.head_dim ** 0.5
        z = z.masked_fill(torch.ones(n, n, dtype=torch.bool, device="cuda").triu(1), float("-inf"))
        o.append((z.softmax(-1) @ vv).transpose(0, 1).reshape(n, -1))
        at += n
    h = h + torch.cat(o) @ w["w_o"].double().T
    g, u = (rms(h, w["ffn_norm"], s.rms_eps) @ w["w_gate_up"].double().T).chunk(2, 1)
    return h + (torch.nn.functional.silu(g) * u) @ w["w_down"].double().T, k, v


@pytest.mark.parametrize("lengths", LENGTHS, ids=lambda v: str(sum(v)))
def test_prefill_units(lengths):
    s, B, T = SHAPE, len(lengths), sum(lengths)
    ws = []
    for l in range(s.n_layers):
        w = pkg.pack_layer(synth.layer_weights(s, 11, l, "cuda"))
        w["w_o"] *= 4   # the averaged values of long contexts are small: as large an update as the FFN's
        ws.append(w)
    ctx = pkg.Context.for_shape(s, max_batch=B, max_pos=max(lengths), max_prefill_tokens=T)
    ctx.buddy_set_weights(ws, synth.dm_weights(s, 11, "cuda"))
    kv = pkg.KVCache(s.n_layers, s.n_kv_heads, s.head_dim, lengths, torch.bfloat16, "cuda")
    x = synth.prompt_inputs(s, 11, lengths, "cuda")
    k = torch.ones(B, dtype=torch.int32, device="cuda")   # all three blocks run
    outs = []
    for _ in range(2):
        kv.len.zero_()
        h = torch.empty(T, s.d_model, device="cuda")
        ctx.buddy_prefill(kv, lengths, x, k, h)
        assert ctx.buddy_device_status() == 0
        outs.append([h] + [t.clone() for t in kv.k + kv.v])
    assert all(torch.equal(a, b) for a, b in zip(*outs))

    def close(got, ref):   # per row: bf16 operands between the projections, as parity.py
        err = (got.double() - ref).abs().amax(-1) / ref.abs().amax(-1)
        assert float(err.max()) < 2e-2, float(err.max())
    h = x.double()
    for l, w in enumerate(ws):
        h, kk, vv = block64(w, h, lengths)
        at = 0
        for i, n in enumerate(lengths):
            close(kv.view("k", l, i)[:, :n].transpose(0, 1).reshape(n, -1), kk[at:at + n].reshape(n, -1))
            close(kv.view("v", l, i)[:, :n].transpose(0, 1).reshape(n, -1), vv[at:at + n].reshape(n, -1))
            at += n
    close(outs[0][0], h)


# decode GEMMs and their fixups up to 256 tokens (gate/up in one K split where its tiles fill most SMs, then
# without a fixup), one launch per projection above
@pytest.mark.parametrize("shape,tokens,per_block", [(C.SMALL_QWEN_BF16, 20, 8), (C.LLAMA3_8B, 16, 7), (C.SMALL_QWEN_BF16, 257, 4)],
                         ids=lambda v: getattr(v, "name", str(v)))
def test_profiler_counts_prefill_launches(shape, tokens, per_block):
    s = dataclasses.replace(shape, n_layers=3)
    w = pkg.pack_layer(synth.layer_weights(s, 1, 0, "cuda"))
    ctx = pkg.Context.for_shape(s, max_batch=1, max_pos=tokens, max_prefill_tokens=tokens)
    ctx.buddy_set_weights([w] * 3, synth.dm_weights(s, 1, "cuda"))
    kv = pkg.KVCache(3, s.n_kv_heads, s.head_dim, [tokens], torch.bfloat16, "cuda")
    x = synth.prompt_inputs(s, 1, [tokens], "cuda")
    ctx.buddy_set_profiling(True)
    ctx.buddy_prefill(kv, [tokens], x, torch.ones(1, dtype=torch.int32, device="cuda"), torch.empty_like(x))
    prof = ctx.buddy_profile_read()
    assert {k: prof[k][1] for k in ("pf_gemm", "pf_attention", "route")} == {
        "pf_gemm": 3 * per_block, "pf_attention": 3, "route": 4}
