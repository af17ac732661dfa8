"""GPU tests at the sizes where a kernel's tile, split or dispatch rule changes:
prefill projections (one or two 128-row M-tiles of the decode GEMM up to 256
tokens, CTA pairs above) and its attention (tiles of 128 (token, head) rows),
small-batch decode modes and attention cluster sizes, the fp32 GEMMs, the router's
and the bulk append's own argument checks, and the wait limits of these paths.
Values are compared with the float64 oracle at the bounds of parity.py.
"""
import dataclasses

import numpy as np
import pytest
import torch

import paper_2606_09514_gb300 as pkg
import test_gpu_fullsize as FS
from paper_2606_09514_gb300 import binding as Bd
from test_gpu_decode import run_parity
from test_gpu_prefill import run_prefill_parity
from workloads import configs as C
from workloads import device as D
from workloads import synth

pytestmark = pytest.mark.gpu


def rows_of(base, batch):
    """The workload's own contexts and budgets, repeated to `batch` rows."""
    if base.ctx_kind != "list":
        return C.scaled(base, batch=batch, name=f"{base.name}-b{batch}")
    n = len(base.ctx_args)
    return C.scaled(base, ctx=[base.ctx_args[i % n] for i in range(batch)],
                    k=[base.k_args[i % n] for i in range(batch)], name=f"{base.name}-b{batch}")


# tokens in all: 1; 16 and 17 (workspace layouts); 128 and 129 (M-tiles); 256 and
# 257 (decode GEMMs and CTA pairs); 126 and 129 rows of a 3-head group (attention
# tiles); the masked variant takes the CTA pairs at any size
@pytest.mark.parametrize("base,lengths,ctx", [
    (C.T_GQA, [1], [0]), (C.T_GQA, [16], [40]), (C.T_GQA, [17], [0]), (C.T_QWEN, [128], [1]),
    (C.T_QWEN, [100, 29], [0, 127]), (C.T_QWEN, [256], [0]), (C.T_QWEN, [1, 256], [128, 3]),
    (C.T_GQA, [42, 43], [0, 86]), (C.T_VARIANTS[2], [5, 40], [0, 65])],
    ids=lambda v: v.shape.name if hasattr(v, "shape") else "-".join(map(str, v)))
def test_prefill_parity_at_tile_edges(base, lengths, ctx):
    w = C.scaled(base, ctx=ctx, k=[1 + i for i in range(len(ctx))], name="pf-edge")
    assert run_prefill_parity(w, lengths, decode_steps=1) < 2e-2


# 2 and 3 rows: panels and deferred fixup; 5, 10 and 21 rows of 3 KV heads: 15, 30
# and 63 streams, in clusters of 8, 4 and 2 CTAs
@pytest.mark.parametrize("base,batch", [(C.T_QWEN, 2), (C.T_QWEN, 3), (C.T_GQA, 2), (C.T_GQA, 5), (C.T_GQA, 10),
                                        (C.T_GQA, 21)], ids=lambda v: v.shape.name if hasattr(v, "shape") else str(v))
def test_decode_parity_small_batch_modes(base, batch):
    assert run_parity(rows_of(base, batch), steps=2)[0] < 2e-2


# 6144 positions per warp or more: a quarter of them claimed in units; short and long
# streams in turn, one row of every part of the sequence checked
def test_decode_parity_claimed_units():
    base = C.P_QWEN_3L_B256
    ctx = [7600 - 3 * i if i % 2 else 5 + 11 * i // 2 for i in range(256)]
    warps = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    assert base.shape.n_kv_heads * sum(ctx) >= 6144 * warps
    w = dataclasses.replace(C.scaled(base, ctx=ctx, k=[1] * 256, name="qwen2.5-7b-3layer-units"), steps=2)
    FS.test_fullsize_trajectory_parity(w, [0, 1, 100, 201, 254, 255])


# fp32: four or eight rows per pass (4, 5), norms and QKV finalisation inside the
# GEMMs up to 28 rows, tiles of 32 rows above (29, 32, 33)
@pytest.mark.parametrize("batch", [4, 5, 24, 25, 28, 29, 32, 33])
def test_decode_parity_f32_batch_modes(batch):
    assert run_parity(rows_of(C.T_F32, batch), steps=2)[0] < 1e-4


def route_scores64(dm, pool, length, h1, group, hd):
    x = (pool.double() / length.double()[:, None]).view(pool.shape[0], -1, 1, hd)
    x = torch.cat([x.expand(-1, -1, group, -1).reshape(pool.shape[0], -1), h1.double()], 1)
    w = {k: v.double() for k, v in dm.items()}
    return torch.nn.functional.silu(x @ w["w1"].T + w["b1"]) @ w["w2"].T + w["b2"]


@pytest.mark.parametrize("batch", [1, 16, 17, 64, 65])
def test_route_scores_at_batch_modes(batch):
    s = C.SMALL_QWEN_BF16
    w = rows_of(C.T_QWEN, batch)
    dw = D.build(w)
    h1 = synth.h_in(s, 5, 0, range(batch), "cuda")
    dw.kv.len.clamp_(min=1)
    sc = torch.empty(batch, s.n_cand, device="cuda")
    dw.ctx.buddy_route(dw.kv, h1, dw.k, scores_out=sc)
    assert dw.ctx.buddy_device_status() == 0
    ref = route_scores64(dw.dm, dw.kv.pool_sum, dw.kv.len, h1, s.group, s.head_dim)
    # sums of 2 d = 1536 and r = 96 fp32 products: 1e-6 of the scores' size
    assert float((sc.double() - ref).abs().max()) < 2e-6 * max(1.0, float(ref.abs().max()))


def test_route_checks_write_nothing():
    w = rows_of(C.T_GQA, 3)
    dw = D.build(w)
    s = w.shape
    h1 = synth.h_in(s, 5, 0, range(3), "cuda")
    dw.kv.len.clamp_(min=1)
    sc = torch.full((3, s.n_cand), 7.0, device="cuda")
    bad = dw.k.clone()
    bad[2] = 0   # no Budget Predictor
    dw.ctx.buddy_route(dw.kv, h1, bad, scores_out=sc)
    assert dw.ctx.buddy_device_status() == Bd.BUDDY_DEV_BAD_BUDGET and bool((sc == 7.0).all())
    good_len = dw.kv.len.clone()
    dw.kv.len[1] = dw.kv.cap[1] + 1
    dw.ctx.buddy_route(dw.kv, h1, dw.k, scores_out=sc)
    assert dw.ctx.buddy_device_status() == Bd.BUDDY_DEV_BAD_POSITION and bool((sc == 7.0).all())
    dw.kv.len.copy_(good_len)
    dw.ctx.buddy_route(dw.kv, h1, dw.k, scores_out=sc)
    assert dw.ctx.buddy_device_status() == 0 and not bool((sc == 7.0).any())


def value_error(d, batch):
    """Stored V of an fp32 model's first block against 64 bits: relative error, 2-norm."""
    s = dataclasses.replace(C.SMALL_F32, d_model=d, n_q_heads=d // 64, n_kv_heads=d // 64, n_layers=3)
    w = synth.layer_weights(s, 5, 0, "cuda")
    layer = pkg.pack_layer(w)
    ctx = pkg.Context.for_shape(s, max_batch=batch, max_pos=4)
    ctx.buddy_set_weights([layer] * 3, synth.dm_weights(s, 5, "cuda"))
    kv = pkg.KVCache(3, s.n_kv_heads, 64, [1] * batch, torch.float32, "cuda")
    h = synth.h_in(s, 5, 0, range(batch), "cuda")
    ctx.buddy_decode_step(kv, h, torch.ones(batch, dtype=torch.int32, device="cuda"), torch.empty_like(h))
    assert ctx.buddy_device_status() == 0
    v = torch.stack([kv.view("v", 0, i)[:, 0].reshape(-1) for i in range(batch)]).double()
    x = h.double()
    x = x * torch.rsqrt(x.square().mean(1, keepdim=True) + s.rms_eps) * layer["attn_norm"].double()
    ref = x @ w["w_v"].double().T + w["b_v"].double()
    return float((v - ref).norm() / ref.norm())


# above 28 rows tiles, up to 28 a warp per sum: a tree of 32 sums of K / 32 products; 2%: other rows, other errors
@pytest.mark.parametrize("d", [256, 512, 2048])
def test_f32_tiles_keep_the_warp_sums_precision(d):
    assert value_error(d, 64) < 1.02 * value_error(d, 24)


def score_error(s, B):
    """Scores of a decode step after one block over a single position, against 64 bits from the stored V on."""
    T = torch.float64
    w = synth.layer_weights(s, 5, 0, "cuda")
    dm = synth.dm_weights(s, 5, "cuda")
    ctx = pkg.Context.for_shape(s, max_batch=B, max_pos=4)
    layer = pkg.pack_layer(w)
    ctx.buddy_set_weights([layer] * s.n_layers, dm)
    kv = pkg.KVCache(s.n_layers, s.n_kv_heads, s.head_dim, [1] * B, torch.bfloat16, "cuda")
    h = synth.h_in(s, 5, 0, range(B), "cuda")
    sc = torch.empty(B, s.n_cand, device="cuda")
    ctx.buddy_decode_step(kv, h, torch.ones(B, dtype=torch.int32, device="cuda"), torch.empty_like(h), scores_out=sc)
    assert ctx.buddy_device_status() == 0
    v = torch.stack([kv.view("v", 0, i)[:, 0] for i in range(B)]).to(T)
    v = v[:, :, None].expand(-1, -1, s.group, -1).reshape(B, s.q_dim)
    x = h.to(T) + v @ layer["w_o"].to(T).T
    y = x * torch.rsqrt(x.square().mean(1, keepdim=True) + s.rms_eps) * layer["ffn_norm"].to(T)
    g, u = (y @ layer["w_gate_up"].to(T).T).chunk(2, 1)
    x = torch.cat([v, x + (torch.nn.functional.silu(g) * u) @ layer["w_down"].to(T).T], 1)
    d = {k: t.to(T) for k, t in dm.items()}
    ref = torch.nn.functional.silu(x @ d["w1"].T + d["b1"]) @ d["w2"].T + d["b2"]
    return float((sc.to(T) - ref).norm() / ref.norm())


@pytest.mark.parametrize("base", [C.LLAMA3_8B, C.LLAMA2_13B], ids=lambda s: s.name)
def test_scores_keep_the_feeding_blocks_precision(base):
    """What is left is the fp32 sums: a tensor-core accumulator truncates at each K = 16 step, about 2^-24 of
    the sum a time, and a sum of n steps (hi and lo) ends n / 2^24 off.  Gate and up in four K splits take 128
    to 160 steps, down about 200: 2e-5 of the block's update, less than half of the scores; gate and up in one
    sum take 512 to 640 and twice that in all."""
    assert score_error(dataclasses.replace(base, n_layers=34), 16) < 1.0e-5


# rows wider than one pass of the epilogue warps holds (8192): 1056 steps if no projection is split
@pytest.mark.parametrize("batch", [1, 2])
def test_panels_of_a_wide_model(batch):
    wide = dataclasses.replace(C.LLAMA3_8B, name="wide", n_layers=34, d_model=8448, n_q_heads=66, n_kv_heads=11,
                               ffn_dim=2048, random_norm=True)
    assert score_error(wide, batch) < 1056 / 2**24


# gate/up split up to 16 rows, whole above: the same step by its profile and by its values
@pytest.mark.parametrize("batch,fixups", [(3, 4), (16, 4), (17, 3)])
def test_gate_up_splits_by_rows(batch, fixups):
    s = dataclasses.replace(C.LLAMA3_8B, n_layers=3)
    layer = pkg.pack_layer(synth.layer_weights(s, 5, 0, "cuda"))
    h, k = synth.h_in(s, 5, 0, range(batch), "cuda"), torch.ones(batch, dtype=torch.int32, device="cuda")
    outs = []
    for max_batch in (batch, 17 if batch < 17 else 200):   # both forms of the rows up to 16
        ctx = pkg.Context.for_shape(s, max_batch=max_batch, max_pos=4)
        ctx.buddy_set_weights([layer] * 3, synth.dm_weights(s, 5, "cuda"))
        kv = pkg.KVCache(3, s.n_kv_heads, s.head_dim, [1] * batch, torch.bfloat16, "cuda")
        out = torch.empty_like(h)
        ctx.buddy_set_profiling(True)
        ctx.buddy_decode_step(kv, h, k, out)
        n = ctx.buddy_profile_read()["gemm_fixup"][1]
        assert n == (2 * fixups + 4 if max_batch == batch else 10)   # the first block's gate/up is always split
        outs.append(out)
    # bf16 activations between the projections, as parity.py
    assert float(((outs[0] - outs[1]).abs().amax(1) / outs[1].abs().amax(1)).max()) < 2e-2


def silu_context(r, n_layers):
    """A router whose scores are silu(x + b1) of the first r channels x of h1."""
    s = dataclasses.replace(C.SMALL_F32, n_layers=n_layers, dm_hidden=r)
    ctx = pkg.Context.for_shape(s, max_batch=256, max_pos=4)
    layer = pkg.pack_layer(synth.layer_weights(s, 0, 0, "cuda"))
    dm = {"w1": torch.zeros(r, 2 * s.d_model, device="cuda"), "b1": torch.zeros(r, device="cuda"),
          "w2": torch.eye(s.n_cand, r, device="cuda"), "b2": torch.zeros(s.n_cand, device="cuda")}
    dm["w1"][:, s.d_model:s.d_model + r] = torch.eye(r, device="cuda")
    kv = pkg.KVCache(s.n_layers, s.n_kv_heads, s.head_dim, [1] * 256, torch.float32, "cuda")
    kv.len.fill_(1)
    h1, k = torch.zeros(256, s.d_model, device="cuda"), torch.ones(256, dtype=torch.int32, device="cuda")
    scores = torch.empty(256, s.n_cand, device="cuda")

    def run(x=None, b1=None):
        if x is not None:
            h1[:, :r] = x
        if b1 is not None:
            dm["b1"].fill_(b1)
        ctx.buddy_set_weights([layer] * s.n_layers, dm)
        ctx.buddy_route(kv, h1, k, scores_out=scores)
        assert ctx.buddy_device_status() == 0
        return scores
    return run


def test_silu_is_the_division():
    """silu(x) over the float range: at most an ulp from the device's own x / (1 + e^-x), where 1 + e^-x
    passes 1e38 (x below -87.5) and overflows (below -88.7) included."""
    run = silu_context(126, 128)
    g = torch.Generator(device="cuda").manual_seed(3)
    n = 256 * 126
    bits = torch.randint(-2**31, 2**31 - 1, (n,), generator=g, device="cuda").int().view(torch.float32)
    for x in (bits.nan_to_num(0.5, 3e38, -3e38), torch.linspace(-89, -87, n, device="cuda"),
              torch.linspace(-110, 30, n, device="cuda"), torch.linspace(-1, 1, n, device="cuda")):
        x = x.view(256, 126)
        got, ref = run(x), x / (1.0 + torch.exp(-x))
        ulp = torch.maximum((torch.nextafter(ref.abs(), ref.new_tensor(float("inf"))) - ref.abs()), ref.new_tensor(2.0**-149))
        assert bool(((got - ref).abs() <= ulp).all()), float(((got - ref).abs() / ulp).max())
    one = silu_context(1, 3)
    for b in (float("inf"), float("-inf"), float("nan"), 3.4e38, -3.4e38, -88.72, -88.73, -0.0):
        x = torch.tensor(b, device="cuda")
        ref = float(x / (1.0 + torch.exp(-x)))
        np.testing.assert_allclose(one(b1=b)[:, 0].cpu().numpy(), np.float32(ref), rtol=1.2e-7, atol=0)


# two groups of rows (the first kernel checks after its products), the bad row in the second
def test_route_checks_write_nothing_two_row_groups():
    w = rows_of(C.T_GQA, 16)
    dw = D.build(w)
    s = w.shape
    h1 = synth.h_in(s, 5, 0, range(16), "cuda")
    dw.kv.len.clamp_(min=1)
    sc, sel = torch.full((16, s.n_cand), 7.0, device="cuda"), torch.full((16, s.n_cand), 7, dtype=torch.int32, device="cuda")
    bad = dw.k.clone()
    bad[15] = s.n_cand + 1
    good_len = dw.kv.len.clone()
    for k, length, flag in ((bad, good_len[15], Bd.BUDDY_DEV_BAD_BUDGET), (dw.k, dw.kv.cap[15] + 1, Bd.BUDDY_DEV_BAD_POSITION),
                            (bad, -1, Bd.BUDDY_DEV_BAD_BUDGET | Bd.BUDDY_DEV_BAD_POSITION)):
        dw.kv.len[15] = length
        dw.ctx.buddy_route(dw.kv, h1, k, sel_out=sel, scores_out=sc)
        assert dw.ctx.buddy_device_status() == flag and bool((sc == 7.0).all()) and bool((sel == 7).all())
    dw.kv.len.copy_(good_len)
    dw.ctx.buddy_route(dw.kv, h1, dw.k, sel_out=sel, scores_out=sc)
    assert dw.ctx.buddy_device_status() == 0 and not bool((sc == 7.0).any())


def append_state(shape, caps, max_batch):
    ctx = pkg.Context.for_shape(shape, max_batch=max_batch, max_pos=max(caps))
    layer = pkg.pack_layer(synth.layer_weights(shape, 0, 0, "cuda"))
    ctx.buddy_set_weights([layer] * shape.n_layers, synth.dm_weights(shape, 0, "cuda"))
    return ctx, pkg.KVCache(shape.n_layers, shape.n_kv_heads, shape.head_dim, caps, synth.storage_dtype(shape), "cuda")


# 16-byte copies (8 positions per CTA) and, from a misaligned source, element
# copies; up to 256 sequences the copy kernel checks the arguments itself
@pytest.mark.parametrize("shape", [C.SMALL_GQA_BF16, C.SMALL_F32], ids=lambda s: s.name)
@pytest.mark.parametrize("n_new,n_seq", [(1, 3), (8, 1), (9, 256), (33, 257)])
def test_append_aligned_and_misaligned(shape, n_new, n_seq):
    dt = synth.storage_dtype(shape)
    n = n_seq * n_new * shape.kv_dim
    g = torch.Generator(device="cuda").manual_seed(n)
    flat = [torch.empty(n + 1, dtype=dt, device="cuda").normal_(generator=g) for _ in range(2)]
    view = lambda t, o: t[o:o + n].view(n_seq, n_new, shape.n_kv_heads, shape.head_dim)
    off = [view(t, 1) for t in flat]                 # not 16-byte aligned
    same = [t.clone() for t in off]                  # aligned
    ids = torch.arange(n_seq, dtype=torch.int32, device="cuda").flip(0).contiguous()
    states = []
    for kn, vn in (same, off):
        ctx, kv = append_state(shape, [2 * n_new + 3] * n_seq, 4)
        for _ in range(2):
            ctx.buddy_kv_append(kv, 0, ids, kn, vn, advance=True)
        assert ctx.buddy_device_status() == 0
        states.append((kv, ctx))
    a, b = states[0][0], states[1][0]
    assert torch.equal(a.k[0], b.k[0]) and torch.equal(a.v[0], b.v[0]) and torch.equal(a.pool_sum, b.pool_sum)
    for j in (0, n_seq - 1):
        s = int(ids[j])
        assert torch.equal(a.view("k", 0, s)[:, n_new:2 * n_new].transpose(0, 1), same[0][j])
        ref = a.view("v", 0, s)[:, :2 * n_new].double().sum(1).reshape(-1)
        np.testing.assert_allclose(a.pool_sum[s].double().cpu(), ref.cpu(), rtol=1e-5, atol=1e-5)
    # a third append does not fit: flagged, nothing written
    k0, len0 = a.k[0].clone(), a.len.clone()
    a.len.add_(4)
    states[0][1].buddy_kv_append(a, 0, ids, same[0], same[1], advance=True)
    assert states[0][1].buddy_device_status() & Bd.BUDDY_DEV_BAD_POSITION
    assert torch.equal(a.k[0], k0) and torch.equal(a.len, len0 + 4)
    a.len.copy_(len0 - n_new)
    ids[0] = n_seq
    states[0][1].buddy_kv_append(a, 0, ids, same[0], same[1], advance=True)
    assert states[0][1].buddy_device_status() & Bd.BUDDY_DEV_BAD_SEQ and torch.equal(a.k[0], k0)


# clusters of 8 CTAs over 1 to 9 positions: CTAs with an empty share reach their
# stores to CTA 0 at once
@pytest.mark.parametrize("shape", [C.SMALL_GQA_BF16, C.SMALL_QWEN_BF16, C.SMALL_F32], ids=lambda s: s.name)
@pytest.mark.parametrize("n_new", [1, 2, 7, 9])
def test_pooled_context_of_shares_shorter_than_the_cluster(shape, n_new):
    g = torch.Generator(device="cuda").manual_seed(n_new)
    ids = torch.tensor([0, 1], dtype=torch.int32, device="cuda")
    kn, vn = (torch.empty(2, n_new, shape.n_kv_heads, shape.head_dim, dtype=synth.storage_dtype(shape),
                          device="cuda").normal_(generator=g) for _ in range(2))
    ctx, kv = append_state(shape, [n_new, n_new], 2)
    pools = []
    for _ in range(20):
        ctx.buddy_kv_append(kv, 0, ids, kn, vn, advance=False)
        pools.append(kv.pool_sum.clone())
    assert ctx.buddy_device_status() == 0
    np.testing.assert_allclose(pools[0].double().cpu(), vn.double().sum(1).reshape(2, -1).cpu(), rtol=1e-5, atol=1e-5)
    assert all(torch.equal(p, pools[0]) for p in pools)


# attention clusters of 16 to 2 CTAs over 1 to 4 positions
@pytest.mark.parametrize("batch", [1, 2, 5, 10, 21])
def test_decode_parity_shares_shorter_than_the_cluster(batch):
    w = C.scaled(C.T_GQA, ctx=[i % 4 for i in range(batch)], k=[1 + i % 4 for i in range(batch)], name="short-ctx")
    assert run_parity(w, steps=2)[0] < 2e-2


# kernel attributes belong to a function on the device, not to a context: contexts of other shapes and batches,
# created in between and smaller or larger, must not take them from one another
def test_contexts_of_other_shapes_side_by_side():
    wide = dataclasses.replace(C.SMALL_QWEN_BF16, name="wide", d_model=4096, n_q_heads=32, n_kv_heads=8)
    ws = [dataclasses.replace(C.scaled(C.T_QWEN, ctx=[40], k=[2], name="wide-b1"), shape=wide),
          C.scaled(C.T_GQA, ctx=[70], k=[1], name="gqa-b1"),
          rows_of(C.T_GQA, 200), rows_of(C.T_GQA, 37), rows_of(C.T_F32, 200), rows_of(C.T_F32, 30)]

    def step(dw, w):
        h = torch.empty(w.batch, w.shape.d_model, device="cuda")
        dw.ctx.buddy_decode_step(dw.kv, synth.workload_h_in(w, 0, "cuda"), dw.k, h)
        assert dw.ctx.buddy_device_status() == 0
        return h
    alone = []
    for w in ws:
        dw = D.build(w)
        alone.append(step(dw, w))
        dw.ctx.close()
    live = [D.build(w) for w in ws]
    for i in list(range(len(ws)))[::-1]:   # the smallest of each kind was prepared last
        if ws[i].batch in (30, 37) or ws[i].name == "gqa-b1":
            assert torch.equal(step(live[i], ws[i]), alone[i])
    for i, w in enumerate(ws):
        if not (w.batch in (30, 37) or w.name == "gqa-b1"):
            assert torch.equal(step(live[i], w), alone[i])


def test_misaligned_router_buffers_rejected_on_host():
    """The Decision Module's and the Budget Predictor's first matrix and the pooled sums, off by 4 bytes."""
    w = rows_of(C.T_GQA, 3)
    dw = D.build(w)
    s = w.shape
    off = lambda t: torch.cat([t.new_zeros(1), t.reshape(-1)])[1:].view(t.shape)
    bad = off(dw.dm["w1"])
    assert bad.data_ptr() % 16 == 4 and bad.is_contiguous()
    h1, sc = synth.h_in(s, 5, 0, range(3), "cuda"), torch.full((3, s.n_cand), 7.0, device="cuda")
    dw.kv.len.clamp_(min=1)
    pred = {k: dw.dm[k] for k in ("b1", "w2", "b2")}
    pool = dw.kv.state.pool_sum
    for call in (lambda: dw.ctx.buddy_set_weights(dw.layers, {**dw.dm, "w1": bad}),
                 lambda: dw.ctx.buddy_set_budget_predictor({**pred, "w1": bad}),
                 lambda: dw.ctx.buddy_route(dw.kv, h1, dw.k, scores_out=sc)):
        dw.kv.state.pool_sum = pool + 4
        with pytest.raises(Bd.BuddyError) as e:
            call()
        assert e.value.code == Bd.BUDDY_ERR_ARG
    dw.kv.state.pool_sum = pool
    torch.cuda.synchronize()
    assert bool((sc == 7.0).all())
    dw.ctx.buddy_route(dw.kv, h1, dw.k, scores_out=sc)
    assert dw.ctx.buddy_device_status() == 0 and not bool((sc == 7.0).any())


def test_panel_wait_limit_runs_out_and_context_recovers():
    """As the other batches' test: 1 ns runs out, the restored limit gives a fresh context's result."""
    w = C.scaled(C.T_GQA, ctx=[5, 200], k=[1, 3], name="t-gqa-b2-timeout")
    h_in = synth.workload_h_in(w, 0, "cuda")
    outs = []
    for limited in (False, True):
        dw = D.build(w)
        h = torch.empty(2, w.shape.d_model, device="cuda")
        len0, pool0 = dw.kv.len.clone(), dw.kv.pool_sum.clone()
        if limited:
            dw.ctx.buddy_set_wait_limit(1)
            dw.ctx.buddy_decode_step(dw.kv, h_in, dw.k, h)
            assert dw.ctx.buddy_device_status() & Bd.BUDDY_DEV_TIMEOUT
            dw.ctx.buddy_set_wait_limit(0)
            dw.kv.len.copy_(len0)
            dw.kv.pool_sum.copy_(pool0)
        dw.ctx.buddy_decode_step(dw.kv, h_in, dw.k, h)
        assert dw.ctx.buddy_device_status() == 0
        outs.append(h)
    assert torch.equal(*outs)


# the decode GEMMs (40 tokens), the CTA pairs and, in the first block's down projection, units cut along K (300
# tokens; test_gpu_prefill_units.py holds the other schedules)
@pytest.mark.parametrize("lengths", [[33, 7], [290, 10]], ids=lambda v: str(sum(v)))
def test_prefill_wait_limit_runs_out_and_context_recovers(lengths):
    w = C.scaled(C.T_QWEN, ctx=[3, 60], k=[2, 4], name="pf-timeout")
    T = sum(lengths)
    x = synth.prompt_inputs(w.shape, w.seed, lengths, "cuda")
    outs = []
    for limited in (False, True):
        dw = D.build(w, extra_steps=max(lengths) + 2, max_prefill_tokens=T)
        h = torch.empty(T, w.shape.d_model, device="cuda")
        len0 = dw.kv.len.clone()
        if limited:
            dw.ctx.buddy_set_wait_limit(1)
            dw.ctx.buddy_prefill(dw.kv, lengths, x, dw.k, h)
            assert dw.ctx.buddy_device_status() & Bd.BUDDY_DEV_TIMEOUT
            dw.ctx.buddy_set_wait_limit(0)
            dw.kv.len.copy_(len0)
        dw.ctx.buddy_prefill(dw.kv, lengths, x, dw.k, h)
        assert dw.ctx.buddy_device_status() == 0
        outs.append(h)
    assert torch.equal(*outs)
