// Routed prefill (Sec. 4.1; App. E "Prefill vs. Decode"): a batch of prompts
// passes blocks 0..c token by token with causal attention; each prompt is
// routed once, from its pooled context-layer cache (the prompt included) and
// its last token's hidden state after block c; the routed blocks each run on
// every token of the prompts that selected them (grouping by mask, App. C.1);
// a prompt that skips a block stores zero K/V at all its positions there (or
// nothing, in the masked variant).
//
// The host orchestrates one call: the token tables go to the device in one copy,
// blocks 0..c and the router run, then one synchronisation brings the routes back
// so that the host can size every later launch exactly (row lists and attention
// work items per block, one copy more) instead of launching empty tiles.  The
// copies use pinned memory: from pageable memory every one of eight cost the host
// a staging copy, and the two reads a wait each, with the GPU idle after the router
// (one prompt of 61 tokens, 4 blocks: 460 -> 449 us).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "internal.h"

namespace buddy {

// ---------------------------------------------------------------------------
// Token tables, checks, gathers and the position advance
// ---------------------------------------------------------------------------
__global__ void pf_tokens_kernel(int T, const int32_t* tok_seq, const int32_t* tok_t, const int32_t* len,
                                 const int64_t* seq_off, const int32_t* cap, int32_t* tok_pos, int64_t* tok_off,
                                 int32_t* tok_cap, const int32_t* status) {
  pdl_wait();
  pdl_trigger();
  if (call_aborted(status)) return;
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= T) return;
  const int s = tok_seq[r];
  tok_pos[r] = len[s] + tok_t[r];
  tok_off[r] = seq_off[s];
  tok_cap[r] = cap[s];
}

// Budgets in range (0 allowed with a Budget Predictor), and room for every
// prompt: len + n_tok <= cap and <= max_pos (masked variant: every layer's
// length within [0, len]).  Publishes the call's abort word.
__global__ void pf_check_kernel(int B, const int32_t* k, int Lm, int k_min, const int32_t* n_tok,
                                const int32_t* len, const int32_t* cap, int max_pos, const int32_t* layer_len, int L,
                                int kv_batch, int32_t* status) {
  pdl_wait();
  pdl_trigger();
  __shared__ int bad;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  int b = 0;
  for (int i = threadIdx.x; i < B; i += blockDim.x) {
    const int ki = k[i];
    if (ki < k_min || ki > Lm) b |= BUDDY_DEV_BAD_BUDGET;
    const int n = len[i], t = n_tok[i];
    if (n < 0 || n + t > cap[i] || n + t > max_pos) b |= BUDDY_DEV_BAD_POSITION;
    if (layer_len != nullptr)
      for (int l = 0; l < L; ++l) {
        const int nl = layer_len[(size_t)l * kv_batch + i];
        if (nl < 0 || nl > n) b |= BUDDY_DEV_BAD_POSITION;
      }
  }
  if (b) atomicOr(&bad, b);
  __syncthreads();
  if (threadIdx.x == 0) {
    status[1] = bad ? 1 : 0;
    if (bad) atomicOr(status, bad);
  }
}

// The router's inputs: the last prompt token's hidden state per sequence and
// the number of positions the pooled context covers (len + n_tok).
__global__ void pf_gather_kernel(int B, int d, const int32_t* tok_end, const float* H, const int32_t* len,
                                 const int32_t* n_tok, float* hlast, int32_t* cnt, const int32_t* status) {
  pdl_wait();
  pdl_trigger();
  if (call_aborted(status)) return;
  const int i = blockIdx.x;
  const float* src = H + (size_t)(tok_end[i] - 1) * d;
  for (int e = threadIdx.x; e < d; e += blockDim.x) hlast[(size_t)i * d + e] = src[e];
  if (threadIdx.x == 0) cnt[i] = len[i] + n_tok[i];
}

// Zero K and V at every prompt position of the routed blocks a prompt skips, a
// CTA per (block, prompt, KV head), 16 bytes at a time (5 prompts of 128..1023
// tokens, 2 routed blocks: 11 us, against 92 us with a CTA per block and prompt
// storing elements).
__global__ void pf_zero_kernel(int B, int L, int first, int nkv, int hd, const uint8_t* mask, LayerPtrs ptrs,
                               const int32_t* len, const int32_t* n_tok, const int64_t* seq_off,
                               const int32_t* cap, const int32_t* status) {
  pdl_wait();
  pdl_trigger();
  if (call_aborted(status)) return;
  const int l = first + blockIdx.x, i = blockIdx.y, g = blockIdx.z;
  if (l >= L - 1 || mask[(size_t)i * L + l]) return;
  const int64_t base = kv_offset(seq_off, cap, i, nkv, hd, g, len[i]);
  uint4* Kc = reinterpret_cast<uint4*>((bf16*)ptrs.k[l] + base);
  uint4* Vc = reinterpret_cast<uint4*>((bf16*)ptrs.v[l] + base);
  const int64_t n = (int64_t)n_tok[i] * hd / 8;
  for (int64_t x = threadIdx.x; x < n; x += blockDim.x) {
    Kc[x] = make_uint4(0u, 0u, 0u, 0u);
    Vc[x] = make_uint4(0u, 0u, 0u, 0u);
  }
}

// len[i] += n_tok[i]; masked variant: layer_len[l][i] += n_tok[i] where the
// prompt executed layer l.
__global__ void pf_advance_kernel(int B, int L, const int32_t* n_tok, const uint8_t* mask, int32_t* len,
                                  int32_t* layer_len, int kv_batch, const int32_t* status) {
  pdl_wait();
  pdl_trigger();
  if (call_aborted(status)) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B) return;
  const int t = n_tok[i];
  len[i] += t;
  if (layer_len != nullptr)
    for (int l = 0; l < L; ++l) layer_len[(size_t)l * kv_batch + i] += mask[(size_t)i * L + l] ? t : 0;
}

// ---------------------------------------------------------------------------
// One block over m prompt-token rows
// ---------------------------------------------------------------------------
struct PfLayerWork {
  const int32_t* rows;     // device [m] token rows, or nullptr (all tokens, identity)
  int m;
  const int4* items;       // device attention work items
  int n_items;
};

static void pf_block(Ctx& c, const buddy_kv_state& kv, int l, const PfLayerWork& w, const float* src, float* H,
                     cudaStream_t s, bool prof) {
  const buddy_layer_weights& W = c.layers[l];
  const bool split = l <= c.cl;   // blocks that feed the router keep ~16-bit activations
  const RowSel sel{w.rows, nullptr, w.m};
  const int32_t* base = cache_len(c, kv, l);
  {
    ProfScope p(c, s, BUDDY_PROF_PF_OTHER, 1, prof);
    launch_rmsnorm(c, src, sel, W.attn_norm, c.pf_xn, split ? c.pf_xn_lo : nullptr, s);
  }
  PfEpi e{};
  e.rows = w.rows;
  e.q_out = c.pf_q;
  e.bias = W.b_qkv;
  e.tok_seq = c.pf_tok_seq;
  e.tok_pos = c.pf_tok_pos;
  e.len = kv.len;
  e.cache_len = base;
  e.seq_off = kv.seq_off;
  e.cap = kv.cap;
  e.kc = kv.k_cache[l];
  e.vc = kv.v_cache[l];
  e.tok_off = c.pf_tok_off;
  e.tok_cap = c.pf_tok_cap;
  {
    ProfScope p(c, s, BUDDY_PROF_PF_GEMM, 1, prof);
    p.rec.launches = launch_gemm_pf(c, EPI_QKV, split, l, 0, 0, w.m, e, s);
  }
  {
    ProfScope p(c, s, BUDDY_PROF_PF_ATTENTION, 1, prof);
    launch_attention_pf(c, w.n_items, w.items, c.pf_n_tok, base, kv, l, c.pf_q, c.pf_attn,
                        split ? c.pf_attn_lo : nullptr, s);
  }
  e = PfEpi{};
  e.rows = w.rows;
  e.resid_src = src;
  e.resid_dst = H;
  {
    ProfScope p(c, s, BUDDY_PROF_PF_GEMM, 1, prof);
    p.rec.launches = launch_gemm_pf(c, EPI_RESID, split, l, 1, 1, w.m, e, s);
  }
  {
    ProfScope p(c, s, BUDDY_PROF_PF_OTHER, 1, prof);
    launch_rmsnorm(c, H, sel, W.ffn_norm, c.pf_xn, split ? c.pf_xn_lo : nullptr, s);
  }
  e = PfEpi{};
  e.out_act = c.pf_act;
  e.out_act_lo = split ? c.pf_act_lo : nullptr;
  {
    ProfScope p(c, s, BUDDY_PROF_PF_GEMM, 1, prof);
    p.rec.launches = launch_gemm_pf(c, EPI_SWIGLU, split, l, 2, 0, w.m, e, s);
  }
  e = PfEpi{};
  e.rows = w.rows;
  e.resid_src = H;
  e.resid_dst = H;
  {
    ProfScope p(c, s, BUDDY_PROF_PF_GEMM, 1, prof);
    p.rec.launches = launch_gemm_pf(c, EPI_RESID, split, l, 3, 2, w.m, e, s);
  }
}

// ---------------------------------------------------------------------------
// The call
// ---------------------------------------------------------------------------
// Arrays packed into a context's pinned area and copied to its device area
// together.
struct PfUpload {
  uint8_t* host;
  uint8_t* dev;
  size_t begin, at, end;
  PfUpload(const Ctx& c, size_t from, size_t to) : host(c.pf_up_host), dev(c.pf_up), begin(from), at(from), end(to) {
    begin = at = (from + 15) & ~size_t(15);
  }
  // Device address of a copy of v[0 .. n), or nullptr when the area is full.
  template <typename T>
  const T* add(const T* v, size_t n) {
    if (at + n * sizeof(T) > end) return nullptr;
    if (n) std::memcpy(host + at, v, n * sizeof(T));
    const T* d = reinterpret_cast<const T*>(dev + at);
    at = (at + n * sizeof(T) + 15) & ~size_t(15);
    return d;
  }
  cudaError_t send(cudaStream_t s) {
    return at == begin ? cudaSuccess
                       : cudaMemcpyAsync(dev + begin, host + begin, std::min(at, end) - begin, cudaMemcpyHostToDevice, s);
  }
};

int run_prefill(Ctx& c, const buddy_kv_state& kv, int B, const int32_t* n_tok_host, const float* x, const int32_t* k,
                float* h_out, uint8_t* mask_out, float* scores_out, cudaStream_t s) {
  const bool prof = c.profiling != 0;
  std::vector<int32_t> off(B + 1, 0);
  for (int i = 0; i < B; ++i) off[i + 1] = off[i] + n_tok_host[i];
  const int T = off[B];
  std::vector<int32_t> tok_seq(T), tok_t(T);
  for (int i = 0; i < B; ++i)
    for (int t = 0; t < n_tok_host[i]; ++t) {
      tok_seq[off[i] + t] = i;
      tok_t[off[i] + t] = t;
    }
  std::vector<int32_t> ends(off.begin() + 1, off.end());
#define PCK(x)                                                                             \
  do {                                                                                     \
    cudaError_t e_ = (x);                                                                  \
    if (e_ != cudaSuccess) {                                                               \
      fprintf(stderr, "libbuddy: prefill: %s -> %s\n", #x, cudaGetErrorString(e_));        \
      return BUDDY_ERR_CUDA;                                                               \
    }                                                                                      \
  } while (0)
  // attention work items for a set of sequences: (token, head of a group) rows
  // of one KV head, those that see the most positions first (the last to start
  // are then the shortest)
  const int G = c.nq / c.nkv;
  auto items_for = [&](const std::vector<int>& seqs, bool split, std::vector<int4>& out) {
    const int rows = attention_pf_rows(split);
    const size_t at = out.size();
    int j = 0;
    for (int i : seqs) {
      for (int r0 = 0; r0 < n_tok_host[i] * G; r0 += rows)
        for (int g = 0; g < c.nkv; ++g) out.push_back(make_int4(i, g, j, r0));
      j += n_tok_host[i];
    }
    std::stable_sort(out.begin() + at, out.end(), [](const int4& a, const int4& b) { return a.w > b.w; });
  };
  std::vector<int> all(B);
  for (int i = 0; i < B; ++i) all[i] = i;
  // the item buffer: every sequence for the blocks that feed the router, every
  // sequence for the last block, then the routed layers
  std::vector<int4> items_all;
  items_for(all, true, items_all);
  const int n_split = (int)items_all.size();
  items_for(all, false, items_all);
  PfUpload up(c, 0, c.pf_up_second);
  c.pf_tok_seq = up.add(tok_seq.data(), T);
  const int32_t* d_tok_t = up.add(tok_t.data(), T);
  c.pf_n_tok = up.add(n_tok_host, B);
  const int32_t* d_ends = up.add(ends.data(), B);
  const int4* d_items = up.add(items_all.data(), items_all.size());
  if (!d_items) return BUDDY_ERR_RANGE;
  PCK(up.send(s));
  const PfLayerWork feed{nullptr, T, d_items, n_split};
  const PfLayerWork every{nullptr, T, d_items + n_split, (int)items_all.size() - n_split};
  const int k_min = c.have_pred ? 0 : 1;
  launch_k(pf_check_kernel, 1, 256, 0, s, c.pdl, B, k, c.Lm, k_min, c.pf_n_tok, (const int32_t*)kv.len, kv.cap,
           c.max_pos, (const int32_t*)(c.masked ? kv.layer_len : nullptr), c.L, kv.batch, c.status);
  launch_k(pf_tokens_kernel, (T + 255) / 256, 256, 0, s, c.pdl, T, c.pf_tok_seq, d_tok_t, (const int32_t*)kv.len,
           kv.seq_off, kv.cap, c.pf_tok_pos, c.pf_tok_off, c.pf_tok_cap, (const int32_t*)c.status);

  // blocks 0..c on every token, then the router per prompt
  for (int l = 0; l <= c.cl; ++l) pf_block(c, kv, l, feed, l == 0 ? x : h_out, h_out, s, prof);
  {
    ProfScope p(c, s, BUDDY_PROF_ROUTE, 4, prof);
    launch_pool_refresh_n(c, kv, B, c.pf_n_tok, s);
    launch_k(pf_gather_kernel, B, 256, 0, s, c.pdl, B, c.d, d_ends, (const float*)h_out,
             (const int32_t*)kv.len, c.pf_n_tok, c.pf_hlast, c.pf_cnt, (const int32_t*)c.status);
    launch_route(c, B, c.pf_hlast, kv.pool_sum, c.pf_cnt, 0, k, c.mask, c.sel, c.scores, s);
  }
  // the routes come back to the host, which sizes every later launch
  const volatile int32_t* st = reinterpret_cast<const volatile int32_t*>(c.pf_down);
  const uint8_t* mask = c.pf_down + 16;
  PCK(cudaMemcpyAsync(c.pf_down, c.status, 2 * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  PCK(cudaMemcpyAsync(c.pf_down + 16, c.mask, (size_t)B * c.L, cudaMemcpyDeviceToHost, s));
  PCK(cudaStreamSynchronize(s));
  if (st[1] != 0) return BUDDY_ERR_DEVICE;   // checks failed: nothing was written

  if (!c.masked) {
    LayerPtrs p;
    for (int l = 0; l < c.L; ++l) {
      p.k[l] = kv.k_cache[l];
      p.v[l] = kv.v_cache[l];
    }
    ProfScope ps(c, s, BUDDY_PROF_PF_OTHER, 1, prof);
    dim3 g(std::max(1, c.Lm), B, c.nkv);
    launch_k(pf_zero_kernel, g, 256, 0, s, c.pdl, B, c.L, c.cl + 1, c.nkv, c.hd, (const uint8_t*)c.mask, p,
             (const int32_t*)kv.len, c.pf_n_tok, kv.seq_off, kv.cap, (const int32_t*)c.status);
  }
  // row lists and work items of the routed layers
  std::vector<int32_t> rows_all;
  std::vector<int4> items_l;
  std::vector<PfLayerWork> work(c.L);
  std::vector<size_t> row_at(c.L), item_at(c.L);
  for (int l = c.cl + 1; l < c.L - 1; ++l) {
    std::vector<int> seqs;
    for (int i = 0; i < B; ++i)
      if (mask[(size_t)i * c.L + l]) seqs.push_back(i);
    row_at[l] = rows_all.size();
    item_at[l] = items_l.size();
    for (int i : seqs)
      for (int t = off[i]; t < off[i + 1]; ++t) rows_all.push_back(t);
    items_for(seqs, false, items_l);
    work[l].m = (int)(rows_all.size() - row_at[l]);
    work[l].n_items = (int)(items_l.size() - item_at[l]);
  }
  PfUpload up2(c, c.pf_up_second, c.pf_up_bytes);
  const int32_t* d_rows = up2.add(rows_all.data(), rows_all.size());
  const int4* d_items_l = up2.add(items_l.data(), items_l.size());
  if (!d_rows || !d_items_l) return BUDDY_ERR_RANGE;
  PCK(up2.send(s));
  for (int l = c.cl + 1; l < c.L - 1; ++l) {
    if (work[l].m == 0) continue;
    work[l].rows = d_rows + row_at[l];
    work[l].items = d_items_l + item_at[l];
    pf_block(c, kv, l, work[l], h_out, h_out, s, prof);
  }
  pf_block(c, kv, c.L - 1, every, h_out, h_out, s, prof);
  {
    ProfScope p(c, s, BUDDY_PROF_PF_OTHER, 1, prof);
    launch_k(pf_advance_kernel, (B + 255) / 256, 256, 0, s, c.pdl, B, c.L, c.pf_n_tok,
             (const uint8_t*)c.mask, kv.len, c.masked ? kv.layer_len : nullptr, kv.batch, (const int32_t*)c.status);
  }
  if (mask_out) PCK(cudaMemcpyAsync(mask_out, c.mask, (size_t)B * c.L, cudaMemcpyDeviceToDevice, s));
  if (scores_out)
    PCK(cudaMemcpyAsync(scores_out, c.scores, (size_t)B * c.Lm * sizeof(float), cudaMemcpyDeviceToDevice, s));
  PCK(cudaGetLastError());
#undef PCK
  return BUDDY_OK;
}

}  // namespace buddy
