// Tensor-core GEMM for the prefill projections on sm_103a.
//
//   C[j][n] = sum_k X[j][k] * W[n][k]      (j < m prompt-token rows, n < N features)
//
// A prefill block runs its projections on every token of the prompts that
// selected it, thousands of rows: the GEMM is bound by the tensor pipe, not
// by the weight stream.  A work unit is a 256-row M-tile of X times one
// 256-row weight tile over the whole K (but for the last units, below), computed by
// a pair of CTAs on two SMs (a cluster of 2, tcgen05 cta_group::2): each CTA holds 128 rows of
// X and half of the weight tile, and 128 rows of the accumulator.  A K block
// thus costs an SM 32 KiB of copies instead of the 48 KiB of a 128 x 256 tile
// of its own, and the ring gets seven stages instead of four; a stage's four
// MMAs run back to back at 128 cycles each, the tensor pipe's rate.  Qwen2.5-7B
// gate/up at 8,000 tokens: 1.13 ms (1.92 PFLOP/s) against 2.38 ms with one-SM
// tiles.  Persistent
// pairs walk the units in groups of kPfGroup M-tiles, weight tile by weight
// tile, so that the pairs running at any time share about as many activation
// tiles as weight tiles.  (M-tile by M-tile, every M-tile streams all the
// weights: for a gate/up projection larger than L2 that is an HBM pass per
// M-tile.)
//
// Units that do not fill a last wave of pairs are cut along K (pf_bound; the cut of
// Stream-K, Osama et al. 2023, for the remainder only): each
// pair takes an equal, contiguous share of their K blocks, first of all its work,
// stages the accumulator of a part in a workspace slot, and the pair that
// completes a unit sums the parts in K order and applies the epilogue.  With one
// short prompt every unit is such a unit: Llama-3-8B's O projection has 16, which
// kept 16 of the 76 pairs busy for 64 K blocks (4 blocks of Llama-3-8B, 5 prompts,
// 2,878 tokens: 4.06 -> 3.93 ms; 61 tokens, which launch_gemm_pf now sends
// elsewhere: 0.85 -> 0.73 ms).
//
// Warp 0 of each CTA issues the TMA loads of its part of a stage ([X 128 x 64]
// [X remainder 128 x 64 with SPLIT][W 128 x 64], 128-byte swizzle; the bytes of
// both CTAs are counted on CTA 0's barrier); warp 1 of CTA 0 issues tcgen05.mma
// M = 256, N = 256, K = 16 into one of two TMEM accumulators (512 columns in
// each CTA); warps 2-9 of each CTA drain the other accumulator and apply the
// epilogue.  Every wait on a barrier is bounded; both CTAs reach the cluster
// barriers at the end whatever happened before (they keep the pair alive while
// MMAs read both CTAs' shared memory).
//
// Epilogues: residual add scattered to the token rows; SwiGLU (a tile holds
// 128 gate rows and the matching 128 up rows); QKV (bias, rotate-half RoPE at
// the token's position, q out in fp32, K/V stored in the layer's cache at the
// token's cache position).
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"
#include "gemm_common.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace buddy {

constexpr int kPfEpiWarps = 8;               // two per TMEM lane quarter, half of the columns each
constexpr int kPfThreads = 64 + 32 * kPfEpiWarps;
constexpr int kPfMaxStages = 8;
constexpr int kPfGroup = 8;                    // M-tiles (of 256 rows) walked together
constexpr uint32_t kPfTileBytes = 128u * 128u; // one 128-row x 64-column bf16 tile

struct PfParams {
  int N, K, m;
  int n_tiles, m_tiles, kb_total;
  int units;               // units computed whole, by pair u % pairs
  int sk_units;            // units after them, cut along K over sk_pairs pairs
  int sk_pairs, sk_gran;   // cuts fall on multiples of sk_gran K blocks of a unit
  float4* ws;              // sk: [pair][part 0, 1][CTA] accumulators in fragment form
  int32_t* ctr;            // sk: [unit][CTA] K blocks that have arrived
  int stages;
  uint32_t stage_bytes, w_off;
  // epilogue
  const int32_t* rows;     // compact row j -> token row (residual, QKV); nullptr = identity
  const float* resid_src;
  float* resid_dst;
  bf16* out_act;
  bf16* out_act_lo;
  float* q_out;            // [m, nq * hd] compact
  const float* bias;
  const float* rope_cos;
  const float* rope_sin;
  const int32_t* tok_seq;  // token row -> sequence
  const int32_t* tok_pos;  // token row -> RoPE position
  const int32_t* len;      // sequence -> tokens before this prefill
  const int32_t* cache_len;  // sequence -> the layer's positions before this prefill
  const int64_t* seq_off;
  const int32_t* cap;
  bf16* kc;
  bf16* vc;
  int nq, nkv, hd;
  int32_t* status;
  uint64_t wait_ns;        // limit of each pipeline wait (the drain waits keep kWaitLimitNs)
};

// M-tile and weight tile of unit u: groups of kPfGroup M-tiles, inside a group
// the M-tile varies fastest.
__device__ __forceinline__ void pf_unit(const PfParams& p, int u, int& mt, int& nt) {
  const int per = kPfGroup * p.n_tiles;
  const int g = u / per, r = u - g * per;
  const int gm = min(kPfGroup, p.m_tiles - g * kPfGroup);
  nt = r / gm;
  mt = g * kPfGroup + (r - nt * gm);
}

// Start of pair i's share of the cut units' K blocks, laid end to end.  A share
// is at least sk_gran blocks (sk_pairs is chosen so) and shorter than a unit: it
// touches one unit or two.
__device__ __forceinline__ int pf_bound(const PfParams& p, int i) {
  const int T = p.sk_units * p.kb_total;
  if (i >= p.sk_pairs) return T;
  const int x = i * T / p.sk_pairs, u = x / p.kb_total;
  return u * p.kb_total + (x - u * p.kb_total) / p.sk_gran * p.sk_gran;
}

// A piece of a pair's work: K blocks [kb0, kb1) of unit u; part >= 0 of a cut unit.
struct PfSeg {
  int u, kb0, kb1, part;
};
struct PfWork {
  int a, b, a0, u;   // cut K blocks left [a, b) (a0: where they began), next whole unit
  __device__ __forceinline__ PfWork(const PfParams& p, int pair) : u(pair) {
    a = a0 = pair < p.sk_pairs ? pf_bound(p, pair) : 0;
    b = pair < p.sk_pairs ? pf_bound(p, pair + 1) : 0;
  }
  __device__ __forceinline__ bool next(const PfParams& p, int pairs, PfSeg& s) {
    if (a < b) {
      const int r = a / p.kb_total;
      s.u = p.units + r;
      s.kb0 = a - r * p.kb_total;
      s.kb1 = min(p.kb_total, s.kb0 + b - a);
      s.part = r == a0 / p.kb_total ? 0 : 1;
      a += s.kb1 - s.kb0;
      return true;
    }
    if (u >= p.units) return false;
    s.u = u;
    s.kb0 = 0;
    s.kb1 = p.kb_total;
    s.part = -1;
    u += pairs;
    return true;
  }
};

// First row of the half of weight tile nt that CTA `rank` of the pair loads.
// SwiGLU: CTA 0 the gate rows, CTA 1 the matching up rows (N + f0..).
template <int EPI>
__device__ __forceinline__ int pf_w_row(const PfParams& p, int nt, uint32_t rank) {
  return EPI == EPI_SWIGLU ? (int)rank * p.N + nt * 128 : nt * 256 + (int)rank * 128;
}

// ---------------------------------------------------------------------------
// Epilogues.  A warp takes 32 rows x 128 columns of the accumulator (columns
// half * 128.., SwiGLU: gate columns half * 64.. and the matching up columns)
// in mma-fragment form: thread t holds 2 neighbouring columns of rows t / 4
// (+ 8, 16, 24), so that four threads read or write 32 contiguous bytes of an
// fp32 row (16 bytes of a bf16 row, 32 after st_bf16_pair's exchange) and a
// warp's access touches 8 whole sectors.  One row per thread touches 32
// sectors for 16 bytes each: 25 us for a 256 x 256 tile's residual epilogue,
// more than the tile's MMAs at K = 4096.
// ---------------------------------------------------------------------------
// Parts of cut units.  A part is stored as the epilogue threads hold it: blocks
// of 16 rows x 64 columns, 8 float4 per thread, a warp's 32 threads side by side.
__device__ __forceinline__ size_t pf_slot(int pair, int part, uint32_t rank) {
  return ((size_t)(pair * 2 + part) * 2 + rank) * (32 * 8 * 32);   // float4
}
__device__ __forceinline__ size_t pf_block(int q, int h16, int col) {
  return (size_t)((q * 2 + h16) * 4 + (col >> 6)) * (8 * 32);
}

// Stages this warp's accumulators (rows of its quarter at ta, its half of the
// columns).
__device__ __noinline__ void pf_stage(float4* slot, uint32_t ta, int q, int half, int lane) {
#pragma unroll 1
  for (int h16 = 0; h16 < 2; ++h16)
#pragma unroll 1
    for (int c = half * 128; c < half * 128 + 128; c += 64) {
      uint32_t r[32];
      ptx::tmem_ld_frag<8>(ta + c + ((uint32_t)(h16 * 16) << 16), r);
      ptx::tmem_wait_ld();
      float4* d = slot + pf_block(q, h16, c) + lane;
#pragma unroll
      for (int k = 0; k < 8; ++k)
        __stcg(d + k * 32, make_float4(__uint_as_float(r[4 * k]), __uint_as_float(r[4 * k + 1]),
                                       __uint_as_float(r[4 * k + 2]), __uint_as_float(r[4 * k + 3])));
    }
}

// The sum of the parts that pairs i0 .. i1 staged (part s0 of pair i0, part 0 of
// the others), in that order, back into the accumulator; two parts' loads in
// flight (four spill the kernel's registers, which costs every launch more than
// the shorter sums give).
__device__ __noinline__ void pf_gather(const float4* ws, int i0, int i1, int s0, uint32_t rank, uint32_t ta, int q,
                                          int half, int lane) {
#pragma unroll 1
  for (int h16 = 0; h16 < 2; ++h16)
#pragma unroll 1
    for (int c = half * 128; c < half * 128 + 128; c += 64) {
      const float4* base = ws + pf_block(q, h16, c) + lane;
      float4 v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
      for (int i = i0; i <= i1; i += 2) {
        float4 x[8], y[8];
        const float4* bx = base + pf_slot(i, i == i0 ? s0 : 0, rank);
        const float4* by = base + pf_slot(i + 1, 0, rank);
        const bool two = i < i1;
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = __ldcg(bx + k * 32);
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if (two) y[k] = __ldcg(by + k * 32);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          v[k].x += x[k].x;
          v[k].y += x[k].y;
          v[k].z += x[k].z;
          v[k].w += x[k].w;
        }
        if (two) {
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            v[k].x += y[k].x;
            v[k].y += y[k].y;
            v[k].z += y[k].z;
            v[k].w += y[k].w;
          }
        }
      }
      uint32_t r[32];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        r[4 * k] = __float_as_uint(v[k].x);
        r[4 * k + 1] = __float_as_uint(v[k].y);
        r[4 * k + 2] = __float_as_uint(v[k].z);
        r[4 * k + 3] = __float_as_uint(v[k].w);
      }
      ptx::tmem_st_frag8(ta + c + ((uint32_t)(h16 * 16) << 16), r);
    }
  ptx::tmem_wait_st();
}

__device__ __forceinline__ uint32_t pf_pack(float a, float b) {
  return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(a)) |
         ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(b)) << 16);
}
__device__ __forceinline__ float pf_rest(float a) { return a - __bfloat162float(__float2bfloat16_rn(a)); }

// Stores this thread's bf16 pairs of column groups g and g + 1 (8 columns
// each) of one row: neighbouring threads exchange a pair, the even one stores
// 4 columns of group g, the odd one 4 of group g + 1.  `row` points at column 0
// of group g; all threads of the warp call, `ok` says which groups are stored.
__device__ __forceinline__ void st_bf16_pair(bf16* row, uint32_t wg, uint32_t wg1, bool ok, bool ok1, int lane) {
  const bool odd = lane & 1;
  const uint32_t got = __shfl_xor_sync(0xffffffffu, odd ? wg : wg1, 1);
  const uint2 v = odd ? make_uint2(got, wg1) : make_uint2(wg, got);
  if (odd ? ok1 : ok) *reinterpret_cast<uint2*>(row + (odd ? 8 : 0) + (lane & 2) * 2) = v;
}

__device__ __forceinline__ void pf_resid(const PfParams& p, int j0, int nt, int half, uint32_t ta, int lane) {
  const int gr = lane >> 2, tc = (lane & 3) * 2;
#pragma unroll 1
  for (int x = 0; x < 4; ++x) {
    const int h16 = x >> 1, c0 = half * 128 + (x & 1) * 64;
    const int n0 = nt * 256 + c0;
    if (n0 >= p.N) continue;   // N is a multiple of 64
    bool live[2];
    size_t at[2];
    float2 s[8][2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int j = j0 + h16 * 16 + gr + 8 * i;
      live[i] = j < p.m;
      at[i] = (size_t)(live[i] ? (p.rows ? p.rows[j] : j) : 0) * p.N + n0 + tc;
#pragma unroll
      for (int g = 0; g < 8; ++g)
        if (live[i]) s[g][i] = *reinterpret_cast<const float2*>(p.resid_src + at[i] + 8 * g);
    }
    __syncwarp();
    uint32_t v[32];
    ptx::tmem_ld_frag<8>(ta + c0 + ((uint32_t)(h16 * 16) << 16), v);
    ptx::tmem_wait_ld();
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int g = 0; g < 8; ++g)
        if (live[i])
          *reinterpret_cast<float2*>(p.resid_dst + at[i] + 8 * g) =
              make_float2(s[g][i].x + __uint_as_float(v[4 * g + 2 * i]),
                          s[g][i].y + __uint_as_float(v[4 * g + 2 * i + 1]));
    __syncwarp();
  }
}

template <bool SPLIT>
__device__ __forceinline__ void pf_swiglu(const PfParams& p, int j0, int nt, int half, uint32_t ta, int lane) {
  const int gr = lane >> 2;
  const int f0 = nt * 128 + half * 64;
#pragma unroll 1
  for (int h16 = 0; h16 < 2; ++h16) {
    uint32_t g_[32], u_[32];
    const uint32_t t16 = ta + ((uint32_t)(h16 * 16) << 16);
    ptx::tmem_ld_frag<8>(t16 + half * 64, g_);
    ptx::tmem_ld_frag<8>(t16 + 128 + half * 64, u_);
    ptx::tmem_wait_ld();
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int j = j0 + h16 * 16 + gr + 8 * i;
      const bool live = j < p.m;
      const size_t at = (size_t)j * p.N + f0;
#pragma unroll
      for (int g = 0; g < 8; g += 2) {
        float a[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int k = 4 * (g + (e >> 1)) + 2 * i + (e & 1);
          a[e] = silu_f(__uint_as_float(g_[k])) * __uint_as_float(u_[k]);
        }
        const bool ok = live && f0 + 8 * g < p.N, ok1 = live && f0 + 8 * g + 8 < p.N;   // N is a multiple of 8
        st_bf16_pair(p.out_act + at + 8 * g, pf_pack(a[0], a[1]), pf_pack(a[2], a[3]), ok, ok1, lane);
        if (SPLIT)
          st_bf16_pair(p.out_act_lo + at + 8 * g, pf_pack(pf_rest(a[0]), pf_rest(a[1])),
                       pf_pack(pf_rest(a[2]), pf_rest(a[3])), ok, ok1, lane);
      }
    }
  }
}

// QKV: the tile's 256 columns are 256 / HD whole heads; bias, rotate-half RoPE
// at the token's position (pairs e, e + HD/2), q out in fp32, K/V stored (bf16)
// at the token's position in the layer's cache.
template <int HD>
__device__ __forceinline__ void pf_qkv(const PfParams& p, int j0, int nt, int half, uint32_t ta, int lane) {
  constexpr int HH = HD / 2, G = HH / 8;
  const int gr = lane >> 2, tc = (lane & 3) * 2;
  int seq[4], pos[4], cpos[4];
  bool live[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int j = j0 + gr + 8 * i;
    live[i] = j < p.m;
    const int row = live[i] ? (p.rows ? p.rows[j] : j) : 0;
    seq[i] = p.tok_seq[row];
    pos[i] = p.tok_pos[row];
    cpos[i] = p.cache_len[seq[i]] + (pos[i] - p.len[seq[i]]);
  }
#pragma unroll 1
  for (int cb = half * 128; cb < half * 128 + 128; cb += HD) {
    const int n0 = nt * 256 + cb;   // first feature of this head
    if (n0 >= p.N) break;
    const int head = n0 / HD;
#pragma unroll
    for (int h16 = 0; h16 < 2; ++h16) {
      __syncwarp();
      uint32_t a_[4 * G], b_[4 * G];
      const uint32_t t16 = ta + cb + ((uint32_t)(h16 * 16) << 16);
      ptx::tmem_ld_frag<G>(t16, a_);
      ptx::tmem_ld_frag<G>(t16 + HH, b_);
      ptx::tmem_wait_ld();
      float x[4 * G], y[4 * G];   // columns e and e + HD/2
#pragma unroll
      for (int g = 0; g < G; ++g) {
        float ba[2] = {0.f, 0.f}, bb[2] = {0.f, 0.f};   // scalar loads: the bias may be 4-byte aligned
        if (p.bias) {
          const float* b = p.bias + n0 + 8 * g + tc;
          ba[0] = b[0];
          ba[1] = b[1];
          bb[0] = b[HH];
          bb[1] = b[HH + 1];
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int k = 4 * g + 2 * i;
          x[k] = __uint_as_float(a_[k]) + ba[0];
          x[k + 1] = __uint_as_float(a_[k + 1]) + ba[1];
          y[k] = __uint_as_float(b_[k]) + bb[0];
          y[k + 1] = __uint_as_float(b_[k + 1]) + bb[1];
        }
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int r = 2 * h16 + i;
        if (head < p.nq + p.nkv) {
          const float* co = p.rope_cos + (size_t)pos[r] * HH + tc;
          const float* si = p.rope_sin + (size_t)pos[r] * HH + tc;
#pragma unroll
          for (int g = 0; g < G; ++g) {
            const float2 c2 = *reinterpret_cast<const float2*>(co + 8 * g);
            const float2 s2 = *reinterpret_cast<const float2*>(si + 8 * g);
            const int k = 4 * g + 2 * i;
            const float u0 = x[k], v0 = y[k], u1 = x[k + 1], v1 = y[k + 1];
            x[k] = u0 * c2.x - v0 * s2.x;
            y[k] = v0 * c2.x + u0 * s2.x;
            x[k + 1] = u1 * c2.y - v1 * s2.y;
            y[k + 1] = v1 * c2.y + u1 * s2.y;
          }
        }
        if (head < p.nq) {
          if (live[r]) {
            float* q = p.q_out + (size_t)(j0 + gr + 8 * r) * p.nq * HD + (size_t)head * HD + tc;
#pragma unroll
            for (int g = 0; g < G; ++g) {
              const int k = 4 * g + 2 * i;
              *reinterpret_cast<float2*>(q + 8 * g) = make_float2(x[k], x[k + 1]);
              *reinterpret_cast<float2*>(q + HH + 8 * g) = make_float2(y[k], y[k + 1]);
            }
          }
        } else {
          const bool isk = head < p.nq + p.nkv;
          bf16* c = (isk ? p.kc : p.vc) + kv_offset(p.seq_off, p.cap, seq[r], p.nkv, HD,
                                                    head - p.nq - (isk ? 0 : p.nkv), cpos[r]);
#pragma unroll
          for (int g = 0; g < G; g += 2) {
            const int k = 4 * g + 2 * i;
            st_bf16_pair(c + 8 * g, pf_pack(x[k], x[k + 1]), pf_pack(x[k + 4], x[k + 5]), live[r], live[r], lane);
            st_bf16_pair(c + HH + 8 * g, pf_pack(y[k], y[k + 1]), pf_pack(y[k + 4], y[k + 5]), live[r], live[r],
                         lane);
          }
        }
      }
    }
  }
}

// Epilogue of rows j0 .. j0 + 31 (this warp's quarter) of unit tile nt, one half
// of its columns.
template <int EPI, bool SPLIT>
__device__ __forceinline__ void pf_epilogue(const PfParams& p, int j0, int nt, int half, uint32_t ta, int lane) {
  if (EPI == EPI_RESID) pf_resid(p, j0, nt, half, ta, lane);
  else if (EPI == EPI_SWIGLU) pf_swiglu<SPLIT>(p, j0, nt, half, ta, lane);
  else if (p.hd == 128) pf_qkv<128>(p, j0, nt, half, ta, lane);
  else pf_qkv<64>(p, j0, nt, half, ta, lane);
}

// Whether `v` holds for any thread of the epilogue warps (a barrier for them).
__device__ __forceinline__ bool pf_epi_any(bool v) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.or.pred q, 1, %2, p;\n"
      " selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)v), "n"(32 * kPfEpiWarps)
      : "memory");
  return r != 0;
}

template <int EPI, bool SPLIT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPfThreads, 1)
    gemm_pf_kernel(const __grid_constant__ CUtensorMap tw, const __grid_constant__ CUtensorMap tx,
                   const __grid_constant__ CUtensorMap txlo, const PfParams p) {
  extern __shared__ uint8_t smem_raw[];
  // full, tempty and done are CTA 0's (its copies in CTA 1 stay unused);
  // empty and tfull exist in both CTAs and are signalled together
  __shared__ __align__(8) uint64_t full_bar[kPfMaxStages], empty_bar[kPfMaxStages];
  __shared__ __align__(8) uint64_t tfull_bar[2], tempty_bar[2], done_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_flag;
  __shared__ int issued_of[2];   // CTA 0: stages each CTA loaded
  __shared__ int last_part;      // the part just staged completed its unit

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = ptx::cluster_rank();
  const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  // The call's first kernel wrote the abort word: it completed before the
  // preceding kernel let this one launch, and both CTAs read the same.
  if (call_aborted(p.status)) {
    pdl_wait();
    return;
  }

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      ptx::mbar_init(&full_bar[s], 2);   // one expect_tx arrival per CTA
      ptx::mbar_init(&empty_bar[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      ptx::mbar_init(&tfull_bar[a], 1);
      ptx::mbar_init(&tempty_bar[a], 2 * kPfEpiWarps);   // the epilogue warps of both CTAs
    }
    ptx::mbar_init(&done_bar, 1);
    abort_flag = 0;
    ptx::fence_mbar_init();
    ptx::tma_prefetch_desc(&tw);
    ptx::tma_prefetch_desc(&tx);
    if (SPLIT) ptx::tma_prefetch_desc(&txlo);
  }
  if (warp == 1) ptx::tmem_alloc_pair(&tmem_slot, 512);
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync();   // both CTAs' barriers are initialised
  ptx::tc_fence_after();
  const uint32_t tmem_base = tmem_slot;

  int consumed = 0;   // CTA 0, MMA warp: stages waited for
  if (warp == 0) {
    // ------------------------------------------------------------------ TMA
    // The first ring of weight tiles, which no earlier kernel writes, is on its
    // way before the dependency wait.
    int pre = 0;
    {
      PfWork work(p, pair);
      PfSeg sg;
      while (pre < p.stages && work.next(p, pairs, sg)) {
        int mt, nt;
        pf_unit(p, sg.u, mt, nt);
        const int wrow = pf_w_row<EPI>(p, nt, rank);
        for (int kb = sg.kb0; kb < sg.kb1 && pre < p.stages; ++kb, ++pre) {
          const uint32_t bar = ptx::dsmem_addr(&full_bar[pre], 0);
          if (ptx::elect_one()) {
            ptx::mbar_expect_tx_cluster(bar, kPfTileBytes);
            ptx::tma_load_2d_pair(smem + (size_t)pre * p.stage_bytes + p.w_off, &tw, bar, kb * kTileK, wrow);
          }
          __syncwarp();
        }
      }
    }
    pdl_wait();
    pdl_trigger();
    constexpr uint32_t x_bytes = (SPLIT ? 2u : 1u) * kPfTileBytes;
    int stage = 0;
    uint32_t ph = 0;
    int issued = 0;
    bool ok = true;
    PfWork work(p, pair);
    PfSeg sg;
    while (ok && work.next(p, pairs, sg)) {
      int mt, nt;
      pf_unit(p, sg.u, mt, nt);
      const int xrow = mt * 256 + (int)rank * 128, wrow = pf_w_row<EPI>(p, nt, rank);
      for (int kb = sg.kb0; kb < sg.kb1; ++kb) {
        const bool have_w = issued < pre;
        if (!have_w) {
          ok = __all_sync(0xffffffffu, ptx::mbar_wait_bounded(&empty_bar[stage], ph ^ 1u, p.wait_ns, &abort_flag));
          if (!ok) break;
        }
        uint8_t* st = smem + (size_t)stage * p.stage_bytes;
        const uint32_t bar = ptx::dsmem_addr(&full_bar[stage], 0);
        if (ptx::elect_one()) {
          ptx::mbar_arrive_expect_tx_cluster(bar, x_bytes + (have_w ? 0u : kPfTileBytes));
          ptx::tma_load_2d_pair(st, &tx, bar, kb * kTileK, xrow);
          if (SPLIT) ptx::tma_load_2d_pair(st + kPfTileBytes, &txlo, bar, kb * kTileK, xrow);
          if (!have_w) ptx::tma_load_2d_pair(st + p.w_off, &tw, bar, kb * kTileK, wrow);
        }
        __syncwarp();
        ++issued;
        if (++stage == p.stages) {
          stage = 0;
          ph ^= 1u;
        }
      }
    }
    if (lane == 0)
      asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(ptx::dsmem_addr(&issued_of[rank], 0)), "r"(issued)
                   : "memory");
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------- MMA (CTA 0 only)
    pdl_wait();
    if (rank == 0) {
      const uint32_t idesc = ptx::idesc_bf16(256u, 256u);
      int stage = 0;
      uint32_t ph = 0;
      int acc = 0;
      uint32_t acc_ph = 0;
      bool ok = true;
      PfWork work(p, pair);
      PfSeg sg;
      while (ok && work.next(p, pairs, sg)) {
        ok = __all_sync(0xffffffffu,
                        ptx::mbar_wait_bounded<true>(&tempty_bar[acc], acc_ph ^ 1u, p.wait_ns, &abort_flag));
        if (!ok) break;
        ptx::tc_fence_after();
        const uint32_t d = tmem_base + (uint32_t)acc * 256u;
        for (int kb = sg.kb0; kb < sg.kb1; ++kb) {
          ok = __all_sync(0xffffffffu, ptx::mbar_wait_bounded(&full_bar[stage], ph, p.wait_ns, &abort_flag));
          if (!ok) break;
          ++consumed;
          ptx::tc_fence_after();
          const uint8_t* st = smem + (size_t)stage * p.stage_bytes;
          const uint64_t da = ptx::smem_desc_sw128(st);
          const uint64_t dl = ptx::smem_desc_sw128(st + kPfTileBytes);
          const uint64_t dw = ptx::smem_desc_sw128(st + p.w_off);
          if (ptx::elect_one()) {
#pragma unroll
            for (int k = 0; k < kTileK / 16; ++k) {
              ptx::mma_bf16_pair(d, da + 2ull * k, dw + 2ull * k, idesc, (kb > sg.kb0 || k > 0) ? 1u : 0u);
              if (SPLIT) ptx::mma_bf16_pair(d, dl + 2ull * k, dw + 2ull * k, idesc, 1u);
            }
            ptx::mma_commit_pair(&empty_bar[stage]);
            if (kb + 1 == sg.kb1) ptx::mma_commit_pair(&tfull_bar[acc]);
          }
          __syncwarp();
          if (++stage == p.stages) {
            stage = 0;
            ph ^= 1u;
          }
        }
        acc ^= 1;
        if (acc == 0) acc_ph ^= 1u;
      }
      // all issued MMAs complete before TMEM is released and CTA 1 may leave
      if (ptx::elect_one()) ptx::mma_commit_pair(&done_bar);
      __syncwarp();
      volatile int dummy = 0;
      ptx::mbar_wait_bounded(&done_bar, 0, kWaitLimitNs, &dummy);
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------- epilogue
    const int q = warp & 3;            // TMEM lane quarter this warp may access
    const int half = (warp - 2) >> 2;  // columns it takes
    pdl_wait();
    int acc = 0;
    uint32_t acc_ph = 0;
    PfWork work(p, pair);
    PfSeg sg;
    while (work.next(p, pairs, sg)) {
      const bool ok = ptx::mbar_wait_bounded(&tfull_bar[acc], acc_ph, p.wait_ns, &abort_flag);
      if (pf_epi_any(!ok)) break;
      ptx::tc_fence_after();
      int mt, nt;
      pf_unit(p, sg.u, mt, nt);
      const int j0 = mt * 256 + (int)rank * 128 + q * 32;
      const uint32_t ta = tmem_base + (uint32_t)acc * 256u + ((uint32_t)(q * 32) << 16);
      bool finish = true;
      if (sg.kb1 - sg.kb0 < p.kb_total) {   // a part of a cut unit
        const bool any = j0 < p.m;   // rows past the last token are neither staged nor summed
        if (any) pf_stage(p.ws + pf_slot(pair, sg.part, rank), ta, q, half, lane);
        pf_epi_any(false);   // every thread's part is stored before the arrival is counted
        const int r = sg.u - p.units;
        if (threadIdx.x == 64) {
          int32_t* ctr = p.ctr + r * 2 + rank;
          const int had = ptx::atom_add_acq_rel(ctr, sg.kb1 - sg.kb0);
          last_part = had + sg.kb1 - sg.kb0 == p.kb_total;
          if (last_part) *ctr = 0;   // re-armed for a later launch
        }
        pf_epi_any(false);
        finish = last_part;
        if (finish) {
          // the pairs whose shares meet this unit
          const int k0 = r * p.kb_total, k1 = k0 + p.kb_total;
          int i0 = min(p.sk_pairs - 1, r * p.sk_pairs / p.sk_units);
          while (i0 > 0 && pf_bound(p, i0) > k0) --i0;
          while (i0 + 1 < p.sk_pairs && pf_bound(p, i0 + 1) <= k0) ++i0;
          int i1 = i0;
          while (i1 + 1 < p.sk_pairs && pf_bound(p, i1 + 1) < k1) ++i1;
          if (any) pf_gather(p.ws, i0, i1, pf_bound(p, i0) < k0 ? 1 : 0, rank, ta, q, half, lane);
          ptx::tc_fence_before();
          pf_epi_any(false);   // SwiGLU reads columns that the other warp of the quarter gathered
          ptx::tc_fence_after();
        }
      }
      if (finish) pf_epilogue<EPI, SPLIT>(p, j0, nt, half, ta, lane);
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive_cluster(ptx::dsmem_addr(&tempty_bar[acc], 0));
      acc ^= 1;
      if (acc == 0) acc_ph ^= 1u;
    }
  }

  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync();   // neither CTA loads, multiplies or drains any more
  ptx::tc_fence_after();
  if (rank == 0 && threadIdx.x == 32) {
    // Never leave with copies in flight: after a wait that ran out, stages may
    // have been loaded that no MMA waited for.  A CTA that did not get to load
    // its part of such a stage is arrived for here.
    for (int it = consumed; it < max(issued_of[0], issued_of[1]); ++it) {
      uint64_t* bar = &full_bar[it % p.stages];
      if (it >= issued_of[0]) ptx::mbar_arrive(bar);
      if (it >= issued_of[1]) ptx::mbar_arrive(bar);
      volatile int dummy = 0;
      ptx::mbar_wait_bounded(bar, (uint32_t)((it / p.stages) & 1), kWaitLimitNs, &dummy);
    }
  }
  if (threadIdx.x == 0 && abort_flag) atomicOr(p.status, BUDDY_DEV_TIMEOUT);
  __syncwarp();
  if (warp == 1) ptx::tmem_dealloc_pair(tmem_base, 512);
  ptx::cluster_sync();   // CTA 1's copies have landed before it leaves
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
int gemm_pf_prepare(Ctx& c) {
  // parts of cut units: two accumulators of 256 x 256 fp32 per pair; arrival
  // counters per cut unit (fewer than pairs) and CTA
  const size_t pairs = c.num_sms / 2;
  if (!c.pf_ws && cudaMalloc(&c.pf_ws, pairs * 2 * 256 * 256 * sizeof(float)) != cudaSuccess) return BUDDY_ERR_CUDA;
  c.pf_ctr_n = (int)pairs * 2;
  if (!c.pf_ctr && cudaMalloc(&c.pf_ctr, c.pf_ctr_n * sizeof(int32_t)) != cudaSuccess) return BUDDY_ERR_CUDA;
  if (cudaMemset(c.pf_ctr, 0, c.pf_ctr_n * sizeof(int32_t)) != cudaSuccess) return BUDDY_ERR_CUDA;
  const int limit = 227 * 1024 - 2 * 1024;
  for (int v = 0; v < 2; ++v) {
    const uint32_t sb = (v ? 3u : 2u) * kPfTileBytes;
    c.pf_stages[v] = std::min(kPfMaxStages, (int)((limit - 1024) / sb));
    c.pf_smem[v] = (int)(c.pf_stages[v] * sb) + 1024;
  }
  const cudaFuncAttribute A = cudaFuncAttributeMaxDynamicSharedMemorySize;
  if (cudaFuncSetAttribute(gemm_pf_kernel<EPI_QKV, false>, A, c.pf_smem[0]) ||
      cudaFuncSetAttribute(gemm_pf_kernel<EPI_RESID, false>, A, c.pf_smem[0]) ||
      cudaFuncSetAttribute(gemm_pf_kernel<EPI_SWIGLU, false>, A, c.pf_smem[0]) ||
      cudaFuncSetAttribute(gemm_pf_kernel<EPI_QKV, true>, A, c.pf_smem[1]) ||
      cudaFuncSetAttribute(gemm_pf_kernel<EPI_RESID, true>, A, c.pf_smem[1]) ||
      cudaFuncSetAttribute(gemm_pf_kernel<EPI_SWIGLU, true>, A, c.pf_smem[1]))
    return BUDDY_ERR_CUDA;
  return BUDDY_OK;
}

// One prefill projection: `which` names the weight (0 qkv, 1 o, 2 gate_up,
// 3 down) of `layer`; `xi` the prefill activation map (0 normalised input,
// 1 attention output, 2 SwiGLU output); m rows.
int launch_gemm_pf(const Ctx& c, int epi, bool split, int layer, int which, int xi, int m, const PfEpi& e,
                   cudaStream_t s) {
  // Few tokens are bound by the weight stream: the decode GEMM (one CTA per weight
  // tile and K split, a fixup over the whole GPU) beats pairs that each hold an
  // M-tile mostly empty and sum their parts alone: 4 blocks of Llama-3-8B, 61 tokens
  // 594 -> 461 us, 256 tokens 862 -> 802 us; Llama-2-13B, 240 tokens 1097 -> 1041 us.
  // Above 256 rows it has no third M-tile.  The masked variant's cache positions
  // differ by block, which its token tables do not hold.
  if (m <= kPfSmallRows && !c.masked) return launch_gemm_pf_small(c, epi, split, layer, which, xi, m, e, s);
  PfParams p{};
  int N, K, tiles;
  gemm_shape(c, which, &N, &K, &tiles);
  p.N = N;
  p.K = K;
  p.m = m;
  p.n_tiles = tiles;
  p.m_tiles = (m + 255) / 256;
  p.kb_total = (K + kTileK - 1) / kTileK;
  // Whole waves of units, then the rest cut along K where that saves more than
  // staging and summing the parts costs (about 8 us; a K block takes 0.26 us,
  // twice that with SPLIT): R units left for P pairs end a fraction (P - R) / P
  // of a unit's time earlier.  With few units a part is a quarter of a unit (a
  // sum of more parts takes as long as the shorter parts save), else cuts fall on
  // multiples of 4 K blocks.
  const int P = c.num_sms / 2, units = p.n_tiles * p.m_tiles, R = units % P;
  const bool cut = (int64_t)(P - R) * p.kb_total * (split ? 52 : 26) > (int64_t)800 * P;
  p.sk_units = R > 0 && cut ? R : 0;
  p.units = units - p.sk_units;
  if (p.sk_units) {
    const int T = p.sk_units * p.kb_total;
    p.sk_gran = std::max(4, P <= 4 * R ? 4 : (p.kb_total + 3) / 4);
    p.sk_pairs = std::max(1, std::min(P, T / p.sk_gran));
    p.ws = c.pf_ws;
    p.ctr = c.pf_ctr;
  }
  const int v = split ? 1 : 0;
  p.stages = c.pf_stages[v];
  p.stage_bytes = (split ? 3u : 2u) * kPfTileBytes;
  p.w_off = (split ? 2u : 1u) * kPfTileBytes;
  p.rows = e.rows;
  p.resid_src = e.resid_src;
  p.resid_dst = e.resid_dst;
  p.out_act = (bf16*)e.out_act;
  p.out_act_lo = (bf16*)e.out_act_lo;
  p.q_out = e.q_out;
  p.bias = e.bias;
  p.rope_cos = c.rope_cos;
  p.rope_sin = c.rope_sin;
  p.tok_seq = e.tok_seq;
  p.tok_pos = e.tok_pos;
  p.len = e.len;
  p.cache_len = e.cache_len;
  p.seq_off = e.seq_off;
  p.cap = e.cap;
  p.kc = (bf16*)e.kc;
  p.vc = (bf16*)e.vc;
  p.nq = c.nq;
  p.nkv = c.nkv;
  p.hd = c.hd;
  p.status = c.status;
  p.wait_ns = c.wait_ns;
  const CUtensorMap& tw = c.pf_wmaps[(size_t)layer * 4 + which];
  const CUtensorMap& tx = c.pf_xmaps[xi].box[3];
  const CUtensorMap& txlo = c.pf_xmaps[3 + xi].box[3];
  const int grid = 2 * (p.units ? std::min(std::max(p.units, p.sk_pairs), P) : p.sk_pairs);
  const size_t smem = c.pf_smem[v];
  if (split) {
    switch (epi) {
      case EPI_QKV: launch_k(gemm_pf_kernel<EPI_QKV, true>, grid, kPfThreads, smem, s, c.pdl, tw, tx, txlo, p); break;
      case EPI_RESID: launch_k(gemm_pf_kernel<EPI_RESID, true>, grid, kPfThreads, smem, s, c.pdl, tw, tx, txlo, p); break;
      default: launch_k(gemm_pf_kernel<EPI_SWIGLU, true>, grid, kPfThreads, smem, s, c.pdl, tw, tx, txlo, p);
    }
  } else {
    switch (epi) {
      case EPI_QKV: launch_k(gemm_pf_kernel<EPI_QKV, false>, grid, kPfThreads, smem, s, c.pdl, tw, tx, txlo, p); break;
      case EPI_RESID: launch_k(gemm_pf_kernel<EPI_RESID, false>, grid, kPfThreads, smem, s, c.pdl, tw, tx, txlo, p); break;
      default: launch_k(gemm_pf_kernel<EPI_SWIGLU, false>, grid, kPfThreads, smem, s, c.pdl, tw, tx, txlo, p);
    }
  }
  return 1;
}

}  // namespace buddy
