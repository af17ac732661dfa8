// Causal attention of a prefill block (App. E, Eq. 9 applied to every prompt
// token): the query of prompt token t of sequence i, at cache position
// c0 + t of the block's cache (c0 = the positions it held before the
// prompt), attends to cache positions 0 .. c0 + t.
//
// The query heads of a KV head share its keys and values, so the rows of a tile
// are (token, head of the group) pairs: row R of a (sequence, KV head) is token
// R / G, head R % G.  A work item is NQ tiles of 128 such rows that walk the
// same key/value tiles of 128 positions: two tiles, or one where the queries
// and probabilities are bf16 hi + lo pairs (SPLIT, the blocks that feed the
// router), whose queries take twice the shared memory.
//
// On the 5th-generation tensor cores:
//   S = Q K^T   tcgen05.mma M = 128, N = 128, K = HD: queries (pre-scaled by
//               log2(e) / sqrt(d_h)) and keys from shared memory, S in TMEM;
//   softmax     four warps per tile, a row per thread: running reference m,
//               p = 2^(s - m) written back as bf16 over S's columns.  m follows
//               the row's maximum only when that rises by more than 8 (p stays
//               below 2^8), so that the output is rescaled a few times per row
//               instead of once per key tile; the final division makes the
//               choice of m immaterial (the online softmax of Milakov and
//               Gimelshein 2018, rescaled late as FlashAttention-4 does);
//   O += P V    M = 128, N = HD, K = 128: P from TMEM, V from shared memory
//               (MN-major), O in TMEM.
// With SPLIT every product is issued for both terms.
//
// Warps: 4 NQ softmax warps, one MMA warp, two copy warps (16-byte cp.async
// into the 128-byte-swizzled layout, two buffers each for K and V; rows past
// the range are zero).  With two tiles the MMAs of one overlap the softmax of
// the other; with one tile S has two buffers and the next S overlaps the
// softmax of this one.  Every wait is bounded.
//
// Bound by the MMA issue (about 100 cycles for the 64 cycles of an N = 128 MMA)
// and the softmax chain.  Two prompts of 2,999 and 5,000 tokens, 28 heads of 128
// over 4 KV heads: 0.28 ms (1.0 PFLOP/s of the visible positions), 0.54 ms with
// SPLIT, against 1.16 and 1.55 ms on mma.sync with 64-row tiles of one head.
#include <cuda_runtime.h>

#include "attn_tc.cuh"
#include "common.cuh"
#include "gemm_common.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace buddy {

constexpr int kPfaRows = 128;    // rows of a tile (MMA M)
constexpr int kPfaKeys = 128;    // positions of a key/value tile
constexpr int kPfaLoadThreads = 64;
constexpr uint32_t kPfaRegion = 128u * 128u;   // 128 rows x 64 channels of bf16

template <bool SPLIT>
__host__ __device__ constexpr int pfa_tiles() { return SPLIT ? 1 : 2; }
template <bool SPLIT>
__host__ __device__ constexpr int pfa_threads() { return 128 * pfa_tiles<SPLIT>() + 32 + kPfaLoadThreads; }
template <int HD, bool SPLIT>
__host__ __device__ constexpr size_t pfa_smem() {
  // queries (hi, and lo with SPLIT), two K and two V buffers, alignment slack
  return (size_t)(HD / 64) * kPfaRegion * (pfa_tiles<SPLIT>() * (SPLIT ? 2 : 1) + 4) + 1024;
}

struct PfaArgs {
  const int4* items;        // (sequence, KV head, first compact row of the sequence, first tile row)
  const int32_t* n_tok;     // sequence -> prompt tokens
  const int32_t* base;      // sequence -> positions the layer's cache held before the prompt
  const float* q;           // [m, nq * hd] compact rows
  const int64_t* seq_off;
  const int32_t* cap;
  const bf16* Kc;
  const bf16* Vc;
  bf16* out;                // [m, nq * hd]
  bf16* out_lo;
  int nq, nkv;
  int32_t* status;
  uint64_t wait_ns;
};

// 16 bytes from global to shared memory, or zeros.
__device__ __forceinline__ void cp_async16_or_zero(uint32_t dst, const void* src, bool real) {
  const uint32_t n = real ? 16u : 0u;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}

// Byte offset of 16-byte piece c of row r in a tile of 64-channel regions
// (128-byte rows, 128-byte swizzle).
__device__ __forceinline__ uint32_t pfa_piece(int r, int c) {
  return (uint32_t)(c >> 3) * kPfaRegion + (uint32_t)r * 128u + (uint32_t)(((c ^ r) & 7) << 4);
}

template <int HD, bool SPLIT>
__global__ void __launch_bounds__(pfa_threads<SPLIT>(), 1) attn_pf_kernel(const PfaArgs A) {
  extern __shared__ uint8_t smem_raw[];
  constexpr int NQ = pfa_tiles<SPLIT>();
  constexpr int V16 = HD / 8;                           // 16-byte pieces per row
  constexpr uint32_t TILE = (HD / 64) * kPfaRegion;     // bytes of a 128-row tile
  // TMEM columns: S slots at 0 and 128 (P over their first half); O of tile q at
  // 256 + 128 q; with SPLIT (one tile) P's remainders of the two slots at 384
  constexpr uint32_t kO = 256, kPLo = 384;
  __shared__ __align__(8) uint64_t q_ready, k_full[2], k_empty[2], v_full[2], v_empty[2];
  __shared__ __align__(8) uint64_t s_full[2], p_ready[2], pv_done, o_full[2], drained;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_flag;
  // (written by the call's first kernel, complete before the preceding kernel let
  // this one launch, as were the items, the token counts and the positions)
  if (call_aborted(A.status)) {
    pdl_wait();
    return;
  }

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sQ = smem;                                   // [tile][hi, lo]
  uint8_t* sK = smem + NQ * (SPLIT ? 2 : 1) * TILE;     // [2]
  uint8_t* sV = sK + 2 * TILE;                          // [2]

  const int4 it = A.items[blockIdx.x];
  const int seq = it.x, g = it.y, row0 = it.w;
  const int G = A.nq / A.nkv;
  const int c0 = A.base[seq];
  const int R = A.n_tok[seq] * G;                       // rows of this (sequence, KV head)
  const int nq = NQ == 2 && R - row0 > kPfaRows ? 2 : 1;   // tiles with rows
  const int last = min(R, row0 + nq * kPfaRows) - 1;
  const int kmax = c0 + last / G + 1;                   // positions the last row sees
  const int n = (kmax + kPfaKeys - 1) / kPfaKeys;

  if (tid == 0) {
    ptx::mbar_init(&q_ready, 128 * nq);
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(&k_full[b], kPfaLoadThreads);
      ptx::mbar_init(&v_full[b], kPfaLoadThreads);
      ptx::mbar_init(&k_empty[b], 1);
      ptx::mbar_init(&v_empty[b], 1);
      ptx::mbar_init(&s_full[b], 1);
      ptx::mbar_init(&p_ready[b], 128);
      ptx::mbar_init(&o_full[b], 1);
    }
    ptx::mbar_init(&pv_done, 1);
    ptx::mbar_init(&drained, 1);
    abort_flag = 0;
    ptx::fence_mbar_init();
  }
  constexpr int kMmaWarp = 4 * NQ;
  if (warp == kMmaWarp) {
    ptx::tmem_alloc(&tmem_slot, 512);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = tmem_slot;
  pdl_wait();   // the queries, keys and values of the preceding kernel
  pdl_trigger();

  if (warp < kMmaWarp) {
    const int q = warp >> 2;                            // this warp's tile
    if (q < nq) {
      // ------------------------------------------------------------- softmax
      const int rt = (warp & 3) * 32 + lane;            // row of the tile
      const int row = min(R - 1, row0 + q * kPfaRows + rt);
      const int t = row / G, h = g * G + row - t * G;
      const size_t at = ((size_t)(it.z + t) * A.nq + h) * HD;
      // The queries of this warp's 32 rows, scaled, as bf16 (hi, lo) in the swizzled
      // K-major layout: the lanes share a row (HD / 4 lanes, 16 bytes each), eight
      // loads in flight.  (A row per lane reads 32 sectors for 16 bytes each: 5 to
      // 7 us of a work item.)
      uint8_t* const qdst = sQ + (size_t)q * (SPLIT ? 2 : 1) * TILE;
      {
        constexpr int LPR = HD / 4, RPL = 32 / LPR;     // lanes per row, rows per load
        const float scale = 1.4426950408889634f * rsqrtf((float)HD);
        const int l4 = lane % LPR;
#pragma unroll 1
        for (int r0 = 0; r0 < 32; r0 += 8 * RPL) {
          float4 v[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const size_t src = __shfl_sync(0xffffffffu, (unsigned long long)at, r0 + u * RPL + lane / LPR);
            v[u] = *reinterpret_cast<const float4*>(A.q + src + l4 * 4);
          }
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int r = (warp & 3) * 32 + r0 + u * RPL + lane / LPR;
            uint32_t hi[2], lo[2];
            tca::split_pack(v[u].x * scale, v[u].y * scale, hi[0], lo[0]);
            tca::split_pack(v[u].z * scale, v[u].w * scale, hi[1], lo[1]);
            uint8_t* d = qdst + pfa_piece(r, l4 >> 1) + (l4 & 1) * 8;
            *reinterpret_cast<uint2*>(d) = make_uint2(hi[0], hi[1]);
            if (SPLIT) *reinterpret_cast<uint2*>(d + TILE) = make_uint2(lo[0], lo[1]);
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        ptx::mbar_arrive(&q_ready);
      }
      const uint32_t tq = tmem + ((uint32_t)((warp & 3) * 32) << 16);
      const uint32_t to = tq + kO + (uint32_t)q * 128u;
      const int seen = c0 + t + 1;                      // positions this row sees
      float m = -INFINITY, l = 0.f;
      bool ok = true;
      for (int j = 0; j < n; ++j) {
        const int slot = NQ == 2 ? q : (j & 1);
        const uint32_t ph = (uint32_t)(NQ == 2 ? j & 1 : (j >> 1) & 1);
        ok = __all_sync(0xffffffffu, ptx::mbar_wait_bounded(&s_full[slot], ph, A.wait_ns, &abort_flag));
        if (!ok) break;
        ptx::tc_fence_after();
        const uint32_t ts = tq + (uint32_t)slot * 128u;
        const int lim = seen - j * kPfaKeys;            // visible columns of this tile (may be <= 0)
        const bool cut = __any_sync(0xffffffffu, lim < kPfaKeys);
        uint32_t s[kPfaKeys];   // the row, read once (P overwrites its columns)
#pragma unroll
        for (int c = 0; c < kPfaKeys; c += 32) ptx::tmem_ld32(ts + c, s + c);
        ptx::tmem_wait_ld();
        if (cut) {
#pragma unroll
          for (int i = 0; i < kPfaKeys; ++i)
            if (i >= lim) s[i] = 0xff800000u;   // -inf: p = 0
        }
        float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int i = 0; i < kPfaKeys; ++i) mx4[i & 3] = fmaxf(mx4[i & 3], __uint_as_float(s[i]));
        const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
        // position 0 is visible to every row: m is finite from tile 0 on
        const bool raise = mx > m + 8.f;
        if (__any_sync(0xffffffffu, raise)) {
          const float al = raise ? tca::exp2a(m - mx) : 1.f;
          if (raise) m = mx;
          l *= al;
          if (j > 0) {
            if (NQ == 1) {   // S of this tile was computed before the previous tile's O += P V ended
              ok = __all_sync(0xffffffffu, ptx::mbar_wait_bounded(&pv_done, (uint32_t)((j - 1) & 1), A.wait_ns,
                                                                  &abort_flag));
              if (!ok) break;
              ptx::tc_fence_after();
            }
#pragma unroll 1
            for (int c = 0; c < HD; c += 32) {
              uint32_t o[32];
              ptx::tmem_ld32(to + c, o);
              ptx::tmem_wait_ld();
#pragma unroll
              for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * al);
              ptx::tmem_st32(to + c, o);
            }
          }
        }
        float ls[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int c = 0; c < kPfaKeys; c += 32) {
          uint32_t hi[16], lo[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float p0 = tca::exp2a(__uint_as_float(s[c + 2 * i]) - m);
            const float p1 = tca::exp2a(__uint_as_float(s[c + 2 * i + 1]) - m);
            ls[i & 3] += p0 + p1;
            if (SPLIT) tca::split_pack(p0, p1, hi[i], lo[i]);
            else hi[i] = tca::pack_bf16(p0, p1);
          }
          ptx::tmem_st16(ts + c / 2, hi);
          if (SPLIT) ptx::tmem_st16(tq + kPLo + (uint32_t)slot * 64u + c / 2, lo);
        }
        l += (ls[0] + ls[1]) + (ls[2] + ls[3]);
        ptx::tmem_wait_st();
        ptx::tc_fence_before();
        ptx::mbar_arrive(&p_ready[slot]);
      }
      if (ok) ok = __all_sync(0xffffffffu, ptx::mbar_wait_bounded(&o_full[q], 0, A.wait_ns, &abort_flag));
      if (ok) {
        ptx::tc_fence_after();
        const float inv = 1.f / l;
        // through this tile's query buffer (its MMAs are done), so that the lanes
        // store whole rows
#pragma unroll 1
        for (int c = 0; c < HD; c += 32) {
          uint32_t o[32];
          ptx::tmem_ld32(to + c, o);
          ptx::tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 32; i += 8) {
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
              tca::split_pack(__uint_as_float(o[i + 2 * e]) * inv, __uint_as_float(o[i + 2 * e + 1]) * inv, hi[e],
                              lo[e]);
            uint8_t* d = qdst + pfa_piece(rt, (c + i) >> 3);
            *reinterpret_cast<uint4*>(d) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
            if (SPLIT) *reinterpret_cast<uint4*>(d + TILE) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
          }
        }
        __syncwarp();
        constexpr int RPS = 32 / V16;                   // rows per store
#pragma unroll 4
        for (int r0 = 0; r0 < 32; r0 += RPS) {
          const int r = r0 + lane / V16, c = lane % V16;
          const size_t dst = __shfl_sync(0xffffffffu, (unsigned long long)at, r) + c * 8;
          const uint8_t* d = qdst + pfa_piece((warp & 3) * 32 + r, c);
          if (row0 + q * kPfaRows + (warp & 3) * 32 + r < R) {
            *reinterpret_cast<uint4*>(A.out + dst) = *reinterpret_cast<const uint4*>(d);
            if (SPLIT) *reinterpret_cast<uint4*>(A.out_lo + dst) = *reinterpret_cast<const uint4*>(d + TILE);
          }
        }
      }
    }
  } else if (warp == kMmaWarp) {
    // -------------------------------------------------------------------- MMA
    if (lane == 0) {
      const uint32_t id_s = ptx::idesc_bf16(128u, (uint32_t)kPfaKeys);
      const uint32_t id_o = ptx::idesc_bf16(128u, (uint32_t)HD) | ptx::kIdescBMnMajor;
      auto wait = [&](uint64_t* bar, int phase) {
        return ptx::mbar_wait_bounded(bar, (uint32_t)(phase & 1), A.wait_ns, &abort_flag);
      };
      auto qk = [&](int q, int slot, int j) {   // S slot = Q_q K_j^T
        const uint8_t* Q = sQ + (size_t)q * (SPLIT ? 2 : 1) * TILE;
        const uint8_t* K = sK + (size_t)(j & 1) * TILE;
#pragma unroll
        for (int k = 0; k < HD / 16; ++k) {
          const uint64_t dk = ptx::smem_desc_sw128(K + (k >> 2) * kPfaRegion) + 2ull * (k & 3);
          const uint64_t dq = ptx::smem_desc_sw128(Q + (k >> 2) * kPfaRegion) + 2ull * (k & 3);
          ptx::mma_bf16(tmem + (uint32_t)slot * 128u, dq, dk, id_s, k > 0 ? 1u : 0u);
          if (SPLIT) {
            const uint64_t dl = ptx::smem_desc_sw128(Q + TILE + (k >> 2) * kPfaRegion) + 2ull * (k & 3);
            ptx::mma_bf16(tmem + (uint32_t)slot * 128u, dl, dk, id_s, 1u);
          }
        }
        ptx::mma_commit(&s_full[slot]);
      };
      auto pv = [&](int q, int slot, int j) {   // O_q += P V_j
        const uint8_t* V = sV + (size_t)(j & 1) * TILE;
        const uint32_t d = tmem + kO + (uint32_t)q * 128u, a = tmem + (uint32_t)slot * 128u;
#pragma unroll
        for (int k = 0; k < kPfaKeys / 16; ++k) {
          const uint64_t dv = ptx::smem_desc_sw128_mn(V + k * 2048, kPfaRegion);   // 16 positions: two 1 KiB groups
          ptx::mma_bf16_ts(d, a + 8u * k, dv, id_o, (j > 0 || k > 0) ? 1u : 0u);
          if (SPLIT) ptx::mma_bf16_ts(d, tmem + kPLo + (uint32_t)slot * 64u + 8u * k, dv, id_o, 1u);
        }
      };
      bool ok = wait(&q_ready, 0) && wait(&k_full[0], 0);
      if (ok) {
        ptx::tc_fence_after();
        for (int q = 0; q < nq; ++q) qk(q, q, 0);
        ptx::mma_commit(&k_empty[0]);
      }
      for (int j = 0; j < n && ok; ++j) {
        const bool more = j + 1 < n;
        if (NQ == 2) {
          for (int q = 0; q < nq && ok; ++q) {
            ok = wait(&p_ready[q], j) && (q > 0 || wait(&v_full[j & 1], j >> 1)) &&
                 (q > 0 || !more || wait(&k_full[(j + 1) & 1], (j + 1) >> 1));
            if (!ok) break;
            ptx::tc_fence_after();
            pv(q, q, j);
            if (q == nq - 1) ptx::mma_commit(&v_empty[j & 1]);
            if (more) {
              qk(q, q, j + 1);   // in issue order after the P V that reads P from the same columns
              if (q == nq - 1) ptx::mma_commit(&k_empty[(j + 1) & 1]);
            } else {
              ptx::mma_commit(&o_full[q]);
            }
          }
        } else {
          if (more) {
            ok = wait(&k_full[(j + 1) & 1], (j + 1) >> 1);
            if (!ok) break;
            ptx::tc_fence_after();
            qk(0, (j + 1) & 1, j + 1);
            ptx::mma_commit(&k_empty[(j + 1) & 1]);
          }
          ok = wait(&p_ready[j & 1], j >> 1) && wait(&v_full[j & 1], j >> 1);
          if (!ok) break;
          ptx::tc_fence_after();
          pv(0, j & 1, j);
          ptx::mma_commit(&v_empty[j & 1]);
          ptx::mma_commit(more ? &pv_done : &o_full[0]);
        }
      }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------ K, V copies
    const int lt = tid - 32 * (kMmaWarp + 1);
    const int64_t kvbase = (A.seq_off[seq] * A.nkv + (int64_t)g * A.cap[seq]) * HD;
    constexpr int RPI = kPfaLoadThreads / V16;   // rows per round
    const int c = lt % V16, r0 = lt / V16;
    auto copy = [&](uint8_t* dst, const bf16* src, int j) {
      const int p0 = j * kPfaKeys;
      const uint32_t d = ptx::smem_u32(dst);
      const bf16* s = src + kvbase + (int64_t)p0 * HD + c * 8;
#pragma unroll 8
      for (int r = r0; r < kPfaKeys; r += RPI) {
        const bool real = p0 + r < kmax;
        cp_async16_or_zero(d + pfa_piece(r, c), real ? s + (int64_t)r * HD : A.Kc, real);
      }
      cp_async_commit();
    };
    // loads K0 V0 K1 V1 ..: a load is announced once the next one is issued
    uint64_t* pending = nullptr;
    bool ok = true;
    for (int x = 0; x < 2 * n && ok; ++x) {
      const int j = x >> 1, b = j & 1;
      const bool isk = (x & 1) == 0;
      ok = ptx::mbar_wait_bounded(isk ? &k_empty[b] : &v_empty[b], (uint32_t)(((j >> 1) & 1) ^ 1), A.wait_ns,
                                  &abort_flag);
      if (!ok) break;
      copy((isk ? sK : sV) + (size_t)b * TILE, isk ? A.Kc : A.Vc, j);
      if (pending) {
        cp_async_wait<1>();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        ptx::mbar_arrive(pending);
      }
      pending = isk ? &k_full[b] : &v_full[b];
    }
    cp_async_wait<0>();
    if (ok && pending) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      ptx::mbar_arrive(pending);
    }
  }

  // every issued MMA completes before TMEM is freed: normally all have (o_full),
  // after a wait that ran out the MMA warp waits for its own
  __syncthreads();
  if (warp == kMmaWarp) {
    if (abort_flag) {
      if (lane == 0) {
        ptx::mma_commit(&drained);
        volatile int dummy = 0;
        ptx::mbar_wait_bounded(&drained, 0, kWaitLimitNs, &dummy);
        atomicOr(A.status, BUDDY_DEV_TIMEOUT);
      }
      __syncwarp();
    }
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, 512);
  }
}

template <int HD, bool SPLIT>
static int pfa_prepare() {
  return cudaFuncSetAttribute(attn_pf_kernel<HD, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)pfa_smem<HD, SPLIT>()) == cudaSuccess
             ? BUDDY_OK
             : BUDDY_ERR_CUDA;
}
int attention_pf_prepare(const Ctx& c) {
  const int a = c.hd == 128 ? pfa_prepare<128, false>() : pfa_prepare<64, false>();
  return a != BUDDY_OK ? a : (c.hd == 128 ? pfa_prepare<128, true>() : pfa_prepare<64, true>());
}

// Rows (tokens x heads of a group) of one work item.
int attention_pf_rows(bool split) { return kPfaRows * (split ? pfa_tiles<true>() : pfa_tiles<false>()); }

template <int HD, bool SPLIT>
static void pfa_launch(const PfaArgs& A, int n_items, bool pdl, cudaStream_t s) {
  launch_k(attn_pf_kernel<HD, SPLIT>, n_items, pfa_threads<SPLIT>(), pfa_smem<HD, SPLIT>(), s, pdl, A);
}

void launch_attention_pf(const Ctx& c, int n_items, const int4* items, const int32_t* n_tok, const int32_t* base,
                         const buddy_kv_state& kv, int layer, const float* q, void* out, void* out_lo,
                         cudaStream_t s) {
  const PfaArgs A{items, n_tok, base, q, kv.seq_off, kv.cap, (const bf16*)kv.k_cache[layer],
                  (const bf16*)kv.v_cache[layer], (bf16*)out, (bf16*)out_lo, c.nq, c.nkv, c.status, c.wait_ns};
  if (c.hd == 128) {
    if (out_lo) pfa_launch<128, true>(A, n_items, c.pdl, s);
    else pfa_launch<128, false>(A, n_items, c.pdl, s);
  } else {
    if (out_lo) pfa_launch<64, true>(A, n_items, c.pdl, s);
    else pfa_launch<64, false>(A, n_items, c.pdl, s);
  }
}

}  // namespace buddy
