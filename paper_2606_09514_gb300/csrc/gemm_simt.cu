// CUDA-core GEMMs of the fp32 decode projections: C[j][n] = sum_k X[j][k] W[n][k]
// (X active rows, W in nn.Linear layout), fp32 throughout (tensor cores would
// round the operands).
//
// Up to kSimtFuseRows rows (gemm_simt_kernel) the step is a chain of small
// dependent kernels, so the GEMMs take in their neighbours: one warp per output
// unit (a weight row, the gate/up row pair of SwiGLU, or a rotate-half row pair of
// QKV), rows four or eight at a time; the QKV and gate/up GEMMs sum the squares
// of their input rows beside the products and scale the result by 1 / rms (no
// RMSNorm kernel), and the QKV GEMM adds the bias, rotates and stores q, K and V
// (no finalisation kernel).  Five kernels per block instead of eight: an 8-block
// model of width 256 decodes 4 rows in 149 us against 190 us.  The first weights
// load before the dependency wait.
//
// Above that (gemm_simt_tiled_kernel) tiles of 32 rows x 32 weight rows, K in
// steps of 32 through a four-stage cp.async ring: the weights are read once per 32
// rows, not once per four.  5 blocks of width 256, 200 rows: 546 us a step against
// 2094 us.  The line lies where the two meet: 25 rows take 286 us fused and 300 us
// tiled, 28 rows 312 and 318 us, 32 rows 328 and 318 us.
#include <cuda_runtime.h>

#include "attn_common.cuh"
#include "common.cuh"
#include "internal.h"

namespace buddy {

// The QKV epilogue's pointers, as in the tensor-core GEMM.
struct SimtArgs {
  const float* W;
  const float* X;           // [m, K] compact rows, or with nsrc:
  const float* nsrc;        // rows nsrc[rows[j]], scaled by 1 / rms and gamma
  const float* gamma;
  float eps;
  int N, K;                 // output units of the GEMM (QKV: q, k and v features)
  const int32_t* rows;
  const int32_t* count;
  int n;
  float* out;               // EPI_STORE_F32: [m, N]; EPI_SWIGLU: [m, N]
  const float* resid_src;
  float* resid_dst;
  const float* bias;
  const float* rope_cos;
  const float* rope_sin;
  const int32_t* len;
  const int32_t* cache_len;
  const int64_t* seq_off;
  const int32_t* cap;
  float* kc;
  float* vc;
  float* q_out;
  float* pool;
  int nq, nkv, hd;
  const int32_t* status;
};

// q, K or V features (head, e) = v0 and (head, e + hd/2) = v1 of row j.
__device__ __forceinline__ void simt_qkv(const SimtArgs& p, int j, int head, int e, float v0, float v1) {
  const int half = p.hd >> 1, c0 = head * p.hd + e;
  const int i = p.rows ? p.rows[j] : j;
  if (p.bias) {
    v0 += p.bias[c0];
    v1 += p.bias[c0 + half];
  }
  if (head < p.nq + p.nkv) {
    const int pos = p.len[i];
    const float co = p.rope_cos[(size_t)pos * half + e], si = p.rope_sin[(size_t)pos * half + e];
    const float y0 = v0 * co - v1 * si, y1 = v1 * co + v0 * si;
    float* d = head < p.nq ? p.q_out + (size_t)j * p.nq * p.hd + c0
                           : p.kc + kv_offset(p.seq_off, p.cap, i, p.nkv, p.hd, head - p.nq, p.cache_len[i]) + e;
    d[0] = y0;
    d[half] = y1;
  } else {
    const int g = head - p.nq - p.nkv;
    float* d = p.vc + kv_offset(p.seq_off, p.cap, i, p.nkv, p.hd, g, p.cache_len[i]) + e;
    d[0] = v0;
    d[half] = v1;
    if (p.pool) {
      float* pl = p.pool + (size_t)i * p.nkv * p.hd + g * p.hd + e;
      pl[0] += v0;
      pl[half] += v1;
    }
  }
}

template <int EPI, int kSimtRows>
__global__ void __launch_bounds__(256) gemm_simt_kernel(const SimtArgs p) {
  constexpr int NR = EPI == EPI_RESID ? 1 : 2;   // weight rows per unit
  const int unit = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  const int units = EPI == EPI_QKV ? p.N / 2 : p.N;
  const int K = p.K, half = p.hd >> 1;
  const bool in = unit < units;
  const float* w[NR];
  int head = 0, e = 0;
  if (EPI == EPI_QKV) {
    head = unit / half;
    e = unit - head * half;
    w[0] = p.W + (size_t)(head * p.hd + e) * K;
    w[NR - 1] = w[0] + (size_t)half * K;
  } else {
    w[0] = p.W + (size_t)unit * K;
    if (EPI == EPI_SWIGLU) w[NR - 1] = p.W + (size_t)(p.N + unit) * K;
  }
  float w0[NR][8];   // this lane's first weights, written by no kernel of the step
  const bool have = in && lane * 8 < K;
#pragma unroll
  for (int a = 0; a < NR; ++a)
    if (have) load8(w[a] + lane * 8, w0[a]);
  pdl_wait();
  pdl_trigger();
  if (!in || call_aborted(p.status)) return;
  const int m = p.count ? *p.count : p.n;
  constexpr bool NORM = EPI == EPI_QKV || EPI == EPI_SWIGLU;
  for (int j0 = 0; j0 < m; j0 += kSimtRows) {
    float acc[NR][kSimtRows], ss[kSimtRows];
    const float* x[kSimtRows];
#pragma unroll
    for (int r = 0; r < kSimtRows; ++r) {
      ss[r] = 0.f;
#pragma unroll
      for (int a = 0; a < NR; ++a) acc[a][r] = 0.f;
      const int j = min(j0 + r, m - 1);
      x[r] = NORM ? p.nsrc + (size_t)(p.rows ? p.rows[j] : j) * K : p.X + (size_t)j * K;
    }
    for (int k = lane * 8; k < K; k += 256) {
      float wv[NR][8], gv[8];
#pragma unroll
      for (int a = 0; a < NR; ++a) {
        if (k == lane * 8) {
#pragma unroll
          for (int u = 0; u < 8; ++u) wv[a][u] = w0[a][u];
        } else {
          load8(w[a] + k, wv[a]);
        }
      }
      if (NORM) load8(p.gamma + k, gv);
#pragma unroll
      for (int r = 0; r < kSimtRows; ++r) {
        float xv[8];
        const float4 a4 = *reinterpret_cast<const float4*>(x[r] + k), b4 = *reinterpret_cast<const float4*>(x[r] + k + 4);
        xv[0] = a4.x; xv[1] = a4.y; xv[2] = a4.z; xv[3] = a4.w;
        xv[4] = b4.x; xv[5] = b4.y; xv[6] = b4.z; xv[7] = b4.w;
        if (NORM) {
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            ss[r] += xv[u] * xv[u];
            xv[u] *= gv[u];
          }
        }
#pragma unroll
        for (int a = 0; a < NR; ++a)
#pragma unroll
          for (int u = 0; u < 8; ++u) acc[a][r] += wv[a][u] * xv[u];
      }
    }
    float v0 = 0.f, v1 = 0.f;
#pragma unroll
    for (int r = 0; r < kSimtRows; ++r) {
      float a0 = warp_sum(acc[0][r]), a1 = NR == 2 ? warp_sum(acc[NR - 1][r]) : 0.f;
      if (NORM) {
        const float inv = rsqrtf(warp_sum(ss[r]) / (float)K + p.eps);
        a0 *= inv;
        a1 *= inv;
      }
      if (r == lane) {
        v0 = a0;
        v1 = a1;
      }
    }
    const int j = j0 + lane;
    if (lane < kSimtRows && j < m) {
      if (EPI == EPI_RESID) {
        const size_t o = (size_t)(p.rows ? p.rows[j] : j) * p.N + unit;
        p.resid_dst[o] = p.resid_src[o] + v0;
      } else if (EPI == EPI_SWIGLU) {
        p.out[(size_t)j * p.N + unit] = silu_f(v0) * v1;
      } else {
        simt_qkv(p, j, head, e, v0, v1);
      }
    }
  }
}

constexpr int kStM = 32, kStN = 32, kStK = 32, kStStages = 4, kStRow = kStK + 4;

// X holds compact rows (normalised already).  A thread accumulates rows ty, ty +
// 16 and weight rows tx, tx + 16 of the tile; the second sixteen weight rows of a
// SwiGLU tile are the up rows of its sixteen gate rows.
template <int EPI>
__global__ void __launch_bounds__(256) gemm_simt_tiled_kernel(const SimtArgs p) {
  __shared__ __align__(16) float sm[kStStages][kStM + kStN][kStRow];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int i0 = blockIdx.y * kStM;
  const int u0 = blockIdx.x * (EPI == EPI_SWIGLU ? 16 : kStN);
  pdl_wait();
  pdl_trigger();
  if (call_aborted(p.status)) return;
  const int m = p.count ? *p.count : p.n;
  if (i0 >= m) return;
  const int K = p.K, steps = (K + kStK - 1) / kStK;
  // this thread's pieces of a step: row rr of X and of W, 4 floats
  const int rr = tid >> 3, kk = (tid & 7) * 4;
  const int wrow = EPI == EPI_SWIGLU ? (rr < 16 ? u0 + rr : p.N + u0 + rr - 16) : u0 + rr;
  const bool wok = EPI == EPI_SWIGLU ? u0 + (rr & 15) < p.N : wrow < p.N;
  const bool xok = i0 + rr < m;
  const float* xs = p.X + (size_t)(xok ? i0 + rr : i0) * K + kk;
  const float* ws = p.W + (size_t)(wok ? wrow : 0) * K + kk;
  auto load = [&](int s) {
    const int k = s * kStK + kk;
    auto cp = [&](float* d, const float* src, bool real) {
      const uint32_t n = real ? 16u : 0u;   // else zeros
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(d)),
                   "l"(src), "r"(n)
                   : "memory");
    };
    const bool kok = k < K;   // K is a multiple of 4
    cp(&sm[s % kStStages][rr][kk], kok ? xs + s * kStK : p.X, xok && kok);
    cp(&sm[s % kStStages][kStM + rr][kk], kok ? ws + s * kStK : p.W, wok && kok);
  };
  for (int s = 0; s < kStStages - 1; ++s) {
    if (s < steps) load(s);
    cp_async_commit();
  }
  // Each output is summed as a tree with short branches, so that its rounding errors
  // are no larger than those of the warps' sums in the other kernel: over k mod 4, of
  // those over the halves of a step (4 products each), then even and odd steps.  (Four
  // chains of K / 4 left stored values 1.6, 1.9 and 2.5 times as far from 64 bits at K =
  // 256, 512 and 2048.)
  auto add4 = [](float4& s, const float4& v) {
    s.x += v.x;
    s.y += v.y;
    s.z += v.z;
    s.w += v.w;
  };
  float4 even[2][2], odd[2][2];
#pragma unroll
  for (int a = 0; a < 2; ++a) even[a][0] = even[a][1] = odd[a][0] = odd[a][1] = make_float4(0.f, 0.f, 0.f, 0.f);
  auto step = [&](int s, float4 (&sum)[2][2]) {
    cp_async_wait<kStStages - 2>();
    __syncthreads();   // step s has landed for every thread, step s - 1 is consumed
    if (s + kStStages - 1 < steps) load(s + kStStages - 1);
    cp_async_commit();
    float4 t[2][2][2];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int a = 0; a < 2; ++a) t[h][a][0] = t[h][a][1] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < kStK; k += 4) {
      const int h = k / (kStK / 2);
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        const float4 x = *reinterpret_cast<const float4*>(&sm[s % kStStages][ty + 16 * a][k]);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          const float4 w = *reinterpret_cast<const float4*>(&sm[s % kStStages][kStM + tx + 16 * b][k]);
          t[h][a][b].x += x.x * w.x;
          t[h][a][b].y += x.y * w.y;
          t[h][a][b].z += x.z * w.z;
          t[h][a][b].w += x.w * w.w;
        }
      }
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        add4(t[0][a][b], t[1][a][b]);
        add4(sum[a][b], t[0][a][b]);
      }
  };
  int s = 0;
  for (; s + 1 < steps; s += 2) {
    step(s, even);
    step(s + 1, odd);
  }
  if (s < steps) step(s, even);
  cp_async_wait<0>();
  float acc[2][2];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      add4(even[a][b], odd[a][b]);
      acc[a][b] = (even[a][b].x + even[a][b].y) + (even[a][b].z + even[a][b].w);
    }
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const int j = i0 + ty + 16 * a;
    if (j >= m) continue;
    if constexpr (EPI == EPI_SWIGLU) {
      if (u0 + tx < p.N) p.out[(size_t)j * p.N + u0 + tx] = silu_f(acc[a][0]) * acc[a][1];
    } else {
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const int u = u0 + tx + 16 * b;
        if (u >= p.N) continue;
        if (EPI == EPI_STORE_F32) {
          p.out[(size_t)j * p.N + u] = acc[a][b];
        } else {
          const size_t o = (size_t)(p.rows ? p.rows[j] : j) * p.N + u;
          p.resid_dst[o] = p.resid_src[o] + acc[a][b];
        }
      }
    }
  }
}

// EPI_QKV: the fused form (in_norm_src set, at most kSimtFuseRows rows);
// EPI_SWIGLU: fused where in_norm_src is set, else tiled; EPI_RESID: by the row
// bound; EPI_STORE_F32: tiled.
void launch_gemm_simt(const Ctx& c, int epi, const GemmArgs& a, cudaStream_t s) {
  SimtArgs p{};
  p.W = (const float*)a.W;
  p.X = (const float*)a.X;
  p.nsrc = a.in_norm_src;
  p.gamma = a.in_norm_gamma;
  p.eps = c.cfg.rms_eps;
  p.N = a.N;
  p.K = a.K;
  p.rows = a.sel.rows;
  p.count = a.sel.count;
  p.n = a.sel.n;
  p.out = epi == EPI_SWIGLU ? (float*)a.out_act : a.out_f32;
  p.resid_src = a.resid_src;
  p.resid_dst = a.resid_dst;
  p.bias = a.qkv_bias;
  p.rope_cos = c.rope_cos;
  p.rope_sin = c.rope_sin;
  p.len = a.kv_len;
  p.cache_len = a.cache_len;
  p.seq_off = a.kv_seq_off;
  p.cap = a.kv_cap;
  p.kc = (float*)a.kc;
  p.vc = (float*)a.vc;
  p.q_out = a.q_out;
  p.pool = a.pool;
  p.nq = c.nq;
  p.nkv = c.nkv;
  p.hd = c.hd;
  p.status = a.status;
  const bool fused = a.sel.n <= kSimtFuseRows;
  const int units = epi == EPI_QKV ? a.N / 2 : a.N;
  const unsigned g = (unsigned)((units + 7) / 8);
  const dim3 t((a.N + (epi == EPI_SWIGLU ? 15 : kStN - 1)) / (epi == EPI_SWIGLU ? 16 : kStN),
               (a.sel.n + kStM - 1) / kStM);
  auto small = [&](auto k4, auto k8) { launch_k(a.sel.n <= 4 ? k4 : k8, g, 256, 0, s, c.pdl, p); };
  if (epi == EPI_QKV) small(gemm_simt_kernel<EPI_QKV, 4>, gemm_simt_kernel<EPI_QKV, 8>);
  else if (epi == EPI_STORE_F32) launch_k(gemm_simt_tiled_kernel<EPI_STORE_F32>, t, 256, 0, s, c.pdl, p);
  else if (epi == EPI_RESID && fused) small(gemm_simt_kernel<EPI_RESID, 4>, gemm_simt_kernel<EPI_RESID, 8>);
  else if (epi == EPI_RESID) launch_k(gemm_simt_tiled_kernel<EPI_RESID>, t, 256, 0, s, c.pdl, p);
  else if (fused) small(gemm_simt_kernel<EPI_SWIGLU, 4>, gemm_simt_kernel<EPI_SWIGLU, 8>);
  else launch_k(gemm_simt_tiled_kernel<EPI_SWIGLU>, t, 256, 0, s, c.pdl, p);
}

}  // namespace buddy
