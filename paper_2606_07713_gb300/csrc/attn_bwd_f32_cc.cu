// fp32 attention backward on CUDA cores (no TF32), for the MOA_FP32 element type.
//
// Computes the same gradients as the bf16 backward (paper Stage 5, Section 9):
//     dS = W * (dO V^T - D),  D_i = sum_c dO_ic O_ic,
//     dQ = scale * dS K,  dK = scale * dS^T Q,  dV = W^T dO,
// with the weights rebuilt from the forward's log-sum-exp, W_ik = exp(scale * s_ik - LSE_i), so
// that no N_q x N_k array is written to global memory.  Two kernels, all fp32 with expf:
//   attn_bwd_f32_pre_kernel   one warp per query row: D_i (and LSE_i copied) into the padded
//                             workspace layout of the bf16 path;
//   attn_bwd_f32_kernel       the first CTAs own rows of keys (dK, dV; the queries stream), the
//                             others rows of queries (dQ; the keys stream), in one launch, so that
//                             the two parts fill each other's last round of CTAs.
// Layout: Q, K, V, O, dO, dQ, dK, dV contiguous row-major [B,H,N,d] float32; d <= 128, d % 4 == 0.
//
// What bounds it: the FMA pipe, seven tile products per (query, key) tile pair (S and dP are formed
// on both sides so that every sum stays in one CTA and its order is fixed).  A thread holds R x 8
// blocks of S and dP and R x 4C blocks of the gradients in registers; tiles, lane map and the
// split over key groups are those of the fp32 forward kernel.
// Measured on a GB300 (2070 MHz; before: one scalar shared load per operand and FMA, 32-row tiles):
// 1x8x1024x1024 d=64 1014 -> 212 us (25.3 TFLOP/s of the five algorithmic products), d=128 1646 ->
// 394 us; two iterations of the product loops together are worth 4 % of it.
#include <cuda_runtime.h>
#include <math.h>
#include <cstdio>

#include "f32_common.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace moa {
namespace {

using namespace f32;
using ptx::grid_dependency_wait;
using ptx::launch_dependents;

constexpr int kBN = 64;          // rows of the streamed axis per group and step
constexpr int kHalf = kBN / 2;   // columns of P or dS held in shared memory at a time
constexpr int kLdp = kHalf + 8;  // floats per row of those: 4 rows of a store or load on disjoint banks
constexpr int kMaxSmem = 232448;

// A tile shape, with the measured time of one step of a CTA (us at d = 64, mean of the two kinds):
// alone on its SM, and per CTA when two share it.
struct BwdShape {
  int r, wr, kw;
  float lone, shared;
};
// Two groups always: a group's sums decide the last bits of a (b, h) slice, which must not depend on
// how many slices a call has.
constexpr BwdShape kTiles[] = {
    {4, 4, 2, 13.2f, 13.2f}, {4, 2, 2, 8.3f, 7.4f}, {2, 2, 2, 5.7f, 5.0f}, {1, 2, 2, 5.0f, 3.5f}};
size_t bwd_smem(const BwdShape& t, int dk, int dv) {
  const size_t rows = 4 * size_t(t.r) * t.wr, step = size_t(kBN) * t.kw;
  const size_t d = odd_stride(dk) + odd_stride(dv), cols = (dk > dv ? dk : dv) > 64 ? 128 : 64;
  const size_t streamed = step * d + rows * t.kw * kLdp + 2 * step;
  const size_t merge = (t.kw - 1) * rows * 2 * cols;  // the groups' sums, where the streamed tiles were
  return sizeof(float) * (rows * d + (streamed > merge ? streamed : merge));
}

// Padded-row workspace (shared with the bf16 path): row r = bh * Nq_pad + i.
int64_t f32_padded_rows(int64_t Nq) { return (Nq + 127) / 128 * 128; }

// One warp per query row: D = sum_c dO * O; LSE copied beside it.
__global__ void __launch_bounds__(256)
attn_bwd_f32_pre_kernel(const float* __restrict__ O, const float* __restrict__ dO,
                        const float* __restrict__ lse, float* __restrict__ Lw,
                        float* __restrict__ Dw, int Nq, int Nq_pad, int dv, long long rows) {
  const long long t = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  launch_dependents();
  grid_dependency_wait();
  if (t >= rows) return;
  const long long bh = t / Nq;
  const int i = int(t % Nq);
  const float* o = O + t * dv;
  const float* g = dO + t * dv;
  float acc = 0.f;
  for (int c = lane; c < dv; c += 32) acc = fmaf(o[c], g[c], acc);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  if (lane == 0) {
    const long long r = bh * Nq_pad + i;
    Lw[r] = lse[t];
    Dw[r] = acc;
  }
}

// Column blocks of 32 (C) cover both d_k and d_v.  R: rows per thread (4R per warp).  WR: row
// warps, KW: groups of the streamed axis (two or more).
template <int C, int R, int WR, int KW>
struct BwdTile {
  static constexpr int kThreads = 32 * WR * KW;
  static constexpr int kBM = 4 * R * WR;   // rows per CTA: keys (dK, dV) or queries (dQ)
  static constexpr int kStep = kBN * KW;   // rows of the streamed axis per step
  static constexpr int kMinBlocks = WR * KW <= 4 ? 2 : 1;
};

// One CTA's gradients.  DKDV: rows are keys, queries stream, and dV += P^T dO, dK += dS^T Q; else
// rows are queries, keys stream, and dQ += dS K.  A1, A2: the rows' tiles (K, V or Q, dO); B1, B2
// the streamed ones (Q, dO or K, V).
template <int C, int R, int WR, int KW, bool DKDV>
__device__ __forceinline__ void bwd_rows(const float* __restrict__ A1, const float* __restrict__ A2,
                                         const float* __restrict__ B1, const float* __restrict__ B2,
                                         const float* __restrict__ Lw, const float* __restrict__ Dw,
                                         float* __restrict__ G1, float* __restrict__ G2, int nA,
                                         int nB, int dk, int dv, long long row_first, float scale,
                                         float* smem) {
  using T = BwdTile<C, R, WR, KW>;
  constexpr int kThreads = T::kThreads, kBM = T::kBM, kStep = T::kStep;
  const int ldk = odd_stride(dk), ldv = odd_stride(dv);
  float* sA1 = smem;                 // [kBM][ldk]
  float* sA2 = sA1 + kBM * ldk;      // [kBM][ldv]
  float* sB1 = sA2 + kBM * ldv;      // [kStep][ldk]
  float* sB2 = sB1 + kStep * ldk;    // [kStep][ldv]
  float* sP = sB2 + kStep * ldv;     // [KW * WR][4R][kLdp]
  float* sL = sP + kBM * KW * kLdp;  // [kStep]
  float* sD = sL + kStep;            // [kStep]

  const int lane = threadIdx.x & 31;
  const int warp = (threadIdx.x >> 5) % WR, kg = (threadIdx.x >> 5) / WR;
  const int cg = (lane >> 1) & 7, rg = (lane & 1) | (lane >> 4) << 1;

  const int seg0 = threadIdx.x & 15, row0 = threadIdx.x >> 4;
  auto request = [&](float* dst, int ld, const float* src, int d, long long r0, int rows, int n) {
    dst += row0 * ld + 4 * seg0;
    src += (r0 + row0) * d + 4 * seg0;
    const int last = int(min((long long)rows, n - r0));
    for (int s = 4 * seg0; s < d; s += 64, dst += 64, src += 64) {
      int r = row0;
#pragma unroll 4
      for (; r < last; r += kThreads / 16) cp_async16(dst + (r - row0) * ld, src + (long long)(r - row0) * d);
#pragma unroll 1
      for (; r < rows; r += kThreads / 16)
        *reinterpret_cast<float4*>(dst + (r - row0) * ld) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  auto request_step = [&](long long k0) {
    request(sB1, ldk, B1, dk, k0, kStep, nB);
    request(sB2, ldv, B2, dv, k0, kStep, nB);
    if constexpr (DKDV) {
      for (int i = threadIdx.x; i < kStep; i += kThreads) {
        const bool in = k0 + i < nB;
        sL[i] = in ? Lw[k0 + i] : 0.f;
        sD[i] = in ? Dw[k0 + i] : 0.f;
      }
    }
    cp_async_commit();
  };
  request(sA1, ldk, A1, dk, row_first, kBM, nA);
  request(sA2, ldv, A2, dv, row_first, kBM, nA);
  request_step(0);

  // This thread: rows 4r + rg (r < R) of its warp; streamed rows cg + 8j (j < 8) of its group's
  // tile; gradient columns 32b + 4cg .. +3.
  const int arow = warp * 4 * R + rg;
  const float* a1 = sA1 + arow * ldk;
  const float* a2 = sA2 + arow * ldv;
  const float* b1 = sB1 + kg * kBN * ldk;
  const float* b2 = sB2 + kg * kBN * ldv;
  float* myP = sP + ((kg * WR + warp) * 4 * R + rg) * kLdp;
  float Lr[R], Dr[R];
  if constexpr (!DKDV) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const long long q = row_first + arow + 4 * r;
      Lr[r] = q < nA ? Lw[q] : INFINITY;
      Dr[r] = q < nA ? Dw[q] : 0.f;
    }
  }
  float g1[R][4 * C], g2[DKDV ? R : 1][4 * C];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int c = 0; c < 4 * C; ++c) {
      g1[r][c] = 0.f;
      if (DKDV) g2[DKDV ? r : 0][c] = 0.f;
    }

  // x = rows . streamed rows over d features
  auto dots = [&](float(&x)[R][8], const float* a, const float* b, int ld, int d) {
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int j = 0; j < 8; ++j) x[r][j] = 0.f;
#pragma unroll 2
    for (int f = 0; f < d; f += 4) {
      float4 kk[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) kk[j] = *reinterpret_cast<const float4*>(b + (cg + 8 * j) * ld + f);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float4 q = *reinterpret_cast<const float4*>(a + 4 * r * ld + f);
#pragma unroll
        for (int j = 0; j < 8; ++j) x[r][j] = fmaf(q.x, kk[j].x, x[r][j]);
#pragma unroll
        for (int j = 0; j < 8; ++j) x[r][j] = fmaf(q.y, kk[j].y, x[r][j]);
#pragma unroll
        for (int j = 0; j < 8; ++j) x[r][j] = fmaf(q.z, kk[j].z, x[r][j]);
#pragma unroll
        for (int j = 0; j < 8; ++j) x[r][j] = fmaf(q.w, kk[j].w, x[r][j]);
      }
    }
  };
  // g += x . streamed rows (x through the warp's rows of shared memory, 32 columns at a time)
  auto accumulate = [&](float(&g)[R][4 * C], const float(&x)[R][8], const float* b, int ld) {
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      __syncwarp();  // what was there has been read
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int j = 0; j < 4; ++j) myP[4 * r * kLdp + cg + 8 * j] = x[r][4 * half + j];
      __syncwarp();
#pragma unroll 2
      for (int k = 0; k < kHalf; k += 4) {
        float4 vv[4][C];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int c = 0; c < C; ++c)
            vv[u][c] = *reinterpret_cast<const float4*>(b + (half * kHalf + k + u) * ld + 32 * c + 4 * cg);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const float4 p = *reinterpret_cast<const float4*>(myP + 4 * r * kLdp + k);
          const float pu[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
          for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int c = 0; c < C; ++c) {
              g[r][4 * c] = fmaf(pu[u], vv[u][c].x, g[r][4 * c]);
              g[r][4 * c + 1] = fmaf(pu[u], vv[u][c].y, g[r][4 * c + 1]);
              g[r][4 * c + 2] = fmaf(pu[u], vv[u][c].z, g[r][4 * c + 2]);
              g[r][4 * c + 3] = fmaf(pu[u], vv[u][c].w, g[r][4 * c + 3]);
            }
        }
      }
    }
  };

  for (long long k0 = 0, left = nB; left > 0; k0 += kStep, left -= kStep) {
    const int mine = int(left) - kg * kBN;  // streamed rows from this group's tile on
    cp_async_wait<0>();
    __syncthreads();
    if (mine > 0) {
      float p[R][8], ds[R][8];
      dots(p, a1, b1, ldk, dk);
      dots(ds, a2, b2, ldv, dv);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int col = cg + 8 * j;
        const float Lj = DKDV ? sL[kg * kBN + col] : 0.f, Dj = DKDV ? sD[kg * kBN + col] : 0.f;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const float w = expf(p[r][j] * scale - (DKDV ? Lj : Lr[r]));
          p[r][j] = w;
          ds[r][j] = w * (ds[r][j] - (DKDV ? Dj : Dr[r]));
        }
      }
      if (mine < kBN) {
        // Streamed rows past the last are zeros, but their products need not be: 0 * inf of a key that
        // scores -inf, or exp(0 - L) past the largest float.  They have no part in the sums.
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if (cg + 8 * j >= mine) p[r][j] = ds[r][j] = 0.f;
      }
      if constexpr (DKDV) accumulate(g2, p, b2, ldv);
      accumulate(g1, ds, b1, ldk);
    }
    __syncthreads();  // every warp has read the streamed tiles
    if (left > kStep) request_step(k0 + kStep);
  }

  launch_dependents();  // not before: see the bf16 forward on CTAs that share an SM
  // Sum over the groups, in their order: groups g > 0 leave theirs where the tiles were
  // (thread-private slots, lane-contiguous).
  constexpr int kState = (DKDV ? 2 : 1) * 4 * R * C;
  float* slot = sB1 + warp * kState * 32 + lane;
  if (kg > 0) {
    float* mine = slot + (kg - 1) * WR * kState * 32;
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int c = 0; c < 4 * C; ++c) {
        mine[32 * (4 * C * r + c)] = g1[r][c];
        if (DKDV) mine[32 * (4 * R * C + 4 * C * r + c)] = g2[DKDV ? r : 0][c];
      }
  }
  __syncthreads();
  if (kg > 0) return;
#pragma unroll 1
  for (int g = 0; g < KW - 1; ++g) {
    const float* other = slot + g * WR * kState * 32;
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int c = 0; c < 4 * C; ++c) {
        g1[r][c] += other[32 * (4 * C * r + c)];
        if (DKDV) g2[DKDV ? r : 0][c] += other[32 * (4 * R * C + 4 * C * r + c)];
      }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const long long row = row_first + arow + 4 * r;
    if (row >= nA) continue;
#pragma unroll
    for (int b = 0; b < C; ++b) {
      const int c = 32 * b + 4 * cg;
      if (c < dk)
        *reinterpret_cast<float4*>(G1 + row * dk + c) =
            make_float4(g1[r][4 * b] * scale, g1[r][4 * b + 1] * scale, g1[r][4 * b + 2] * scale,
                        g1[r][4 * b + 3] * scale);
      if (DKDV && c < dv) {
        const float* g = g2[DKDV ? r : 0];
        *reinterpret_cast<float4*>(G2 + row * dv + c) =
            make_float4(g[4 * b], g[4 * b + 1], g[4 * b + 2], g[4 * b + 3]);
      }
    }
  }
}

// CTAs [0, n_dkdv) take dK and dV of their keys, the rest dQ of their queries.
template <int C, int R, int WR, int KW>
__global__ void __launch_bounds__(BwdTile<C, R, WR, KW>::kThreads, BwdTile<C, R, WR, KW>::kMinBlocks)
attn_bwd_f32_kernel(const float* __restrict__ Q, const float* __restrict__ K,
                    const float* __restrict__ V, const float* __restrict__ dO,
                    const float* __restrict__ Lw, const float* __restrict__ Dw,
                    float* __restrict__ dQ, float* __restrict__ dK, float* __restrict__ dV, int Nq,
                    int Nk, int Nq_pad, int dk, int dv, unsigned n_dkdv, int n_ktiles, int n_qtiles,
                    float scale) {
  extern __shared__ __align__(16) float smem[];
  constexpr int kBM = BwdTile<C, R, WR, KW>::kBM;
  grid_dependency_wait();
  if (blockIdx.x < n_dkdv) {
    const long long bh = blockIdx.x / n_ktiles;
    const long long k0 = (long long)(blockIdx.x % n_ktiles) * kBM;
    const long long q = bh * Nq, k = bh * Nk;
    bwd_rows<C, R, WR, KW, true>(K + k * dk, V + k * dv, Q + q * dk, dO + q * dv, Lw + bh * Nq_pad,
                                 Dw + bh * Nq_pad, dK + k * dk, dV + k * dv, Nk, Nq, dk, dv, k0, scale,
                                 smem);
  } else {
    const unsigned t = blockIdx.x - n_dkdv;
    const long long bh = t / n_qtiles;
    const long long q0 = (long long)(t % n_qtiles) * kBM;
    const long long q = bh * Nq, k = bh * Nk;
    bwd_rows<C, R, WR, KW, false>(Q + q * dk, dO + q * dv, K + k * dk, V + k * dv, Lw + bh * Nq_pad,
                                  Dw + bh * Nq_pad, dQ + q * dk, nullptr, Nq, Nk, dk, dv, q0, scale,
                                  smem);
  }
}

template <int C, int R, int WR, int KW>
cudaError_t launch_rows(const BwdArgs& a, const float* Lw, const float* Dw, int64_t nq_pad) {
  using T = BwdTile<C, R, WR, KW>;
  const int64_t BH = a.B * a.H;
  const int64_t n_kt = (a.Nk + T::kBM - 1) / T::kBM, n_qt = (a.Nq + T::kBM - 1) / T::kBM;
  const size_t smem = bwd_smem({R, WR, KW, 0, 0}, int(a.dk), int(a.dv));
  auto kern = attn_bwd_f32_kernel<C, R, WR, KW>;
  const cudaError_t e = ensure_smem_limit(reinterpret_cast<const void*>(kern), int(smem));
  if (e != cudaSuccess) return e;
  return launch_dependent(
      kern, dim3(unsigned(BH * (n_kt + n_qt))), dim3(T::kThreads), smem, a.stream,
      static_cast<const float*>(a.Q), static_cast<const float*>(a.K),
      static_cast<const float*>(a.V), static_cast<const float*>(a.dO), Lw, Dw,
      static_cast<float*>(a.dQ), static_cast<float*>(a.dK), static_cast<float*>(a.dV), int(a.Nq),
      int(a.Nk), int(nq_pad), int(a.dk), int(a.dv), unsigned(BH * n_kt), int(n_kt), int(n_qt), a.scale);
}

// The shape with the least estimated time: all CTAs' steps spread over the SMs plus a third of the
// longest CTA, and at least that CTA's own chain (within 10 % of the measured times of 18 sizes).
int pick_tile(const BwdArgs& a, int sms) {
  const double bh = double(a.B * a.H);
  int best = -1;
  double best_time = 0;
  for (int i = 0; i < int(sizeof(kTiles) / sizeof(kTiles[0])); ++i) {
    const BwdShape& t = kTiles[i];
    const size_t smem = bwd_smem(t, int(a.dk), int(a.dv));
    if (smem > size_t(kMaxSmem)) continue;
    const bool two = t.wr * t.kw <= 4 && smem <= size_t(kMaxSmem + 1024) / 2 - 1024;
    const int64_t rows = 4 * t.r * t.wr, step = int64_t(kBN) * t.kw;
    // dK and dV take four of the seven products, dQ three
    const double kv = 8.0 / 7 * double((a.Nq + step - 1) / step), q = 6.0 / 7 * double((a.Nk + step - 1) / step);
    const double ctas_kv = bh * double((a.Nk + rows - 1) / rows), ctas_q = bh * double((a.Nq + rows - 1) / rows);
    const double chain = (kv > q ? kv : q) * t.lone;
    double time = (ctas_kv * kv + ctas_q * q) * (two ? t.shared : t.lone) / sms + 0.35 * chain;
    if (time < chain) time = chain;
    if (best < 0 || time < best_time) {
      best = i;
      best_time = time;
    }
  }
  return best;
}

template <int C>
cudaError_t launch_shape(int tile, const BwdArgs& a, const float* Lw, const float* Dw, int64_t nq_pad) {
  switch (tile) {
    case 0: return launch_rows<C, 4, 4, 2>(a, Lw, Dw, nq_pad);
    case 1: return launch_rows<C, 4, 2, 2>(a, Lw, Dw, nq_pad);
    case 2: return launch_rows<C, 2, 2, 2>(a, Lw, Dw, nq_pad);
    case 3: return launch_rows<C, 1, 2, 2>(a, Lw, Dw, nq_pad);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

int launch_attn_bwd_f32(const BwdArgs& a, char* msg, size_t msglen) {
  const int64_t BH = a.B * a.H;
  const int64_t nq_pad = f32_padded_rows(a.Nq);
  int sms = 0;
  cudaError_t e = device_sm_count(&sms);
  if (e != cudaSuccess) {
    snprintf(msg, msglen, "fp32 backward: SM count: %s", cudaGetErrorString(e));
    return 5;
  }
  const int tile = pick_tile(a, sms);
  const int64_t bm = 4 * kTiles[tile].r * kTiles[tile].wr;
  const int64_t n_ctas = BH * ((a.Nk + bm - 1) / bm + (a.Nq + bm - 1) / bm);
  if (n_ctas > 0x7fffffffLL || BH * a.Nq / 8 > 0x7fffffffLL) {
    snprintf(msg, msglen, "fp32 backward: grid too large");
    return 3;
  }
  const int dk = int(a.dk), dv = int(a.dv);
  float* Lw = static_cast<float*>(a.ws);
  float* Dw = Lw + BH * nq_pad;
  const long long rows = BH * a.Nq;
  e = launch_dependent(attn_bwd_f32_pre_kernel, dim3(unsigned((rows + 7) / 8)), dim3(256), 0, a.stream,
                       static_cast<const float*>(a.O), static_cast<const float*>(a.dO), a.lse, Lw, Dw,
                       int(a.Nq), int(nq_pad), dv, rows);
  if (e == cudaSuccess) {
    const int d = dk > dv ? dk : dv;
    e = d <= 32 ? launch_shape<1>(tile, a, Lw, Dw, nq_pad)
        : d <= 64 ? launch_shape<2>(tile, a, Lw, Dw, nq_pad) : launch_shape<4>(tile, a, Lw, Dw, nq_pad);
  }
  if (e != cudaSuccess) {
    snprintf(msg, msglen, "fp32 backward launch: %s", cudaGetErrorString(e));
    return 5;
  }
  return 0;
}

}  // namespace moa
