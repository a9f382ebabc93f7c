// fp32 attention forward on CUDA cores (no TF32), for the MOA_FP32 element type.
//
// Computes O = softmax(scale * Q K^T) V (paper Section 4.1, Eq. attention) in
// the DNF's memory pattern: one CTA owns BM query rows of one (b, h) slice
// (the independent 2-D problems of the Remark in Section 4.2), streams K and V
// through shared memory in BN-key tiles, and keeps the scores of one tile, the
// running row maximum and the running denominator in registers.  The row max
// (Step I, Section 4.3), the exponentials (Step II, Section 4.4) and their sum
// (Step III, Section 4.5) are combined online: when a tile raises the running
// maximum from m to m', the partial sums are rescaled by exp(m - m'), which is
// the exact identity exp(s - m') = exp(s - m) * exp(m - m').  The division of
// Step IV happens once per row at the end.  Nothing but O is written to global
// memory.
//
// Layout: Q, K, V, O contiguous row-major [B,H,N,d] float32.
//
// What bounds it: the FMA pipe (152 SMs x 128 FMA/clk), provided that shared memory and issue keep
// up.  Each thread therefore holds an R x 8 block of scores and an R x 4 VC block of O in registers:
// per 4 features an R x 8 block costs R + 8 16-byte shared loads (two wavefronts each, see the lane
// map) for 32 R FMAs, which at R = 8 is half of what shared memory can deliver, at R = 4 three
// quarters.  K and V tiles come by cp.async while the previous tile's softmax and products run.
// A CTA is WR row warps (4R rows each) x KW key groups; the groups take alternate 64-key tiles and
// merge their (m, l, O) at the end, so that a short problem still puts 4 to 8 warps on an SM.
// Small R and more groups shorten the dependent chain of one CTA; large R does the least work per
// score.  pick_tile weighs the two from measured step times.
//
// Measured on a GB300 (2070 MHz; before: one lane per output column, 8-row warps, scalar loads):
// 2x8x1000x1500 d=64 482 -> 171 us (36 TFLOP/s), 1x8x1024x1024 d=128 517 -> 125 us, 1x8x256x256
// d=64 27 -> 10 us, 1x16x100x1500 133 -> 37 us, 1x1x300x2048 d=64 115 -> 33 us, 1x1x128x128 d=64 10.4 -> 4.8 us.  The tile's
// former fill by cp.async with a zero-fill source size cost more than its products (16-row tile,
// one 256-key step: 13 us with it, 6.4 us with the plain form and stores of zeros).
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

constexpr int kBN = 64;                     // keys per key group and step
constexpr int kHalf = kBN / 2;              // keys of P held in shared memory at a time
constexpr int kLdp = kHalf + 8;             // floats per row of P: 4 rows of a store or load on disjoint banks
constexpr int kMaxSmem = 232448;            // shared memory a CTA can have

// VC: 32-column blocks of V (ceil(d_v / 32)).  R: rows per thread (4R per warp).  WR: row warps,
// KW: key groups (two or more).
template <int VC, int R, int WR, int KW>
struct F32Tile {
  static constexpr int kThreads = 32 * WR * KW;
  static constexpr int kBM = 4 * R * WR;     // query rows per CTA
  static constexpr int kStep = kBN * KW;     // keys per step of the CTA
  static constexpr int kLdv = 32 * VC;
  // 128 registers hold an R = 4 thread with d_v <= 64 (two 8-warp CTAs an SM); the rest need more.
  static constexpr int kMinBlocks = (R == 4 && VC <= 2 ? 16 : 8) / (WR * KW) > 0
                                        ? (R == 4 && VC <= 2 ? 16 : 8) / (WR * KW) : 1;
  static size_t smem_bytes(int dk) {
    return sizeof(float) * (size_t(kBM) * odd_stride(dk) + size_t(kStep) * (odd_stride(dk) + kLdv) +
                            size_t(kBM) * KW * kLdp);
  }
};

template <int VC, int R, int WR, int KW>
__global__ void __launch_bounds__(F32Tile<VC, R, WR, KW>::kThreads, F32Tile<VC, R, WR, KW>::kMinBlocks)
attn_fwd_f32_cc_kernel(const float* __restrict__ Q, const float* __restrict__ K,
                       const float* __restrict__ V, float* __restrict__ O,
                       float* __restrict__ lse, int Nq, int Nk, int dk, int dv, int n_qtiles,
                       float scale) {
  using T = F32Tile<VC, R, WR, KW>;
  constexpr int kThreads = T::kThreads, kBM = T::kBM, kStep = T::kStep, kLdv = T::kLdv;
  // two iterations of the product loops together: 2 to 5 % where registers are left (R <= 4)
  constexpr int kUnroll = R == 8 ? 1 : 2;
  extern __shared__ __align__(16) float smem[];
  const int ldk = odd_stride(dk);
  float* sQ = smem;                // [kBM][ldk]
  float* sK = sQ + kBM * ldk;      // [kStep][ldk]
  float* sV = sK + kStep * ldk;    // [kStep][kLdv]
  float* sP = sV + kStep * kLdv;   // [KW * WR][4R][kLdp]

  const int lane = threadIdx.x & 31;
  const int warp = (threadIdx.x >> 5) % WR, kg = (threadIdx.x >> 5) / WR;  // row warp, key group
  // Column group 0..7 and row group 0..3.  Lanes 2i and 2i + 1 share their columns: a 16-byte shared
  // load then takes two wavefronts; with the column group in the low lane bits it takes four.
  const int cg = (lane >> 1) & 7, rg = (lane & 1) | (lane >> 4) << 1;
  const long long bh = blockIdx.x / n_qtiles;
  const int q0 = (blockIdx.x % n_qtiles) * kBM;
  const float* Qh = Q + bh * (long long)Nq * dk;
  const float* Kh = K + bh * (long long)Nk * dk;
  const float* Vh = V + bh * (long long)Nk * dv;

  // rows [r0, r0 + rows) of a [n, d] array -> shared rows of ld floats; rows past n are zeros
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
  grid_dependency_wait();
  request(sQ, ldk, Qh, dk, q0, kBM, Nq);
  request(sK, ldk, Kh, dk, 0, kStep, Nk);
  cp_async_commit();
  request(sV, kLdv, Vh, dv, 0, kStep, Nk);
  cp_async_commit();

  // This thread: rows 4r + rg (r < R) of its warp; keys cg + 8j (j < 8) of its group's tile;
  // output columns 32b + 4cg .. +3 (b < VC).
  float m[R], l[R], acc[R][4 * VC];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    m[r] = -INFINITY;
    l[r] = 0.f;
#pragma unroll
    for (int c = 0; c < 4 * VC; ++c) acc[r][c] = 0.f;
  }
  const float* myQ = sQ + (warp * 4 * R + rg) * ldk;                        // row r: + 4r*ldk
  const float* myK = sK + (kg * kBN + cg) * ldk;                            // key j: + 8j*ldk
  const float* myV = sV + kg * kBN * kLdv + 4 * cg;
  float* myP = sP + ((kg * WR + warp) * 4 * R + rg) * kLdp;                 // row r: + 4r*kLdp

  // left: keys from k0 on
  for (long long k0 = 0, left = Nk; left > 0; k0 += kStep, left -= kStep) {
    const int mine = int(left) - kg * kBN;  // keys from this group's tile on
    const bool live = mine > 0;  // warp-uniform
    cp_async_wait<1>();  // K tile (and Q) here; V may be on its way
    __syncthreads();
    float s[R][8];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int j = 0; j < 8; ++j) s[r][j] = 0.f;
    const int f_end = live ? dk : 0;
#pragma unroll kUnroll
    for (int f = 0; f < f_end; f += 4) {
      float4 kk[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) kk[j] = *reinterpret_cast<const float4*>(myK + 8 * j * ldk + f);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float4 q = *reinterpret_cast<const float4*>(myQ + 4 * r * ldk + f);
#pragma unroll
        for (int j = 0; j < 8; ++j) s[r][j] = fmaf(q.x, kk[j].x, s[r][j]);
#pragma unroll
        for (int j = 0; j < 8; ++j) s[r][j] = fmaf(q.y, kk[j].y, s[r][j]);
#pragma unroll
        for (int j = 0; j < 8; ++j) s[r][j] = fmaf(q.z, kk[j].z, s[r][j]);
#pragma unroll
        for (int j = 0; j < 8; ++j) s[r][j] = fmaf(q.w, kk[j].w, s[r][j]);
      }
    }
    __syncthreads();  // every warp has read the K tile
    if (left > kStep) request(sK, ldk, Kh, dk, k0 + kStep, kStep, Nk);
    cp_async_commit();

    // Online softmax; the 8 lanes of a row share its maximum, each keeps its own part of the sum.
    if (live) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
#pragma unroll
        for (int j = 0; j < 8; ++j) s[r][j] = cg + 8 * j < mine ? __fmul_rn(s[r][j], scale) : -INFINITY;
        float t = s[r][0];
#pragma unroll
        for (int j = 1; j < 8; ++j) t = fmaxf(t, s[r][j]);
#pragma unroll
        for (int off = 8; off > 1; off >>= 1) t = fmaxf(t, __shfl_xor_sync(0xffffffffu, t, off));
        const float mnew = fmaxf(m[r], t);
        // A group whose keys so far all score -inf (a mask) must not turn into NaN, for the other
        // groups may have the row's other keys.
        const float shift = mnew == -INFINITY ? 0.f : mnew;
        const float alpha = expf(m[r] - shift);    // exp(-inf) = 0 on the first tile
        m[r] = mnew;
        float sum = 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          s[r][j] = expf(s[r][j] - shift);
          sum += s[r][j];
        }
        l[r] = fmaf(l[r], alpha, sum);
#pragma unroll
        for (int c = 0; c < 4 * VC; ++c) acc[r][c] *= alpha;
      }
    }
    cp_async_wait<1>();  // V tile here; the next K may be on its way
    __syncthreads();
    if (live) {
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        if (half) __syncwarp();  // the first half's P has been read
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int j = 0; j < 4; ++j) myP[4 * r * kLdp + cg + 8 * j] = s[r][4 * half + j];
        __syncwarp();
#pragma unroll kUnroll
        for (int k = 0; k < kHalf; k += 4) {
          float4 vv[4][VC];
#pragma unroll
          for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int b = 0; b < VC; ++b)
              vv[u][b] = *reinterpret_cast<const float4*>(myV + (half * kHalf + k + u) * kLdv + 32 * b);
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const float4 p = *reinterpret_cast<const float4*>(myP + 4 * r * kLdp + k);
            const float pu[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
              for (int b = 0; b < VC; ++b) {
                acc[r][4 * b] = fmaf(pu[u], vv[u][b].x, acc[r][4 * b]);
                acc[r][4 * b + 1] = fmaf(pu[u], vv[u][b].y, acc[r][4 * b + 1]);
                acc[r][4 * b + 2] = fmaf(pu[u], vv[u][b].z, acc[r][4 * b + 2]);
                acc[r][4 * b + 3] = fmaf(pu[u], vv[u][b].w, acc[r][4 * b + 3]);
              }
          }
        }
      }
    }
    __syncthreads();  // every warp has read the V tile
    if (left > kStep) request(sV, kLdv, Vh, dv, k0 + kStep, kStep, Nk);
    cp_async_commit();
  }

  launch_dependents();  // not before: see the bf16 kernel on CTAs that share an SM
  // Merge of the key groups: O = sum_g e^(m_g - M) O_g, l = sum_g e^(m_g - M) l_g, M = max m_g.
  // Groups g > 0 leave their state where the tiles were (thread-private slots, lane-contiguous).
  constexpr int kState = 2 * R + 4 * R * VC;
  static_assert((KW - 1) * WR * kState * 32 <= kStep * (4 + kLdv) + kBM * KW * kLdp, "merge slots");
  float* slot = sK + lane;
  if (kg > 0) {
    float* mine = slot + ((kg - 1) * WR + warp) * kState * 32;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      mine[32 * r] = m[r];
      mine[32 * (R + r)] = l[r];
#pragma unroll
      for (int c = 0; c < 4 * VC; ++c) mine[32 * (2 * R + 4 * VC * r + c)] = acc[r][c];
    }
  }
  __syncthreads();
  if (kg > 0) return;
#pragma unroll 1
  for (int g = 1; g < KW && g * kBN < Nk; ++g) {  // groups that had a key
    const float* other = slot + ((g - 1) * WR + warp) * kState * 32;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float mo = other[32 * r], mn = fmaxf(m[r], mo);
      const float shift = mn == -INFINITY ? 0.f : mn;  // as in the loop: a later group may have keys
      const float a = expf(m[r] - shift), b = expf(mo - shift);
      m[r] = mn;
      l[r] = fmaf(other[32 * (R + r)], b, l[r] * a);
#pragma unroll
      for (int c = 0; c < 4 * VC; ++c)
        acc[r][c] = fmaf(other[32 * (2 * R + 4 * VC * r + c)], b, acc[r][c] * a);
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
#pragma unroll
    for (int off = 8; off > 1; off >>= 1) l[r] += __shfl_xor_sync(0xffffffffu, l[r], off);
    const int row = q0 + warp * 4 * R + 4 * r + rg;
    if (row >= Nq) continue;
    const float inv = 1.0f / l[r];
    // ln sum_k exp(scale s_k) = m + ln l (m is the exact row maximum here).
    if (lse != nullptr && cg == 0) lse[bh * Nq + row] = m[r] + logf(l[r]);
    float* orow = O + (bh * Nq + row) * (long long)dv;
#pragma unroll
    for (int b = 0; b < VC; ++b) {
      const int c = 32 * b + 4 * cg;
      if (c < dv)
        *reinterpret_cast<float4*>(orow + c) =
            make_float4(acc[r][4 * b] * inv, acc[r][4 * b + 1] * inv, acc[r][4 * b + 2] * inv,
                        acc[r][4 * b + 3] * inv);
    }
  }
}

template <int VC, int R, int WR, int KW>
int launch_tiled(const AttnArgs& a, char* msg, size_t msglen) {
  using T = F32Tile<VC, R, WR, KW>;
  const int n_qtiles = int((a.Nq + T::kBM - 1) / T::kBM);
  const long long grid = (long long)a.B * a.H * n_qtiles;
  if (grid > 0x7fffffffLL) {
    snprintf(msg, msglen, "fp32 path: B*H*ceil(N_q/%d) = %lld CTAs exceeds the grid limit", T::kBM, grid);
    return 3;
  }
  auto kern = attn_fwd_f32_cc_kernel<VC, R, WR, KW>;
  const size_t smem = T::smem_bytes(int(a.dk));
  cudaError_t e = ensure_smem_limit(reinterpret_cast<const void*>(kern), int(smem));
  if (e != cudaSuccess) {
    snprintf(msg, msglen, "cudaFuncSetAttribute (fp32 kernel): %s", cudaGetErrorString(e));
    return 5;
  }
  e = launch_dependent(kern, dim3(unsigned(grid)), dim3(T::kThreads), smem, a.stream,
                       static_cast<const float*>(a.Q), static_cast<const float*>(a.K),
                       static_cast<const float*>(a.V), static_cast<float*>(a.O), a.lse, int(a.Nq),
                       int(a.Nk), int(a.dk), int(a.dv), n_qtiles, a.scale);
  if (e != cudaSuccess) {
    snprintf(msg, msglen, "fp32 kernel launch: %s", cudaGetErrorString(e));
    return 5;
  }
  return 0;
}

// The tile shapes, with the measured time of one step of a CTA (us at d = 64; the ratios hold for
// other d): alone on its SM, and per CTA when `occ` of them share it.
struct TileShape {
  int r, wr, kw, occ;
  float lone, shared;
};
constexpr TileShape kTiles[] = {
    {8, 4, 2, 1, 14.0f, 14.0f}, {4, 4, 2, 2, 8.7f, 7.75f}, {4, 2, 2, 2, 5.6f, 4.3f},
    {2, 2, 2, 2, 3.9f, 3.0f},   {1, 2, 2, 2, 3.0f, 2.4f},  {4, 2, 4, 1, 9.0f, 9.0f},
    {4, 1, 4, 1, 6.4f, 6.4f},   {2, 1, 4, 1, 4.6f, 4.6f},  {1, 1, 4, 1, 4.0f, 4.0f}};
constexpr float kRoundStart = 2.0f;  // first tiles of a CTA and the merge, same unit

// Shared memory of a tile shape (F32Tile::smem_bytes with run-time sizes).
size_t tile_smem(const TileShape& t, int dk, int vc) {
  const size_t rows = 4 * size_t(t.r) * t.wr;
  return sizeof(float) * (rows * odd_stride(dk) +
                          size_t(kBN) * t.kw * (odd_stride(dk) + 32 * vc) + rows * t.kw * kLdp);
}

// Key groups, from the sizes of one (b, h) slice alone: the groups' merge decides the last bits of
// a slice, which must not depend on how many slices a call has.  Four groups where a slice has few
// rows (its calls are bound by the chain over the keys: 1x4x60x2000 64 -> 33 us, 1x32x300x700 83 ->
// 80 us) and their tiles fit; two else (at N_q >= 512 larger row tiles do the same work in less:
// 1x16x512x512 56 -> 39 us).
int key_groups(const AttnArgs& a, int dk, int vc) {
  return a.Nq < 512 && a.Nk > 2 * kBN && tile_smem({4, 2, 4, 1, 0, 0}, dk, vc) <= size_t(kMaxSmem) ? 4 : 2;
}

// The shape with the least estimated time: rounds of CTAs over the SMs x key steps x step time.
int pick_tile(const AttnArgs& a, int sms) {
  const int dk = int(a.dk), vc = int((a.dv + 31) / 32);
  const int kw = key_groups(a, dk, vc);
  int best = -1;
  double best_time = 0;
  for (int i = 0; i < int(sizeof(kTiles) / sizeof(kTiles[0])); ++i) {
    const TileShape& t = kTiles[i];
    const size_t smem = tile_smem(t, dk, vc);
    if (t.kw != kw || smem > size_t(kMaxSmem)) continue;
    // two CTAs an SM need the 128-register instances (d_v <= 64) and half the shared memory each
    const int occ = t.occ == 2 && vc <= 2 && smem <= size_t(kMaxSmem + 1024) / 2 - 1024 ? 2 : 1;
    const int64_t rows = 4 * t.r * t.wr, keys = int64_t(kBN) * t.kw;
    const double n = double(a.B * a.H) * double((a.Nq + rows - 1) / rows);
    const double steps = double((a.Nk + keys - 1) / keys);
    const double slots = double(sms) * occ, full = floor(n / slots), rem = n - full * slots;
    const double busy = occ * t.shared * steps + kRoundStart;
    const double tail = rem <= 0 ? 0.0 : rem <= sms ? t.lone * steps + kRoundStart : busy;
    const double time = full * busy + tail;
    if (best < 0 || time < best_time) {
      best = i;
      best_time = time;
    }
  }
  return best;
}

template <int VC>
int launch_shape(int tile, const AttnArgs& a, char* msg, size_t msglen) {
  switch (tile) {
    case 0: return launch_tiled<VC, 8, 4, 2>(a, msg, msglen);
    case 1: return launch_tiled<VC, 4, 4, 2>(a, msg, msglen);
    case 2: return launch_tiled<VC, 4, 2, 2>(a, msg, msglen);
    case 3: return launch_tiled<VC, 2, 2, 2>(a, msg, msglen);
    case 4: return launch_tiled<VC, 1, 2, 2>(a, msg, msglen);
    case 5: return launch_tiled<VC, 4, 2, 4>(a, msg, msglen);
    case 6: return launch_tiled<VC, 4, 1, 4>(a, msg, msglen);
    case 7: return launch_tiled<VC, 2, 1, 4>(a, msg, msglen);
    case 8: return launch_tiled<VC, 1, 1, 4>(a, msg, msglen);
  }
  snprintf(msg, msglen, "fp32 path: no tile fits d_k=%lld d_v=%lld", (long long)a.dk, (long long)a.dv);
  return 3;
}

}  // namespace

int launch_attn_fwd_f32(const AttnArgs& a, char* msg, size_t msglen) {
  int sms = 0;
  const cudaError_t e = device_sm_count(&sms);
  if (e != cudaSuccess) {
    snprintf(msg, msglen, "fp32 path: SM count: %s", cudaGetErrorString(e));
    return 5;
  }
  const int tile = pick_tile(a, sms);
  if (a.dv <= 32) return launch_shape<1>(tile, a, msg, msglen);
  if (a.dv <= 64) return launch_shape<2>(tile, a, msg, msglen);
  if (a.dv <= 96) return launch_shape<3>(tile, a, msg, msglen);
  return launch_shape<4>(tile, a, msg, msglen);
}

}  // namespace moa
