// Fused input projections on the fifth-generation tensor cores (tcgen05 + TMEM + TMA), sm_103a.
//
// What it computes (paper Section 4.1): Q = X W_Q, K = X W_K, V = X W_V for one input X
// [B, N, d] and the three weight matrices side by side in W [d, 2 H d_k + H d_v] (row-major,
// columns W_Q | W_K | W_V; column h*d_k + j of W_Q gives feature j of head h).  One GEMM
// C = X W over all B*N tokens reads X once for all three products, and its epilogue stores
// every 64-column block of C directly at its place in the head-major Q, K, V arrays
// [B, H, N, d] that the attention entry points read: no [B, N, 3, H, d] intermediate and no
// permute copy exists.
//
// Tiling: persistent pairs of CTAs on neighbouring SMs (clusters of two, tcgen05 cta_group::2) walk
// the 256-token x 256-column tiles of C.  Each CTA loads its own 128 tokens of X and half of the W
// tile's columns, so a pair reads 64 KB of L2 per 64 features where two single CTAs with 128 x 256
// tiles read 96 KB: the kernel is bound by operand delivery from L2 (512 tensor cycles a stage), not
// by DRAM (X and W are read once).  d in steps of 64 through a 6-stage TMA ring (X 128 x 64 K-major,
// W 64 x 128 MN-major: the weights are read as stored).  Two 256-column TMEM accumulators alternate
// between tiles, so the epilogue of one tile overlaps the main loop of the next.  If the last round
// of tiles fills at most half of the pairs, its tiles are cut into two 128-column halves.
// Warps of each CTA: 0 TMA; 1 TMEM allocation and, in the pair's first CTA, the MMA issue for both;
// 2-9 epilogue (warp w owns TMEM lanes 32*(w%4): the CTA's 128 token rows).  The second CTA's copies
// and epilogue signal the first CTA's barriers; commits signal both CTAs'.  Waits are bounded
// (status word g_moa_proj_status).  Up to 128 tokens a second kernel takes over (below).
//
// Measured on a GB300 against one-CTA 128 x 256 tiles with row-per-lane stores: 2x8192x4096 -> 12288
// 1316 -> 985 us back to back under the power cap (1253 -> 1674 TFLOP/s; 1158 -> 909 us in a burst),
// 4x2048x1024 -> 3072 46.7 -> 42.6 us, 1x512x4096 -> 12288 57.4 -> 43.3 us.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdio>

#include "internal.h"
#include "ptx.cuh"
#include "tc_common.cuh"

namespace moa {

__device__ unsigned int g_moa_proj_status = 0;

namespace {

using namespace ptx;
using namespace tc;

constexpr int kBM = 128;        // tokens per CTA (= TMEM lanes); a pair's tile has 2 kBM
constexpr int kBN = 256;        // output columns per tile (= TMEM columns per accumulator)
constexpr int kBK = 64;         // model features per stage (one 128-byte swizzle panel of X)
constexpr int kStages = 6;
constexpr int kAccs = 2;        // TMEM accumulators (2 x 256 = 512 columns)
constexpr int kThreads = 320;
constexpr int kLoadWarp = 0;
constexpr int kMmaWarp = 1;
constexpr int kEpiWarps = 8;    // two per TMEM lane quarter, each half of the columns
constexpr int kGroupM = 8;      // token blocks walked together (tile order)
constexpr int kXBytes = kBM * kBK * 2;       // 16 KB: 128 rows x 128 B
constexpr int kWPanelBytes = kBK * 64 * 2;   // 8 KB: 64 rows x 64 columns
constexpr int kWBytes = 2 * kWPanelBytes;    // this CTA's half of the tile's columns
constexpr int kStageBytes = kXBytes + kWBytes;
constexpr int kOutBytes = 32 * 128;          // one epilogue warp's staging: 32 rows x 64 columns, bf16
constexpr int kOffOut = kStages * kStageBytes;
constexpr int kOffBar = kOffOut + kEpiWarps * kOutBytes;
// full[NS] (used in the first CTA), empty[NS], acc_full[2], acc_empty[2] (first CTA), drain
constexpr int kNumBars = 2 * kStages + 2 * kAccs + 1;
constexpr int kOffMisc = kOffBar + kNumBars * 8;
constexpr int kSmemBytes = kOffMisc + 16 + 1024;
static_assert(kSmemBytes <= 232448, "shared memory budget");

struct ProjDims {
  int N;        // tokens per batch entry (rows of one head's Q/K/V)
  int M;        // B * N
  int H, dk, dv;
  int ncol;     // 2 H dk + H dv
  int n_ktiles; // ceil(d / 64)
  int n_ntiles; // ceil(ncol / 256)
  int n_mtiles; // ceil(M / 256)
  int n_whole;  // tiles [0, n_whole) in one piece, the rest as two 128-column halves
  int n_items;  // n_whole + 2 * (tiles - n_whole)
};

// One work item: token block, first column, width (256 or 128).
struct Item {
  int m, c0, width;
};
// Tiles run over groups of kGroupM token blocks, token blocks fastest: the pairs working at one time
// then cover a near-square patch of C and share its X and W through L2.
__device__ __forceinline__ Item item_of(int i, const ProjDims& p) {
  const int t = i < p.n_whole ? i : p.n_whole + (i - p.n_whole) / 2;
  const int per_group = kGroupM * p.n_ntiles, g = t / per_group, r = t - g * per_group;
  const int rows = min(kGroupM, p.n_mtiles - g * kGroupM);
  Item it;
  it.m = g * kGroupM + r % rows;
  it.c0 = (r / rows) * kBN;
  it.width = kBN;
  if (i >= p.n_whole) {
    it.width = kBN / 2;
    it.c0 += ((i - p.n_whole) & 1) * (kBN / 2);
  }
  return it;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
qkv_proj_bf16_tc_kernel(const __grid_constant__ CUtensorMap tmX,
                        const __grid_constant__ CUtensorMap tmW, __nv_bfloat16* __restrict__ Q,
                        __nv_bfloat16* __restrict__ K, __nv_bfloat16* __restrict__ V, ProjDims p,
                        uint64_t wait_limit_ns) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar0 = smem_u32(smem + kOffBar);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kStages + s); };
  auto acc_full = [&](int a) { return bar0 + 8u * (2 * kStages + a); };
  auto acc_empty = [&](int a) { return bar0 + 8u * (2 * kStages + kAccs + a); };
  const uint32_t drain = bar0 + 8u * (2 * kStages + 2 * kAccs);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kOffMisc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kOffMisc + 4);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int rank = int(blockIdx.x & 1);  // cluster rank: clusters are (2, 1, 1)
  const int pair = int(blockIdx.x >> 1), n_pairs = int(gridDim.x >> 1);
  const WaitCtl wc{abort_flag, wait_limit_ns, 0u, &g_moa_proj_status};

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < kAccs; ++a) {
      mbar_init(acc_full(a), 1);
      mbar_init(acc_empty(a), 2 * kEpiWarps);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == kMmaWarp) {
    tmem_alloc_2cta(smem_u32(tmem_slot), kAccs * kBN);
    tmem_relinquish_2cta();
  }
  tc_fence_before_sync();
  cluster_sync();  // both CTAs' barriers are initialised before either is signalled
  tc_fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  launch_dependents();     // what follows on the stream may take SMs as they come free
  grid_dependency_wait();  // what came before has ended: its results are visible

  if (warp == kLoadWarp) {
    if (lane == 0) {
      tma_prefetch_desc(&tmX);
      tma_prefetch_desc(&tmW);
      int slot = 0;
      uint32_t phase = 0, issued = 0, issued_phase = 0;
      bool ok = true;
      for (int i = pair; ok && i < p.n_items; i += n_pairs) {
        const Item it = item_of(i, p);
        const int m0 = it.m * (2 * kBM) + rank * kBM;
        const int panels = it.width / 128;  // 64-column panels of this CTA's half of the columns
        const int c0 = it.c0 + rank * (it.width / 2);
        const uint32_t bytes = uint32_t(kXBytes + panels * kWPanelBytes);
        for (int kt = 0; kt < p.n_ktiles; ++kt) {
          if (!wait_bounded(empty_bar(slot), phase ^ 1u, wc)) {
            ok = false;
            break;
          }
          issued |= 1u << slot;
          issued_phase = (issued_phase & ~(1u << slot)) | (phase << slot);
          const uint32_t st = sbase + slot * kStageBytes;
          const uint32_t bar = cluster_addr(full_bar(slot), 0);  // the first CTA's barrier
          if (rank == 0) mbar_arrive_expect_tx(full_bar(slot), 2 * bytes);
          // X: columns [kt*64, +64) of rows [m0, +128); W: rows [kt*64, +64), 64-column panels
          // (rows past M or d and columns past ncol read as 0)
          tma_load_3d_2cta(st, &tmX, bar, kt * kBK, m0, 0);
          for (int q = 0; q < panels; ++q)
            tma_load_3d_2cta(st + kXBytes + q * kWPanelBytes, &tmW, bar, c0 + 64 * q, kt * kBK, 0);
          if (++slot == kStages) {
            slot = 0;
            phase ^= 1u;
          }
        }
      }
      if (!ok || *abort_flag) {
        // Let every copy already issued land before the CTA can exit.  The second CTA's copies
        // signal the other CTA, so it allows them a fixed time, many times a copy's.
        if (rank == 0) {
          for (int sl = 0; sl < kStages; ++sl)
            if (issued & (1u << sl))
              wait_quiesce(full_bar(sl), (issued_phase >> sl) & 1u, wait_limit_ns, &g_moa_proj_status);
        } else {
          const uint64_t t0 = globaltimer_ns();
          while (globaltimer_ns() - t0 < 10000000ull) {
          }
        }
      }
    }
  } else if (warp == kMmaWarp) {
    if (lane == 0 && rank == 0) {
      // C (+)= X W for the pair: M = 256 tokens, N = 256 or 128 columns, K = 16 per MMA.  A = X
      // tiles K-major (32 B per step inside the 128-byte panel).  B = W tiles MN-major: groups of 8
      // rows 1024 B apart (stride byte offset), 64-column panels kWPanelBytes apart (leading byte
      // offset), 16 rows = 2048 B per step.  Both operands at the same offsets in the two CTAs.
      int slot = 0;
      uint32_t phase = 0;
      bool ok = true;
      int n = 0;
      for (int i = pair; ok && i < p.n_items; i += n_pairs, ++n) {
        const int a = n & 1;
        const uint32_t tacc = tmem + a * kBN;
        const uint32_t idesc = item_of(i, p).width == kBN ? make_idesc(2 * kBM, kBN, true)
                                                          : make_idesc(2 * kBM, kBN / 2, true);
        // both CTAs' epilogues have drained this accumulator (its use before last)
        ok = wait_bounded(acc_empty(a), (uint32_t(n >> 1) & 1u) ^ 1u, wc);
        if (!ok) break;
        tc_fence_after_sync();
        for (int kt = 0; kt < p.n_ktiles; ++kt) {
          ok = wait_bounded(full_bar(slot), phase, wc);
          if (!ok) break;
          tc_fence_after_sync();
          const uint32_t st = sbase + slot * kStageBytes;
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk)
            mma_f16_ss_2cta(tacc, make_sdesc_sw128(st + kk * 32, 16, 1024),
                            make_sdesc_sw128(st + kXBytes + kk * 2048, kWPanelBytes, 1024), idesc,
                            (kt > 0 || kk > 0) ? 1u : 0u);
          mma_commit_2cta(empty_bar(slot));
          if (++slot == kStages) {
            slot = 0;
            phase ^= 1u;
          }
        }
        if (ok) mma_commit_2cta(acc_full(a));
      }
      mma_commit_2cta(drain);  // TMEM quiescent before it is freed, also on the abort path
    }
  } else {
    // Epilogue: every 64-column block of C goes to one head of Q, K or V.  A warp turns its 32 rows
    // through shared memory (16-byte chunk c of row r at c ^ r % 8), so that 8 lanes store the 128
    // bytes of a row together: a row per lane, 16 bytes at a time, wrote half sectors and took as
    // long as the main loop of a d_model = 1024 tile.
    const int lane_base = (warp & 3) * 32;
    const int half = (warp - 2) >> 2;  // which half of the tile's 64-column blocks
    uint8_t* stage = smem + kOffOut + (warp - 2) * kOutBytes;
    uint8_t* stage_w = stage + lane * 128;
    const int sub = lane >> 3, chunk = lane & 7;  // stores: rows 4i + sub, 16 bytes `chunk`
    const int hq = p.H * p.dk;
    int n = 0;
    for (int i = pair; i < p.n_items; i += n_pairs, ++n) {
      const int a = n & 1;
      const Item it = item_of(i, p);
      const int m0 = it.m * (2 * kBM) + rank * kBM + lane_base + sub;
      long long base[8];  // row of head 0 in [B, H, N, *]; -1: past the last token
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int m = m0 + 4 * t, b = m / p.N;
        base[t] = m < p.M ? (long long)b * p.H * p.N + (m - b * p.N) : -1;
      }
      if (!wait_bounded(acc_full(a), uint32_t(n >> 1) & 1u, wc)) break;
      tc_fence_after_sync();
      const int blocks = it.width / 128;  // 64-column blocks of this warp
#pragma unroll 1
      for (int c = half * (it.width / 2), e = c + 64 * blocks; c < e; c += 64) {
        uint32_t o[64];
        const uint32_t src = tmem + (uint32_t(lane_base) << 16) + a * kBN + c;
        tmem_ld_32x32b_x32(src, o);
        tmem_ld_32x32b_x32(src + 32, o + 32);
        tmem_wait_ld();
        reg_anchor_x32(o);
        reg_anchor_x32(o + 32);
        const int col = it.c0 + c;
        if (col >= p.ncol) break;  // warp-uniform: ncol is a multiple of 64
#pragma unroll
        for (int t = 0; t < 8; ++t)
          *reinterpret_cast<uint4*>(stage_w + ((t ^ (lane & 7)) << 4)) =
              make_uint4(pack_bf16x2(__uint_as_float(o[8 * t]), __uint_as_float(o[8 * t + 1])),
                         pack_bf16x2(__uint_as_float(o[8 * t + 2]), __uint_as_float(o[8 * t + 3])),
                         pack_bf16x2(__uint_as_float(o[8 * t + 4]), __uint_as_float(o[8 * t + 5])),
                         pack_bf16x2(__uint_as_float(o[8 * t + 6]), __uint_as_float(o[8 * t + 7])));
        __syncwarp();
        __nv_bfloat16* out = col < hq ? Q : col < 2 * hq ? K : V;
        const int d = col < 2 * hq ? p.dk : p.dv;
        const int cc = col < hq ? col : col < 2 * hq ? col - hq : col - 2 * hq;
        out += size_t(cc / d) * p.N * d + cc % d + 8 * chunk;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          const int r = 4 * t + sub;
          const uint4 v = *reinterpret_cast<const uint4*>(stage + r * 128 + ((chunk ^ (r & 7)) << 4));
          if (base[t] >= 0) *reinterpret_cast<uint4*>(out + base[t] * d) = v;
        }
        __syncwarp();
      }
      // this accumulator may now take the tile after next
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(cluster_addr(acc_empty(a), 0));
    }
  }

  // All roles of this CTA have ended, so the last commit is due: the second CTA's MMA warp, which issues
  // nothing, must not spend one wait's limit on the whole run.
  __syncthreads();
  if (warp == kMmaWarp) wait_quiesce(drain, 0, wait_limit_ns, &g_moa_proj_status);
  tc_fence_before_sync();
  __syncwarp();
  cluster_sync();  // neither CTA leaves while the other may still signal it or read its tiles
  if (warp == kMmaWarp) {
    tc_fence_after_sync();
    tmem_dealloc_2cta(tmem, kAccs * kBN);
  }
}

// ------------------------------------------------------------------------------------------
// At most 128 tokens (decoding, short prompts)
// ------------------------------------------------------------------------------------------
// W is then nearly all of the traffic and a 256-token tile nearly all padding, so the roles turn:
// 128 columns of W are the M side (A operand, MN-major as stored), the NT tokens (16, 32, 64 or 128)
// the N side.  Few column blocks would leave SMs idle, so a cluster of KS CTAs splits d for one
// block and adds its partial sums, in rank order, through distributed shared memory.  Two CTAs an SM
// (about 100 KB of ring each) keep enough of W in flight.  Warps: 0 TMA, 1 TMEM allocation and MMA
// issue, 2-5 epilogue (lane = column).
// Measured on a GB300, d_model 4096 -> 12288 columns (100 MB of W), against the 256-token tile: 1
// token 33.0 -> 15.9 us (6.3 TB/s), 40 tokens 29 -> 21 us, 128 tokens 28.7 -> 26.3 us; at 129 tokens
// the tile here would need a second pass over W, so the line is at 128.
constexpr int kSmallCols = 128;
constexpr int kSmallThreads = 192;
constexpr int kSmallWBytes = 2 * kWPanelBytes;  // 64 rows x 128 columns
constexpr int kSmallMaxStages = 6;
constexpr int kSmallRingBytes = 108 * 1024;

struct SmallCfg {
  int nt;      // tokens of the tile: 16, 32, 64 or 128
  int stages;
  int ks;      // CTAs per cluster
};

__host__ __device__ constexpr int small_stage_bytes(int nt) { return kSmallWBytes + nt * 128; }
__host__ __device__ constexpr int small_smem_bytes(const SmallCfg& c) {
  return c.stages * small_stage_bytes(c.nt) + (2 * kSmallMaxStages + 1) * 8 + 16 + 1024;
}

constexpr int kSmallMaxSmem = kSmallRingBytes + (2 * kSmallMaxStages + 1) * 8 + 16 + 1024;
static_assert(2 * (kSmallMaxSmem + 1024) <= 233472, "two CTAs per SM");

__global__ void __launch_bounds__(kSmallThreads, 2)
qkv_proj_small_kernel(const __grid_constant__ CUtensorMap tmX,
                      const __grid_constant__ CUtensorMap tmW, __nv_bfloat16* __restrict__ Q,
                      __nv_bfloat16* __restrict__ K, __nv_bfloat16* __restrict__ V, ProjDims p,
                      SmallCfg cfg, uint64_t wait_limit_ns) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  const int stage_bytes = small_stage_bytes(cfg.nt);
  uint8_t* bars = smem + cfg.stages * stage_bytes;
  const uint32_t sbase = smem_u32(smem), bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kSmallMaxStages + s); };
  const uint32_t drain = bar0 + 8u * (2 * kSmallMaxStages);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + (2 * kSmallMaxStages + 1) * 8);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* part = reinterpret_cast<float*>(smem);  // [nt][128] partial sums, once the ring is done

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int rank = int(blockIdx.x) % cfg.ks;  // cluster rank: clusters are (ks, 1, 1)
  const int c0 = int(blockIdx.x) / cfg.ks * kSmallCols;
  // this CTA's 64-feature steps: an even share, at least one (ks <= n_ktiles)
  const int kt0 = int((long long)p.n_ktiles * rank / cfg.ks);
  const int kt1 = int((long long)p.n_ktiles * (rank + 1) / cfg.ks);
  const uint32_t tmem_cols = cfg.nt < 32 ? 32 : cfg.nt;
  const WaitCtl wc{abort_flag, wait_limit_ns, 0u, &g_moa_proj_status};

  if (threadIdx.x == 0) {
    for (int s = 0; s < cfg.stages; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  grid_dependency_wait();  // what came before has ended: its results are visible

  if (warp == 0) {
    if (lane == 0) {
      tma_prefetch_desc(&tmX);
      tma_prefetch_desc(&tmW);
      int slot = 0;
      uint32_t phase = 0, issued = 0, issued_phase = 0;
      bool ok = true;
      for (int kt = kt0; kt < kt1; ++kt) {
        if (!wait_bounded(empty_bar(slot), phase ^ 1u, wc)) {
          ok = false;
          break;
        }
        issued |= 1u << slot;
        issued_phase = (issued_phase & ~(1u << slot)) | (phase << slot);
        const uint32_t st = sbase + slot * stage_bytes;
        mbar_arrive_expect_tx(full_bar(slot), stage_bytes);
        tma_load_3d(st, &tmW, full_bar(slot), c0, kt * kBK, 0);
        tma_load_3d(st + kWPanelBytes, &tmW, full_bar(slot), c0 + 64, kt * kBK, 0);
        tma_load_3d(st + kSmallWBytes, &tmX, full_bar(slot), kt * kBK, 0, 0);
        if (++slot == cfg.stages) {
          slot = 0;
          phase ^= 1u;
        }
      }
      if (!ok || *abort_flag)
        for (int sl = 0; sl < cfg.stages; ++sl)
          if (issued & (1u << sl))
            wait_quiesce(full_bar(sl), (issued_phase >> sl) & 1u, wait_limit_ns, &g_moa_proj_status);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // C^T (+)= W^T X^T: M = 128 columns, N = nt tokens, K = 16 per MMA.  A = W tile MN-major (16
      // rows = 2048 B per step, 64-column panels kWPanelBytes apart), B = X tile K-major.
      const uint32_t idesc = make_idesc_a_mn(kSmallCols, cfg.nt, false);
      int slot = 0;
      uint32_t phase = 0;
      for (int kt = kt0; kt < kt1; ++kt) {
        if (!wait_bounded(full_bar(slot), phase, wc)) break;
        tc_fence_after_sync();
        const uint32_t st = sbase + slot * stage_bytes;
#pragma unroll
        for (int kk = 0; kk < kBK / 16; ++kk)
          mma_f16_ss(tmem, make_sdesc_sw128(st + kk * 2048, kWPanelBytes, 1024),
                     make_sdesc_sw128(st + kSmallWBytes + kk * 32, 16, 1024), idesc,
                     (kt > kt0 || kk > 0) ? 1u : 0u);
        mma_commit(empty_bar(slot));
        if (++slot == cfg.stages) {
          slot = 0;
          phase ^= 1u;
        }
      }
      mma_commit(drain);  // TMEM quiescent, also on the abort path
    }
    __syncwarp();
    wait_quiesce(drain, 0, wait_limit_ns, &g_moa_proj_status);
  } else if (wait_bounded(drain, 0, wc)) {
    launch_dependents();  // not before: see the bf16 forward on CTAs that share an SM
    // The products have read every stage: the ring's memory now takes the partial sums.
    tc_fence_after_sync();
    const int col = (warp & 3) * 32 + lane;
#pragma unroll 1
    for (int t = 0; t < cfg.nt; t += 16) {
      uint32_t o[16];
      tmem_ld_32x32b_x16(tmem + (uint32_t((warp & 3) * 32) << 16) + t, o);
      tmem_wait_ld();
      reg_anchor_x16(o);
#pragma unroll
      for (int i = 0; i < 16; ++i) part[(t + i) * kSmallCols + col] = __uint_as_float(o[i]);
    }
  }
  tc_fence_before_sync();
  __syncwarp();
  cluster_sync();  // every CTA's partial sums are in its shared memory
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, tmem_cols);
  }
  if (warp >= 2) {
    // One warp per token, four columns per lane; the cluster's CTAs take turns over the tokens.
    const int gc = c0 + 4 * lane, hq = p.H * p.dk;
    if (gc < p.ncol) {
      __nv_bfloat16* out = gc < hq ? Q : gc < 2 * hq ? K : V;
      const int d = gc < 2 * hq ? p.dk : p.dv;
      const int cc = gc < hq ? gc : gc < 2 * hq ? gc - hq : gc - 2 * hq;
      out += size_t(cc / d) * p.N * d + cc % d;
#pragma unroll 4
      for (int t = rank + cfg.ks * (warp - 2); t < p.M; t += cfg.ks * 4) {  // M <= nt
        float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int r = 0; r < cfg.ks; ++r) {
          const float4 v = ld_cluster_f32x4(cluster_addr(sbase + uint32_t(t * kSmallCols + 4 * lane) * 4u, r));
          sum.x += v.x, sum.y += v.y, sum.z += v.z, sum.w += v.w;
        }
        const int b = t / p.N;
        *reinterpret_cast<uint2*>(out + (size_t(b) * p.H * p.N + (t - b * p.N)) * d) =
            make_uint2(pack_bf16x2(sum.x, sum.y), pack_bf16x2(sum.z, sum.w));
      }
    }
  }
  __syncwarp();
  cluster_sync();  // no CTA leaves while another still reads its sums
}

// Tokens of the tile, ring depth and cluster size for M <= 128 tokens: the largest power of two of
// CTAs per column block that keeps all CTAs resident (two per SM) with at least two steps each.
SmallCfg small_cfg(int M, int ncol, int n_ktiles, int sms) {
  SmallCfg c;
  c.nt = M <= 16 ? 16 : M <= 32 ? 32 : M <= 64 ? 64 : 128;
  c.stages = kSmallRingBytes / small_stage_bytes(c.nt);
  if (c.stages > kSmallMaxStages) c.stages = kSmallMaxStages;
  const int blocks = (ncol + kSmallCols - 1) / kSmallCols;
  c.ks = 1;
  while (c.ks < 8 && int64_t(blocks) * c.ks * 2 <= 2 * sms && n_ktiles >= 4 * c.ks) c.ks *= 2;
  return c;
}

}  // namespace

int launch_qkv_proj_bf16(const ProjArgs& a, char* msg, size_t msglen) {
  ProjDims p;
  p.N = int(a.N);
  p.M = int(a.B * a.N);
  p.H = int(a.H);
  p.dk = int(a.dk);
  p.dv = int(a.dv);
  p.ncol = int(2 * a.H * a.dk + a.H * a.dv);
  p.n_ktiles = int((a.d + kBK - 1) / kBK);
  p.n_ntiles = (p.ncol + kBN - 1) / kBN;
  p.n_mtiles = int((int64_t(p.M) + 2 * kBM - 1) / (2 * kBM));
  const int64_t n_tiles = int64_t(p.n_mtiles) * p.n_ntiles;
  int sm_count = 0;
  cudaError_t se = device_sm_count(&sm_count);
  if (se != cudaSuccess) {
    snprintf(msg, msglen, "projection: SM count: %s", cudaGetErrorString(se));
    return 5;
  }
  CUtensorMap mx, mw;
  // X as [1, M, d] (box 64 x 128 rows, or the small tile's rows); W as [1, d, ncol] (box 64 columns
  // x 64 rows)
  const bool small = p.M <= 128;
  const SmallCfg sc = small_cfg(p.M, p.ncol, p.n_ktiles, sm_count);
  if (!encode_bf16_map_box(&mx, a.X, 1, p.M, a.d, small ? sc.nt : 128, msg, msglen)) return 5;
  if (!encode_bf16_map_box(&mw, a.W, 1, a.d, p.ncol, 64, msg, msglen)) return 5;
  const void* kern = small ? reinterpret_cast<const void*>(qkv_proj_small_kernel)
                           : reinterpret_cast<const void*>(qkv_proj_bf16_tc_kernel);
  const cudaError_t attr_err =
      ensure_smem_limit(kern, small ? kSmallMaxSmem : kSmemBytes);
  if (attr_err != cudaSuccess) {
    snprintf(msg, msglen, "cudaFuncSetAttribute (projection): %s", cudaGetErrorString(attr_err));
    return 5;
  }
  if (small) {
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(unsigned((p.ncol + kSmallCols - 1) / kSmallCols) * unsigned(sc.ks));
    lc.blockDim = dim3(kSmallThreads);
    lc.dynamicSmemBytes = small_smem_bytes(sc);
    lc.stream = a.stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim = {unsigned(sc.ks), 1, 1};
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&lc, qkv_proj_small_kernel, mx, mw,
                                             static_cast<__nv_bfloat16*>(a.Q),
                                             static_cast<__nv_bfloat16*>(a.K),
                                             static_cast<__nv_bfloat16*>(a.V), p, sc, wait_limit_ns());
    if (e != cudaSuccess) {
      snprintf(msg, msglen, "projection launch: %s", cudaGetErrorString(e));
      return 5;
    }
    return 0;
  }
  if (n_tiles > 0x3fffffffLL) {
    snprintf(msg, msglen, "projection: too many tiles");
    return 3;
  }
  // Halves in the last round if they still fit one round: 4x2048x1024 -> 3072 is 384 tiles for 76
  // pairs, 5 whole rounds and 8 halves.
  const int64_t pairs = sm_count / 2 > 0 ? sm_count / 2 : 1, rest = n_tiles % pairs;
  p.n_whole = int(2 * rest <= pairs ? n_tiles - rest : n_tiles);
  p.n_items = int(p.n_whole + 2 * (n_tiles - p.n_whole));
  const int grid = 2 * int(p.n_items < pairs ? p.n_items : pairs);
  const cudaError_t e = launch_dependent(
      qkv_proj_bf16_tc_kernel, dim3(unsigned(grid)), dim3(kThreads), kSmemBytes, a.stream, mx, mw,
      static_cast<__nv_bfloat16*>(a.Q), static_cast<__nv_bfloat16*>(a.K),
      static_cast<__nv_bfloat16*>(a.V), p, wait_limit_ns());
  if (e != cudaSuccess) {
    snprintf(msg, msglen, "projection launch: %s", cudaGetErrorString(e));
    return 5;
  }
  return 0;
}

cudaError_t proj_read_and_clear_status(unsigned* value) {
  cudaError_t e = cudaMemcpyFromSymbol(value, g_moa_proj_status, sizeof(unsigned));
  if (e != cudaSuccess) return e;
  const unsigned zero = 0;
  return cudaMemcpyToSymbol(g_moa_proj_status, &zero, sizeof(unsigned));
}

}  // namespace moa
