// E0 on the 5th-generation tensor cores: accumulated attention mass
//     s_j = sum_r softmax_j(q_r . K^T / sqrt(d))
// (Appendix B harness, H2O-style accumulated attention from R observation
// query rows of a KV head's group), bf16 inputs, f32 accumulation in tensor
// memory, head_dim 64/128, R up to 4096.
//
// Pass 1, score_lse_tc_kernel: one CTA per (unit, 128 query rows), or a
// cluster of 2-8 CTAs that split the unit's keys where that leaves SMs idle
// otherwise.  The rows are the MMA's M (= tensor-memory lanes), 256-key tiles its N, so the
// accumulator S[128 x 256] = Q K^T holds one query row per lane and the
// epilogue thread that owns a lane keeps that row's running
// (max, sum 2^(x - max)) without any cross-thread traffic.  Two accumulators
// (256 columns each) alternate so the MMA of tile j + 1 overlaps the epilogue
// of tile j; three shared-memory stages of K let the copy of tile j + 2 start
// when the MMA of tile j - 1 is done.  Output: the base-2 log-sum-exp of
// every row (workspace).
// Pass 2, R <= 512, score_col_tc_kernel: the transposed product S^T = K Q^T,
// keys as M (one key per lane), all R query rows as N (split in two halves of <= 256
// columns, one per accumulator), so key j's thread sums 2^(x_rj - lse_r) over
// its own row.  A persistent grid walks (unit, 128-key tile) items in order,
// reloading Q only when the unit changes.
// Pass 2, R > 512, score_col_stream_tc_kernel: the same product with the query
// rows in chunks of at most 256 that stream through a ring (they no longer fit
// in shared memory beside K), a chunk per accumulator in turn.
//
// Both kernels are programmatic dependents: pass 1 of whatever precedes it
// (the query gather, say), pass 2 of pass 1.  Pass 1 waits before it reads
// anything and lets pass 2 go only then; so K and Q are complete when pass 2
// starts, and it loads them at once and waits only for the log-sum-exps
// (32 units x 448 rows x 6144 keys with the gather before them: 55.5 -> 52.5
// us).
//
// Roles (score_lse_tc_kernel, score_col_tc_kernel): warps 0-15 are the epilogue (warps w, w + 4, w + 8, w + 12 read
// tensor-memory lanes 32 (w % 4) .. + 31; in pass 1 warp w takes the 64
// columns from 64 (w / 4) on, in pass 2 every fourth 32-column chunk of the
// accumulator); warp 16 allocates tensor memory and one of its lanes
// issues the TMA copies (128-byte swizzle) and the tcgen05.mma instructions.
// Hand-offs use mbarriers: TMA -> MMA (transaction counts), MMA -> epilogue
// and MMA -> smem reuse (tcgen05.commit), epilogue -> MMA (512 arrivals).  The
// four warps of a lane quarter combine their parts of a row (pass 1) or of a
// key's sum (pass 2) through shared memory, in a fixed order.
// Every wait is bounded (~2 s); a timeout raises EBD_DEV_TIMEOUT, the roles
// leave their loops and the tensor memory is released.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>
#include <math.h>

#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "ptx.cuh"
#include "tcgen05.cuh"

namespace ebd {

constexpr int kTcRows1 = 128;   // pass 1: query rows per CTA (MMA M)
constexpr int kTcKeys1 = 256;   // pass 1: keys per tile (MMA N)
constexpr int kTcKeys2 = 128;   // pass 2: keys per tile (MMA M)
constexpr int kTcMaxRows = 512; // pass 2: query rows held as accumulator columns
constexpr int kTcGroups = 4;    // epilogue warps per tensor-memory lane quarter
constexpr int kTcEpi = 128 * kTcGroups;  // epilogue threads
constexpr int kTcThreads = kTcEpi + 32;  // + 1 issue warp
constexpr int kTcIssueWarp = kTcEpi / 32;
constexpr uint32_t kTmemCols = 512;

template <int D>
struct Tc1Layout {
  static constexpr int kHalves = D / 64;             // 64-column (128-byte) boxes
  static constexpr int kQBox = kTcRows1 * 128;       // 16 KB
  static constexpr int kKBox = kTcKeys1 * 128;       // 32 KB
  static constexpr int kKOff = kHalves * kQBox;
  static constexpr int kStages = 3;                  // K tiles in flight
  static constexpr int kBarOff = kKOff + kStages * kHalves * kKBox;
  // [groups][128][2] f32 of the final combine, over the K stages (all MMAs
  // have completed by then)
  static constexpr int kPartOff = kKOff;
  static constexpr int kLeadOff = kPartOff + kTcGroups * 128 * 8;  // [8][128][2] f32, in CTA 0
  static constexpr int kBytes = kBarOff + 16 * 8 + 1024;  // + alignment slack
};

template <int D>
struct Tc2Layout {
  static constexpr int kHalves = D / 64;
  static constexpr int kQBox = kTcMaxRows * 128;     // 64 KB (rows beyond R unused)
  static constexpr int kKBox = kTcKeys2 * 128;       // 16 KB
  static constexpr int kKOff = kHalves * kQBox;
  static constexpr int kLseOff = kKOff + 2 * kHalves * kKBox;  // [2][kTcMaxRows] f32
  static constexpr int kPartOff = kLseOff + 2 * kTcMaxRows * 4;  // [2][groups][128] f32
  static constexpr int kBarOff = kPartOff + 2 * kTcGroups * 128 * 4;
  static constexpr int kBytes = kBarOff + 16 * 8 + 1024;
};

struct TcArgs {
  int units;
  int n_ctx;     // N
  int n_obs;     // R
  int mtiles;    // pass 1: ceil(R / 128)
  int csize;     // pass 1: CTAs per (unit, 128 rows)
  int rows_pad;  // pass 2: R rounded up to 32
  int n_a;       // pass 2: accumulator A columns (<= 256)
  int n_b;       // pass 2: accumulator B columns (rows_pad - n_a)
  int blocks;    // streamed pass 2: ceil(R / 64), 64-row blocks
  int chunks;    // streamed pass 2: ceil(blocks / 4), chunks of at most 256 rows
  int items;     // pass 2: units * ceil(N / 128)
  float scale2;  // log2(e) / sqrt(d)
  float* lse2;   // [units, R] base-2 log-sum-exp (pass 1 out, pass 2 in)
  float* scores; // [units, N]
  int32_t* dev_status;
};

// max(a, b, c) in one instruction (three-input form of max.f32).
__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

__device__ __forceinline__ unsigned char* align1024(unsigned char* p) {
  return (unsigned char*)(((uintptr_t)p + 1023) & ~(uintptr_t)1023);
}

template <int D>
__global__ void __launch_bounds__(kTcThreads, 1)
    score_lse_tc_kernel(const __grid_constant__ CUtensorMap tmQ,
                        const __grid_constant__ CUtensorMap tmK, TcArgs a) {
  using L = Tc1Layout<D>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = align1024(smem_raw);
  constexpr int KS = L::kStages;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::kBarOff);
  uint64_t* q_full = bars;
  uint64_t* k_full = bars + 1;          // [KS]
  uint64_t* k_empty = k_full + KS;      // [KS]
  uint64_t* acc_full = k_empty + KS;    // [2]
  uint64_t* acc_empty = acc_full + 2;   // [2]
  uint64_t* mma_done = acc_empty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int C = a.csize;
  const int rank = C > 1 ? (int)cluster_rank() : 0;
  const int rt = blockIdx.x / C;
  const int unit = rt / a.mtiles, mt = rt - unit * a.mtiles;
  const int nk_all = (a.n_ctx + kTcKeys1 - 1) / kTcKeys1;
  const int k0 = (int)((long long)rank * nk_all / C);  // this CTA's key tiles
  const int nk = (int)((long long)(rank + 1) * nk_all / C) - k0;
  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    for (int s = 0; s < KS; ++s) {
      mbar_init(&k_full[s], 1);
      mbar_init(&k_empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&acc_full[s], 1);
      mbar_init(&acc_empty[s], kTcEpi);
    }
    mbar_init(mma_done, 1);
    fence_barrier_init();
  }
  if (warp == kTcIssueWarp) {
    tmem_alloc(tmem_slot, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  grid_dependency_wait();  // nothing is read before this
  grid_launch_dependents();
  bool ok = true;
  const int quarter = warp & 3, grp = warp >> 2;  // epilogue lane quarter, chunk group
  const int row = quarter * 32 + lane;
  float m = -INFINITY, ssum = 0.f;  // epilogue: raw max logit and sum 2^((x - m) scale2)

  if (warp == kTcIssueWarp) {
    if (lane == 0) {
      const int krow0 = unit * a.n_ctx;
      mbar_arrive_expect_tx(q_full, L::kHalves * L::kQBox);
#pragma unroll
      for (int h = 0; h < L::kHalves; ++h)
        tma_load_3d(smem + h * L::kQBox, &tmQ, h * 64, mt * kTcRows1, unit, q_full);
      auto load_k = [&](int j) {
        const int s = j % KS;
        mbar_arrive_expect_tx(&k_full[s], L::kHalves * L::kKBox);
#pragma unroll
        for (int h = 0; h < L::kHalves; ++h)
          tma_load_2d(smem + L::kKOff + (s * L::kHalves + h) * L::kKBox, &tmK, h * 64,
                      krow0 + (k0 + j) * kTcKeys1, &k_full[s]);
      };
      int issued = 0, consumed = 0;
      for (; issued < nk && issued < KS; ++issued) load_k(issued);
      const bool q_ok = mbar_wait_bounded(q_full, 0);
      ok = q_ok;
      const uint32_t idesc = umma_idesc_bf16_f32(128, kTcKeys1);
      const uint32_t qbase = smem_u32(smem);
      for (int j = 0; ok && j < nk; ++j) {
        const int s = j % KS, b = j & 1;  // K stage, accumulator
        if (!mbar_wait_bounded(&k_full[s], (j / KS) & 1)) {
          ok = false;
          break;
        }
        ++consumed;
        if (j >= 2 && !mbar_wait_bounded(&acc_empty[b], ((j - 2) >> 1) & 1)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t kbase = smem_u32(smem + L::kKOff + s * L::kHalves * L::kKBox);
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
          const uint32_t off = (uint32_t)((kk & 3) * 32);
          const uint64_t ad = umma_desc_k_sw128(qbase + (kk >> 2) * L::kQBox + off);
          const uint64_t bd = umma_desc_k_sw128(kbase + (kk >> 2) * L::kKBox + off);
          umma_bf16(tmem + b * kTcKeys1, ad, bd, idesc, kk > 0);
        }
        umma_commit(&k_empty[s]);
        umma_commit(&acc_full[b]);
        // the stage of tile j - 1 takes tile j - 1 + KS once its MMAs are done
        // (MMA j is queued behind them meanwhile)
        if (j >= 1 && issued < nk) {
          if (!mbar_wait_bounded(&k_empty[(j - 1) % KS], ((j - 1) / KS) & 1)) {
            ok = false;
            break;
          }
          load_k(issued++);
        }
      }
      // unwind: copies still in flight, then every MMA issued
      if (!q_ok) mbar_wait_bounded(q_full, 0);
      for (int t = consumed; t < issued; ++t) mbar_wait_bounded(&k_full[t % KS], (t / KS) & 1);
      umma_commit(mma_done);
      mbar_wait_bounded(mma_done, 0);
    }
    __syncwarp();
  } else {
    // epilogue: thread = query row (tensor-memory lane) x 64 keys of each tile
    const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
    const float sc = a.scale2;
    for (int j = 0; j < nk; ++j) {
      const int b = j & 1;
      if (!mbar_wait_bounded(&acc_full[b], (j >> 1) & 1)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const int kvalid = a.n_ctx - (k0 + j) * kTcKeys1;  // keys of this tile inside the unit
      // this warp's 64 keys (columns 64 grp ..) in one load, one wait, one
      // running-max update and one pass of exponentials
      const int nv = kvalid - grp * 64;
      if (nv > 0) {
        uint32_t r[64];
        tmem_ld64(tmem + lane_base + b * kTcKeys1 + grp * 64, r);
        tmem_ld_wait();
        if (nv < 64) {  // the unit's last keys: the rest belongs to the next unit
#pragma unroll
          for (int i = 0; i < 64; ++i)
            if (i >= nv) r[i] = __float_as_uint(-INFINITY);
        }
        float m4[4] = {__uint_as_float(r[0]), __uint_as_float(r[1]), __uint_as_float(r[2]),
                       __uint_as_float(r[3])};
#pragma unroll
        for (int i = 4; i < 64; i += 8) {
          m4[0] = fmax3(m4[0], __uint_as_float(r[i]), __uint_as_float(r[i + 1]));
          m4[1] = fmax3(m4[1], __uint_as_float(r[i + 2]), __uint_as_float(r[i + 3]));
          m4[2] = fmax3(m4[2], __uint_as_float(r[i + 4]), __uint_as_float(r[i + 5]));
          m4[3] = fmax3(m4[3], __uint_as_float(r[i + 6]), __uint_as_float(r[i + 7]));
        }
        const float cm = fmaxf(fmax3(m4[0], m4[1], m4[2]), m4[3]);
        if (cm > m) {
          ssum *= exp2f((m - cm) * sc);
          m = cm;
        }
        // 2^(x sc - m sc), two lanes of f32x2 arithmetic per instruction
        const float2 sc2 = make_float2(sc, sc), nmc = make_float2(-m * sc, -m * sc);
        float2 s2a = make_float2(0.f, 0.f), s2b = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < 64; i += 4) {
          const float2 ea = __ffma2_rn(make_float2(__uint_as_float(r[i]), __uint_as_float(r[i + 1])),
                                       sc2, nmc);
          const float2 eb = __ffma2_rn(
              make_float2(__uint_as_float(r[i + 2]), __uint_as_float(r[i + 3])), sc2, nmc);
          s2a = __fadd2_rn(s2a, make_float2(exp2f(ea.x), exp2f(ea.y)));
          s2b = __fadd2_rn(s2b, make_float2(exp2f(eb.x), exp2f(eb.y)));
        }
        ssum += (s2a.x + s2a.y) + (s2b.x + s2b.y);
      }
      tc_fence_before();
      mbar_arrive(&acc_empty[b]);
    }
  }
  // the four parts of each row meet in shared memory
  float* part = reinterpret_cast<float*>(smem + L::kPartOff);
  if (warp < kTcIssueWarp) {
    part[(grp * 128 + row) * 2] = m;
    part[(grp * 128 + row) * 2 + 1] = ssum;
  }
  __syncthreads();
  // the four parts of a row, then (C > 1) the CTAs' in rank order, in CTA 0; a
  // part without keys has M = -infinity
  auto combine = [&](const float* p, int n, float& M, float& tot) {
    M = -INFINITY;
    for (int q = 0; q < n; ++q) M = fmaxf(M, p[(q * 128 + row) * 2]);
    tot = 0.f;
    for (int q = 0; q < n; ++q) {
      const float m_q = p[(q * 128 + row) * 2];
      if (m_q != -INFINITY) tot += p[(q * 128 + row) * 2 + 1] * exp2f((m_q - M) * a.scale2);
    }
  };
  const bool combines = warp < kTcIssueWarp && grp == 0;
  float M = -INFINITY, tot = 0.f;
  if (combines) combine(part, kTcGroups, M, tot);
  if (C > 1) {
    float* lead = reinterpret_cast<float*>(smem + L::kLeadOff);
    cluster_barrier();  // CTA 0's K stages are free
    if (combines) {
      const uint32_t dst = cluster_map(smem_u32(lead + (rank * 128 + row) * 2), 0);
      asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(dst), "f"(M), "f"(tot)
                   : "memory");
    }
    cluster_barrier();
    if (combines && rank == 0) combine(lead, C, M, tot);
  }
  if (combines && rank == 0) {
    const int r = mt * kTcRows1 + row;
    if (ok && r < a.n_obs) a.lse2[(size_t)unit * a.n_obs + r] = M * a.scale2 + log2_near_one(tot);
  }
  if (!ok) raise_status(a.dev_status, EBD_DEV_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  if (warp == kTcIssueWarp) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

template <int D>
__global__ void __launch_bounds__(kTcThreads, 1)
    score_col_tc_kernel(const __grid_constant__ CUtensorMap tmQ,
                        const __grid_constant__ CUtensorMap tmK, TcArgs a) {
  using L = Tc2Layout<D>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = align1024(smem_raw);
  float* lse_s = reinterpret_cast<float*>(smem + L::kLseOff);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::kBarOff);
  uint64_t* q_full = bars;
  uint64_t* k_full = bars + 1;     // [2] key stages
  uint64_t* k_empty = bars + 3;    // [2]
  uint64_t* acc_full = bars + 5;   // [2] accumulator halves
  uint64_t* acc_empty = bars + 7;  // [2]
  uint64_t* lse_ready = bars + 9;   // the epilogue staged a unit's row log-sum-exps
  uint64_t* part_ready = bars + 10;  // [2] warps 4-15 left their partial key sums (item parity)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 12);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nkt = (a.n_ctx + kTcKeys2 - 1) / kTcKeys2;
  const int i0 = (int)((long long)blockIdx.x * a.items / gridDim.x);
  const int i1 = (int)((long long)(blockIdx.x + 1) * a.items / gridDim.x);
  const int n = i1 - i0;
  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(&k_full[s], 1);
      mbar_init(&k_empty[s], 1);
      mbar_init(&acc_full[s], 1);
      mbar_init(&acc_empty[s], kTcEpi);
    }
    mbar_init(lse_ready, kTcEpi);
    mbar_init(&part_ready[0], kTcEpi - 128);
    mbar_init(&part_ready[1], kTcEpi - 128);
    fence_barrier_init();
  }
  if (warp == kTcIssueWarp) {
    tmem_alloc(tmem_slot, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  bool ok = true;
  const int nq_loads = (a.rows_pad + 255) / 256;  // 256-row TMA boxes of Q

  if (warp == kTcIssueWarp) {
    if (lane == 0 && n > 0) {
      auto load_k = [&](int i) {
        const int item = i0 + i, u = item / nkt, kt = item - u * nkt;
        const int s = i & 1;
        mbar_arrive_expect_tx(&k_full[s], L::kHalves * L::kKBox);
#pragma unroll
        for (int h = 0; h < L::kHalves; ++h)
          tma_load_2d(smem + L::kKOff + (s * L::kHalves + h) * L::kKBox, &tmK, h * 64,
                      u * a.n_ctx + kt * kTcKeys2, &k_full[s]);
      };
      const uint32_t idesc_a = umma_idesc_bf16_f32(128, a.n_a);
      const uint32_t idesc_b = umma_idesc_bf16_f32(128, a.n_b > 0 ? a.n_b : 16);
      const uint32_t qbase = smem_u32(smem);
      int cur_u = -1, qloads = 0;
      bool qwait = false;
      load_k(0);
      for (int i = 0; ok && i < n; ++i) {
        const int item = i0 + i, u = item / nkt;
        const int s = i & 1;
        if (u != cur_u) {  // new unit: Q once every MMA reading the old one is done
          if (i > 0 && !mbar_wait_bounded(&k_empty[s ^ 1], ((i - 1) >> 1) & 1)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(q_full, L::kHalves * nq_loads * 256 * 128);
#pragma unroll
          for (int h = 0; h < L::kHalves; ++h)
            for (int l = 0; l < nq_loads; ++l)
              tma_load_3d(smem + h * L::kQBox + l * 256 * 128, &tmQ, h * 64, l * 256, u, q_full);
          cur_u = u;
          qwait = true;
        }
        if (i + 1 < n) {
          if (i >= 1 && !mbar_wait_bounded(&k_empty[s ^ 1], ((i - 1) >> 1) & 1)) {
            ok = false;
            break;
          }
          load_k(i + 1);
        }
        if (!mbar_wait_bounded(&k_full[s], (i >> 1) & 1)) {
          ok = false;
          break;
        }
        if (qwait) {
          if (!mbar_wait_bounded(q_full, qloads & 1)) {
            ok = false;
            break;
          }
          ++qloads;
          qwait = false;
        }
        const uint32_t kbase = smem_u32(smem + L::kKOff + s * L::kHalves * L::kKBox);
        for (int hh = 0; hh < 2; ++hh) {
          const int ncols = hh == 0 ? a.n_a : a.n_b;
          if (ncols == 0) continue;
          if (i >= 1 && !mbar_wait_bounded(&acc_empty[hh], (i - 1) & 1)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t row_off = (uint32_t)(hh * a.n_a) * 128u;  // first query row of the half
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk) {
            const uint32_t off = (uint32_t)((kk & 3) * 32);
            const uint64_t ad = umma_desc_k_sw128(kbase + (kk >> 2) * L::kKBox + off);
            const uint64_t bd = umma_desc_k_sw128(qbase + (kk >> 2) * L::kQBox + row_off + off);
            umma_bf16(tmem + hh * 256, ad, bd, hh == 0 ? idesc_a : idesc_b, kk > 0);
          }
          umma_commit(&acc_full[hh]);
        }
        if (!ok) break;
        umma_commit(&k_empty[s]);
      }
    }
    __syncwarp();
  } else {
    // epilogue: thread = key (tensor-memory lane); the 32-column chunks of the
    // [A | B] accumulator columns go round-robin to warps w, w + 4, w + 8, w + 12
    const int quarter = warp & 3, grp = warp >> 2;
    const int row = quarter * 32 + lane;
    const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
    float* part = reinterpret_cast<float*>(smem + L::kPartOff);
    const int nch = a.rows_pad / 32;
    grid_dependency_wait();  // pass 1's log-sum-exps are complete (and nothing is written before)
    int cur_u = -1, par = 0, changes = 0;
    for (int i = 0; i < n; ++i) {
      const int item = i0 + i, u = item / nkt, kt = item - u * nkt;
      if (u != cur_u) {  // this unit's row log-sum-exps (padding rows contribute 0)
        par ^= 1;
        float* ls = lse_s + par * kTcMaxRows;
        for (int r = threadIdx.x; r < a.rows_pad; r += kTcEpi)
          ls[r] = r < a.n_obs ? -a.lse2[(size_t)u * a.n_obs + r] : -INFINITY;
        mbar_arrive(lse_ready);  // release: the rows this thread staged
        if (!mbar_wait_bounded(lse_ready, changes & 1)) {
          ok = false;
          break;
        }
        ++changes;
        cur_u = u;
      }
      const float* ls = lse_s + par * kTcMaxRows;  // minus the row log-sum-exps
      const float2 sc2 = make_float2(a.scale2, a.scale2);
      float2 s2a = make_float2(0.f, 0.f), s2b = make_float2(0.f, 0.f);
      for (int hh = 0; hh < 2; ++hh) {
        const int ncols = hh == 0 ? a.n_a : a.n_b;
        if (ncols == 0) continue;
        if (!mbar_wait_bounded(&acc_full[hh], i & 1)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const int c0 = hh == 0 ? 0 : a.n_a / 32, c1 = hh == 0 ? a.n_a / 32 : nch;
        // first chunk c >= c0 with c % groups == grp
        const int cfirst = c0 + ((grp - c0 % kTcGroups) + kTcGroups) % kTcGroups;
#pragma unroll 1
        for (int c = cfirst; c < c1; c += kTcGroups) {
          uint32_t r[32];
          tmem_ld32(tmem + lane_base + hh * 256 + (c - c0) * 32, r);
          tmem_ld_wait();
          const float4* l4 = reinterpret_cast<const float4*>(ls + c * 32);
#pragma unroll
          for (int t = 0; t < 8; ++t) {
            const float4 lv = l4[t];
            const float2 ea = __ffma2_rn(make_float2(__uint_as_float(r[4 * t]),
                                                     __uint_as_float(r[4 * t + 1])),
                                         sc2, make_float2(lv.x, lv.y));
            const float2 eb = __ffma2_rn(make_float2(__uint_as_float(r[4 * t + 2]),
                                                     __uint_as_float(r[4 * t + 3])),
                                         sc2, make_float2(lv.z, lv.w));
            s2a = __fadd2_rn(s2a, make_float2(exp2f(ea.x), exp2f(ea.y)));
            s2b = __fadd2_rn(s2b, make_float2(exp2f(eb.x), exp2f(eb.y)));
          }
        }
        tc_fence_before();
        mbar_arrive(&acc_empty[hh]);
      }
      if (!ok) break;
      const float sum = (s2a.x + s2a.y) + (s2b.x + s2b.y);
      float* pb = part + (i & 1) * kTcGroups * 128;
      if (grp != 0) {
        pb[grp * 128 + row] = sum;
        mbar_arrive(&part_ready[i & 1]);  // release
      } else {
        // one barrier per buffer: an arrival for item i + 1 can never count
        // toward item i's phase
        if (!mbar_wait_bounded(&part_ready[i & 1], (i >> 1) & 1)) {
          ok = false;
          break;
        }
        float tot = sum;
#pragma unroll
        for (int q = 1; q < kTcGroups; ++q) tot += pb[q * 128 + row];
        const int key = kt * kTcKeys2 + row;
        if (key < a.n_ctx) a.scores[(size_t)u * a.n_ctx + key] = tot;
      }
    }
  }
  if (!ok) raise_status(a.dev_status, EBD_DEV_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  if (warp == kTcIssueWarp) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

// ---------------------------------------------------------------------------
// Pass 2 for more than 512 query rows.  Warps 0-15 are the epilogue (quarter
// w / 4 of an accumulator's columns, in one tensor-memory load, after which
// the accumulator is handed back and its next MMA runs under the
// exponentials); one lane of warp 16 issues the MMAs, one of warp 17 the
// copies.  Bound by the exponentials and the sums around them (without them
// the pass takes 17.8 us): 24 us on 8 units x 1024 rows x 8189 keys, d = 128
// (0.7 PFLOP/s), where mma.sync on 64-key tiles took 98 us.
// ---------------------------------------------------------------------------
constexpr int kTsCols = 256;     // columns of one accumulator (MMA N, at most)
constexpr int kTsSlots = 2;      // accumulators
constexpr int kTsMaxRows = 4096; // query rows of a unit
constexpr int kTsQBoxRows = 64;  // rows of one TMA box of Q
constexpr int kTsParts = 4;      // items whose quarter sums may be pending
constexpr int kTsMmaWarp = kTcEpi / 32;
constexpr int kTsTmaWarp = kTsMmaWarp + 1;
constexpr int kTsThreads = kTcEpi + 64;

template <int D>
struct TsLayout {
  static constexpr int kHalves = D / 64;
  static constexpr int kQStages = 2;                 // chunks of query rows in flight
  static constexpr int kQBox = kTsCols * 128;        // 32 KB
  static constexpr int kKBox = kTcKeys2 * 128;       // 16 KB
  static constexpr int kKStages = 2;
  static constexpr int kKOff = kQStages * kHalves * kQBox;
  static constexpr int kLseOff = kKOff + kKStages * kHalves * kKBox;  // [kTsMaxRows] f32
  static constexpr int kPartOff = kLseOff + kTsMaxRows * 4;  // [kTsParts][groups][128] f32
  static constexpr int kBarOff = kPartOff + kTsParts * kTcGroups * 128 * 4;
  static constexpr int kBytes = kBarOff + 32 * 8 + 1024;
};
static_assert(TsLayout<128>::kBytes <= 227 * 1024, "shared memory of one CTA");

// D[tmem] = A B^T over the whole head dimension (K-major tiles in 64-column
// boxes of a_box / b_box bytes).
template <int D>
__device__ __forceinline__ void mma_tile(uint32_t d_tmem, uint32_t abase, int a_box,
                                         uint32_t bbase, int b_box, uint32_t idesc) {
#pragma unroll
  for (int kk = 0; kk < D / 16; ++kk) {
    const uint32_t off = (uint32_t)((kk & 3) * 32);
    umma_bf16(d_tmem, umma_desc_k_sw128(abase + (kk >> 2) * a_box + off),
              umma_desc_k_sw128(bbase + (kk >> 2) * b_box + off), idesc, kk > 0);
  }
}

// 2^x; volatile, so that the compiler keeps a run of them together.
__device__ __forceinline__ float ex2(float x) {
  float r;
  asm volatile("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Sum of 2^(x sc + add) over NC columns; `r` is used up.  In three sweeps over
// the registers, so that a warp issues its exponentials one after another:
// taken four at a time with their sums between them, each four waited for the
// last (measured: 5.4 instead of 7.0 exponentials per clock and scheduler with
// two warps on it).
template <int NC, typename Add>
__device__ __forceinline__ float exp_sum(uint32_t (&r)[NC], float sc, Add add) {
  const float2 sc2 = make_float2(sc, sc);
  float2 e[NC / 2];
#pragma unroll
  for (int t = 0; t < NC / 4; ++t) {
    const float4 av = add(t);
    e[2 * t] = __ffma2_rn(make_float2(__uint_as_float(r[4 * t]), __uint_as_float(r[4 * t + 1])),
                          sc2, make_float2(av.x, av.y));
    e[2 * t + 1] = __ffma2_rn(
        make_float2(__uint_as_float(r[4 * t + 2]), __uint_as_float(r[4 * t + 3])), sc2,
        make_float2(av.z, av.w));
  }
#pragma unroll
  for (int t = 0; t < NC / 2; ++t) e[t] = make_float2(ex2(e[t].x), ex2(e[t].y));
#pragma unroll
  for (int t = 8; t < NC / 2; ++t) e[t & 7] = __fadd2_rn(e[t & 7], e[t]);
#pragma unroll
  for (int w = 4; w > 0; w >>= 1)
#pragma unroll
    for (int t = 0; t < w; ++t) e[t] = __fadd2_rn(e[t], e[t + w]);
  return e[0].x + e[0].y;
}

template <int D>
__global__ void __launch_bounds__(kTsThreads, 1)
    score_col_stream_tc_kernel(const __grid_constant__ CUtensorMap tmQ,
                        const __grid_constant__ CUtensorMap tmK, TcArgs a) {
  using L = TsLayout<D>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = align1024(smem_raw);
  constexpr int QS = L::kQStages, KS = L::kKStages;
  float* lse_s = reinterpret_cast<float*>(smem + L::kLseOff);
  float* part = reinterpret_cast<float*>(smem + L::kPartOff);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::kBarOff);
  uint64_t* q_full = bars;                    // [2]
  uint64_t* q_empty = bars + 2;               // [2]
  uint64_t* acc_full = bars + 4;              // [slots]
  uint64_t* acc_empty = bars + 6;             // [slots]
  uint64_t* k_full = bars + 8;                // [KS]
  uint64_t* k_empty = bars + 12;              // [KS]
  uint64_t* part_full = bars + 16;            // [kTsParts] the other quarters' sums of an item
  uint64_t* part_empty = bars + 20;           // [kTsParts]
  uint64_t* lse_sync = bars + 24;             // epilogue threads, twice per unit
  uint64_t* mma_done = bars + 25;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 26);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nkt = (a.n_ctx + kTcKeys2 - 1) / kTcKeys2;
  const int i0 = (int)((long long)blockIdx.x * a.items / gridDim.x);
  const int i1 = (int)((long long)(blockIdx.x + 1) * a.items / gridDim.x);
  const int n = i1 - i0;
  const int nch = a.chunks;
  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(&q_full[s], 1);
      mbar_init(&q_empty[s], 1);
      mbar_init(&acc_full[s], 1);
      mbar_init(&acc_empty[s], kTcEpi);
    }
    for (int s = 0; s < KS; ++s) {
      mbar_init(&k_full[s], 1);
      mbar_init(&k_empty[s], 1);
    }
    for (int s = 0; s < kTsParts; ++s) {
      mbar_init(&part_full[s], kTcEpi - 128);
      mbar_init(&part_empty[s], 128);
    }
    mbar_init(lse_sync, kTcEpi);
    mbar_init(mma_done, 1);
    fence_barrier_init();
  }
  if (warp == kTsMmaWarp) {
    tmem_alloc(tmem_slot, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  bool ok = true;
  // chunk c of the query rows: 64-row blocks [block0(c), block0(c + 1))
  auto block0 = [&](int c) { return c * a.blocks / nch; };

  if (warp == kTsTmaWarp) {
    // K and Q were complete when pass 1 began: nothing to wait for
    if (lane == 0) {
      int t = 0, ki = 0;  // chunks and K tiles issued
      for (int i = 0; ok && i < n; ++i) {
        const int item = i0 + i, u = item / nkt, kt = item - u * nkt;
        const int s = i % KS;
        if (i >= KS && !mbar_wait_bounded(&k_empty[s], (i / KS - 1) & 1)) {
          ok = false;
          break;
        }
        mbar_arrive_expect_tx(&k_full[s], L::kHalves * L::kKBox);
#pragma unroll
        for (int h = 0; h < L::kHalves; ++h)
          tma_load_2d(smem + L::kKOff + (s * L::kHalves + h) * L::kKBox, &tmK, h * 64,
                      u * a.n_ctx + kt * kTcKeys2, &k_full[s]);
        ++ki;
        auto load_q = [&](int stage, int pa, int pb) {
          mbar_arrive_expect_tx(&q_full[stage], L::kHalves * (pb - pa) * kTsQBoxRows * 128);
#pragma unroll
          for (int h = 0; h < L::kHalves; ++h)
            for (int p = pa; p < pb; ++p)
              tma_load_3d(smem + (stage * L::kHalves + h) * L::kQBox +
                              (p - pa) * kTsQBoxRows * 128,
                          &tmQ, h * 64, p * kTsQBoxRows, u, &q_full[stage]);
        };
        for (int c = 0; c < nch; ++c, ++t) {
          const int qs = t % QS;
          if (t >= QS && !mbar_wait_bounded(&q_empty[qs], (t / QS - 1) & 1)) {
            ok = false;
            break;
          }
          load_q(qs, block0(c), block0(c + 1));
        }
      }
      // never leave with copies in flight into shared memory
      for (int x = t > QS ? t - QS : 0; x < t; ++x)
        mbar_wait_bounded(&q_full[x % QS], (x / QS) & 1);
      for (int x = ki > KS ? ki - KS : 0; x < ki; ++x)
        mbar_wait_bounded(&k_full[x % KS], (x / KS) & 1);
    }
    __syncwarp();
  } else if (warp == kTsMmaWarp) {
    if (lane == 0) {
      const uint32_t qbase = smem_u32(smem);
      int t = 0;
      for (int i = 0; ok && i < n; ++i) {
        const int s = i % KS;
        if (!mbar_wait_bounded(&k_full[s], (i / KS) & 1)) {
          ok = false;
          break;
        }
        const uint32_t kbase = smem_u32(smem + L::kKOff + s * L::kHalves * L::kKBox);
        for (int c = 0; c < nch; ++c, ++t) {
          const int b = t % kTsSlots, qs = t % QS;
          const int rows = (block0(c + 1) - block0(c)) * kTsQBoxRows;
          if (!mbar_wait_bounded(&q_full[qs], (t / QS) & 1) ||
              (t >= kTsSlots && !mbar_wait_bounded(&acc_empty[b], (t / kTsSlots - 1) & 1))) {
            ok = false;
            break;
          }
          tc_fence_after();
          mma_tile<D>(tmem + b * kTsCols, kbase, L::kKBox,
                      qbase + qs * L::kHalves * L::kQBox, L::kQBox,
                      umma_idesc_bf16_f32(128, rows));
          umma_commit(&acc_full[b]);
          umma_commit(&q_empty[qs]);
        }
        if (!ok) break;
        umma_commit(&k_empty[s]);
      }
      umma_commit(mma_done);  // every MMA issued has completed before the end
      mbar_wait_bounded(mma_done, 0);
    }
    __syncwarp();
  } else {
    // epilogue: thread = key (tensor-memory lane), a quarter of each chunk's rows
    grid_dependency_wait();  // pass 1's log-sum-exps are complete (and nothing is written before)
    const int quarter = warp & 3, party = warp >> 2;
    const int row = quarter * 32 + lane;
    const uint32_t tlane = tmem + ((uint32_t)(quarter * 32) << 16);
    int cur_u = -1, syncs = 0, t = 0;
    for (int i = 0; ok && i < n; ++i) {
      const int item = i0 + i, u = item / nkt, kt = item - u * nkt;
      if (u != cur_u) {  // this unit's row log-sum-exps (padding rows contribute 0)
        for (int step = 0; step < 2; ++step) {
          if (step == 1)
            for (int r = threadIdx.x; r < a.blocks * 64; r += kTcEpi)
              lse_s[r] = r < a.n_obs ? -a.lse2[(size_t)u * a.n_obs + r] : -INFINITY;
          // every warp is done with the old unit's rows; the new ones are in
          mbar_arrive(lse_sync);
          if (!mbar_wait_bounded(lse_sync, syncs & 1)) {
            ok = false;
            break;
          }
          ++syncs;
        }
        if (!ok) break;
        cur_u = u;
      }
      float sum = 0.f;
      for (int c = 0; c < nch; ++c, ++t) {
        const int b = t % kTsSlots;
        if (!mbar_wait_bounded(&acc_full[b], (t / kTsSlots) & 1)) {
          ok = false;
          break;
        }
        tc_fence_after();
        // this quarter's 48 or 64 columns of the chunk: nine blocks or more in
        // ceil(blocks / 4) chunks are three or four each
        const int pc = block0(c), nb = block0(c + 1) - pc;
        const uint32_t tbase = tlane + b * kTsCols + party * 16 * nb;
        const float4* l4 = reinterpret_cast<const float4*>(lse_s + pc * 64 + party * 16 * nb);
        auto take = [&](auto n) {
          uint32_t r[decltype(n)::value];
          tmem_read(tbase, r);
          tc_fence_before();
          mbar_arrive(&acc_empty[b]);
          sum += exp_sum(r, a.scale2, [&](int q) { return l4[q]; });
        };
        if (nb == 4) take(std::integral_constant<int, 64>{});
        else take(std::integral_constant<int, 48>{});
      }
      if (!ok) break;
      // the first quarter's warps add the four parts, in order
      const int slot = i % kTsParts, use = i / kTsParts;
      float* pb = part + slot * kTcGroups * 128;
      if (party != 0) {
        if (use > 0 && !mbar_wait_bounded(&part_empty[slot], (use - 1) & 1)) {
          ok = false;
          break;
        }
        pb[party * 128 + row] = sum;
        mbar_arrive(&part_full[slot]);  // release
        continue;
      }
      if (!mbar_wait_bounded(&part_full[slot], use & 1)) {
        ok = false;
        break;
      }
#pragma unroll
      for (int q = 1; q < kTcGroups; ++q) sum += pb[q * 128 + row];
      mbar_arrive(&part_empty[slot]);
      const int key = kt * kTcKeys2 + row;
      if (key < a.n_ctx) a.scores[(size_t)u * a.n_ctx + key] = sum;
    }
  }
  if (!ok) raise_status(a.dev_status, EBD_DEV_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  if (warp == kTsMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
static PFN_cuTensorMapEncodeTiled_v12000 tc_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// [units, rows, D] bf16, box = 64 columns x box_rows rows of one unit, 128-byte
// swizzle.  Rows past a unit's last read as zeros: an accumulator column of
// the padding adds 2^(0 - infinity) = 0, whatever the next unit's rows hold (a
// NaN there would reach this unit's sums).
static bool encode_bf16_units(CUtensorMap* map, const void* base, int units, int rows, int D,
                              int box_rows) {
  auto enc = tc_encoder();
  if (!enc) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)rows, (cuuint64_t)units};
  const cuuint64_t strides[2] = {(cuuint64_t)D * 2, (cuuint64_t)rows * D * 2};
  const cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box,
             estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// [rows, D] bf16 as 2D; box = 64 columns x box_rows rows, 128-byte swizzle.
static bool encode_bf16_rows(CUtensorMap* map, const void* base, long long rows, int D,
                             int box_rows) {
  auto enc = tc_encoder();
  if (!enc) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)D, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)D * 2};
  const cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
             estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool score_tc_supported(ebd_dtype dtype, int head_dim, int n_obs, const void* q_obs,
                        const void* K) {
  return dtype == EBD_BF16 && (head_dim == 64 || head_dim == 128) && n_obs >= 1 &&
         n_obs <= kTsMaxRows && ((uintptr_t)q_obs & 15u) == 0 && ((uintptr_t)K & 15u) == 0 &&
         tc_encoder() != nullptr;
}

// One E0 kernel as a programmatic dependent of what precedes it, on clusters
// of `cluster` CTAs.
template <typename Kernel>
static ebd_status launch_tc_kernel(Kernel kernel, int grid, int threads, int cluster, int smem,
                                   cudaStream_t s,
                                   const CUtensorMap& tmQ, const CUtensorMap& tmK,
                                   const TcArgs& a) {
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
      cudaSuccess)
    return EBD_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cuda_status(cudaLaunchKernelEx(&cfg, kernel, tmQ, tmK, a));
}

template <int D>
static ebd_status launch_score_tc_t(int units, int n_ctx, int n_obs, const void* q_obs,
                                    const void* K, float* scores, float* lse2,
                                    int32_t* dev_status, cudaStream_t s) {
  const bool stream = n_obs > kTcMaxRows;
  CUtensorMap tmQ1, tmK1, tmQ2, tmK2;
  const long long krows = (long long)units * n_ctx;
  if (!encode_bf16_units(&tmQ1, q_obs, units, n_obs, D, kTcRows1) ||
      !encode_bf16_rows(&tmK1, K, krows, D, kTcKeys1) ||
      !encode_bf16_units(&tmQ2, q_obs, units, n_obs, D, stream ? kTsQBoxRows : 256) ||
      !encode_bf16_rows(&tmK2, K, krows, D, kTcKeys2))
    return EBD_ERR_CUDA;
  TcArgs a;
  a.units = units;
  a.n_ctx = n_ctx;
  a.n_obs = n_obs;
  a.mtiles = (n_obs + kTcRows1 - 1) / kTcRows1;
  a.rows_pad = (n_obs + 31) / 32 * 32;
  a.n_a = a.rows_pad < 256 ? a.rows_pad : 256;
  a.n_b = a.rows_pad - a.n_a;
  a.blocks = (n_obs + kTsQBoxRows - 1) / kTsQBoxRows;
  a.chunks = (a.blocks * kTsQBoxRows + kTsCols - 1) / kTsCols;
  a.items = units * ((n_ctx + kTcKeys2 - 1) / kTcKeys2);
  a.scale2 = kLog2e / sqrtf((float)D);
  a.lse2 = lse2;
  a.scores = scores;
  a.dev_status = dev_status;
  // pass 1: the keys of a row tile over 2, 4 or 8 CTAs while that still fits
  // one wave and leaves each at least 4 key tiles (a split of fewer is all
  // start-up: the query tile, the first key tile and the cluster's combine).
  // 8 units x 1024 rows x 8189 keys on 128 instead of 64 CTAs: 18.7 us
  const int nk = (n_ctx + kTcKeys1 - 1) / kTcKeys1;
  const int smem1 = Tc1Layout<D>::kBytes;
  int C = 1;
  for (int lg = 1; lg < 4 && nk >= 4 << lg &&
                   (long long)units * a.mtiles <=
                       resident_clusters<score_lse_tc_kernel<D>>(lg, kTcThreads, smem1, smem1);
       ++lg)
    C = 1 << lg;
  a.csize = C;
  ebd_status st = launch_tc_kernel(score_lse_tc_kernel<D>, units * a.mtiles * C, kTcThreads, C,
                                   smem1, s, tmQ1, tmK1, a);
  if (st != EBD_OK && C > 1) {  // the cluster could not be placed: one CTA per row tile
    (void)cudaGetLastError();
    a.csize = 1;
    st = launch_tc_kernel(score_lse_tc_kernel<D>, units * a.mtiles, kTcThreads, 1, smem1, s, tmQ1,
                          tmK1, a);
  }
  if (st != EBD_OK) return st;
  const int ctas = a.items < sm_count() ? a.items : sm_count();
  if (stream)
    return launch_tc_kernel(score_col_stream_tc_kernel<D>, ctas, kTsThreads, 1,
                            TsLayout<D>::kBytes, s, tmQ2, tmK2, a);
  return launch_tc_kernel(score_col_tc_kernel<D>, ctas, kTcThreads, 1, Tc2Layout<D>::kBytes, s,
                          tmQ2, tmK2, a);
}

ebd_status launch_score_tc(int units, int head_dim, int n_ctx, int n_obs, const void* q_obs,
                           const void* K, float* scores, float* lse, int32_t* dev_status,
                           cudaStream_t s) {
  if ((long long)units * n_ctx >= 0x7fffffffLL || (long long)units * n_obs >= 0x7fffffffLL)
    return EBD_ERR_UNSUPPORTED;
  if (head_dim == 128)
    return launch_score_tc_t<128>(units, n_ctx, n_obs, q_obs, K, scores, lse, dev_status, s);
  if (head_dim == 64)
    return launch_score_tc_t<64>(units, n_ctx, n_obs, q_obs, K, scores, lse, dev_status, s);
  return EBD_ERR_UNSUPPORTED;
}

}  // namespace ebd
