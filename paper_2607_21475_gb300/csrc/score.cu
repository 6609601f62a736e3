// E0: accumulated-attention importance scores (Appendix B of the paper,
// H2O-style accumulated attention from observation queries):
//     s_j = sum_r softmax_j(q_r . K^T / sqrt(d))
// over the R observation rows of a KV head's query group.
//
// Two passes per (batch row, KV head) unit:
//   pass 1  lse_r = log sum_j exp(q_r . k_j / sqrt(d))
//   pass 2  s_j   = sum_r exp(q_r . k_j / sqrt(d) - lse_r)
// Pass 2 owns each key column, so the sums are deterministic (no atomics).
// float32 inputs on 16-byte boundaries: score_lse_f32_kernel and
// score_col_f32_kernel, register-tiled products.  Anything else that the
// tensor-core kernels do not take (inputs off a 16-byte boundary): a warp per
// query row (score_lse_kernel) and a thread per key (score_col_kernel).
#include <cuda_runtime.h>
#include <math.h>

#include "common.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace ebd {

constexpr int kLseWarps = 8;
constexpr int kColThreads = 128;
constexpr int kColRows = 16;

template <typename T, int D>
__global__ void __launch_bounds__(kLseWarps * 32) score_lse_kernel(const T* __restrict__ q_obs,
                                                                   const T* __restrict__ K,
                                                                   int n_ctx, int n_obs,
                                                                   float* __restrict__ lse) {
  __shared__ float qs[kLseWarps][D];
  const int unit = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = blockIdx.y * kLseWarps + warp;
  const bool active = r < n_obs;
  const float scale = rsqrtf((float)D);
  if (active) {
    const T* q = q_obs + ((size_t)unit * n_obs + r) * D;
    for (int e = lane; e < D; e += 32) qs[warp][e] = to_f32(q[e]) * scale;
  }
  __syncwarp();
  if (!active) return;
  const T* Ku = K + (size_t)unit * n_ctx * D;
  float M = -INFINITY, S = 0.f;
  for (int j = lane; j < n_ctx; j += 32) {
    const T* kj = Ku + (size_t)j * D;
    float x = 0.f;
#pragma unroll 16
    for (int e = 0; e < D; ++e) x = fmaf(qs[warp][e], to_f32(kj[e]), x);
    if (x > M) {
      S = S * expf(M - x) + 1.f;
      M = x;
    } else {
      S += expf(x - M);
    }
  }
  // combine the lanes' (M, S)
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float Mo = __shfl_xor_sync(0xffffffffu, M, o);
    const float So = __shfl_xor_sync(0xffffffffu, S, o);
    const float Mn = fmaxf(M, Mo);
    S = (M == -INFINITY ? 0.f : S * expf(M - Mn)) + (Mo == -INFINITY ? 0.f : So * expf(Mo - Mn));
    M = Mn;
  }
  if (lane == 0) lse[(size_t)unit * n_obs + r] = M + logf(S);
}

template <typename T, int D>
__global__ void __launch_bounds__(kColThreads) score_col_kernel(const T* __restrict__ q_obs,
                                                                const T* __restrict__ K,
                                                                int n_ctx, int n_obs,
                                                                const float* __restrict__ lse,
                                                                float* __restrict__ scores) {
  extern __shared__ float smem[];
  float* ks = smem;                             // [kColThreads][D + 1]
  float* qs = smem + kColThreads * (D + 1);     // [kColRows][D]
  float* ls = qs + kColRows * D;                // [kColRows]
  const int unit = blockIdx.x;
  const int j0 = blockIdx.y * kColThreads;
  const int t = threadIdx.x;
  const float scale = rsqrtf((float)D);
  const T* Ku = K + (size_t)unit * n_ctx * D;
  for (int x = t; x < kColThreads * D; x += kColThreads) {
    const int row = x / D, e = x - row * D;
    const int j = j0 + row;
    ks[row * (D + 1) + e] = j < n_ctx ? to_f32(Ku[(size_t)j * D + e]) : 0.f;
  }
  float acc = 0.f;
  const T* Qu = q_obs + (size_t)unit * n_obs * D;
  for (int r0 = 0; r0 < n_obs; r0 += kColRows) {
    __syncthreads();
    for (int x = t; x < kColRows * D; x += kColThreads) {
      const int row = x / D, e = x - row * D;
      qs[x] = (r0 + row < n_obs) ? to_f32(Qu[(size_t)(r0 + row) * D + e]) * scale : 0.f;
    }
    for (int x = t; x < kColRows; x += kColThreads)
      ls[x] = (r0 + x < n_obs) ? lse[(size_t)unit * n_obs + r0 + x] : INFINITY;
    __syncthreads();
    const int nr = min(kColRows, n_obs - r0);
    for (int rr = 0; rr < nr; ++rr) {
      float x = 0.f;
#pragma unroll 16
      for (int e = 0; e < D; ++e) x = fmaf(qs[rr * D + e], ks[t * (D + 1) + e], x);
      acc += expf(x - ls[rr]);
    }
  }
  if (j0 + t < n_ctx) scores[(size_t)unit * n_ctx + j0 + t] = acc;
}

// ---------------------------------------------------------------------------
// float32, register tiles.  A CTA of four warps multiplies 8 I query rows (I =
// 4 or 8) by 128 keys, both row-major in shared memory (rows padded by 16
// bytes, so that 8 consecutive rows fall on different banks); a thread holds I
// x 8 logits, each as two partial sums over the even and the odd channels
// (f32x2 arithmetic straight on the 16-byte loads: no transposition, no
// packing).  Four channels take I + 8 loads of 16 bytes for 16 I two-wide
// FMAs: bound by the FMA pipe at I = 8, by shared memory at I = 4 (5.2 and 3.2
// us for 64 and 32 rows), which pass 1 takes where 64 rows would leave SMs
// idle.  In pass 1 the CTA keeps its query rows and streams key tiles through
// two buffers, a running (max, sum 2^(x - max)) of its own columns per thread,
// combined once at the end; clusters of CTAs split the keys.  In pass 2 it
// keeps its key tile and streams the query rows.
// Measured on 8 units x 128 rows x 2048 keys, d = 128: 36 us for both passes
// (22 + 16 alone; 30 TFLOP/s), where a warp per query row and a thread per key
// took 1045 + 92 us.
// ---------------------------------------------------------------------------
constexpr int kFKeys = 128;     // keys of a tile
constexpr int kFThreads = 128;  // 2 x 2 warps of 4 I rows x 64 keys

template <int D, int I>
struct F32Layout {
  static constexpr int kRows = 8 * I;    // query rows of a tile
  static constexpr int kStride = D + 4;  // floats per row
  static constexpr int kQ = kRows * kStride, kK = kFKeys * kStride;
  static constexpr int kLseBytes = (kQ + 2 * kK) * 4;
  static constexpr int kColBytes = (kK + 2 * kQ) * 4;
};

// Rows [row0, row0 + ROWS) of src (n_rows rows of D floats; zeros past them)
// to shared memory; the caller commits the group.
template <int D, int ROWS>
__device__ __forceinline__ void f32_copy_rows(float* dst, const float* src, int row0, int n_rows) {
#pragma unroll
  for (int n = 0; n < ROWS * D / 4 / kFThreads; ++n) {
    const int c = threadIdx.x + n * kFThreads;
    const int r = c / (D / 4), ch = c - r * (D / 4);
    const bool live = row0 + r < n_rows;
    cp_async16_zfill(dst + r * (D + 4) + 4 * ch,
                     src + (size_t)(live ? row0 + r : 0) * D + 4 * ch, live);
  }
}

// This thread's I x 8 products: rows q[4 i], keys k[8 j] (in rows of kStride).
template <int D, int I>
__device__ __forceinline__ void f32_tile(const float* q, const float* k, float (&x)[I][8]) {
  constexpr int S = D + 4;
  float2 acc[I][8];
#pragma unroll
  for (int i = 0; i < I; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int e = 0; e < D; e += 4) {
    float4 a[I], b[8];
#pragma unroll
    for (int i = 0; i < I; ++i) a[i] = *reinterpret_cast<const float4*>(q + 4 * i * S + e);
#pragma unroll
    for (int j = 0; j < 8; ++j) b[j] = *reinterpret_cast<const float4*>(k + 8 * j * S + e);
#pragma unroll
    for (int i = 0; i < I; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        acc[i][j] = __ffma2_rn(make_float2(a[i].x, a[i].y), make_float2(b[j].x, b[j].y), acc[i][j]);
        acc[i][j] = __ffma2_rn(make_float2(a[i].z, a[i].w), make_float2(b[j].z, b[j].w), acc[i][j]);
      }
  }
#pragma unroll
  for (int i = 0; i < I; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) x[i][j] = acc[i][j].x + acc[i][j].y;
}

// Merge (M2, S2) into the running (M, S) of raw logits, scaled by sc in base 2.
__device__ __forceinline__ void lse_merge(float& M, float& S, float M2, float S2, float sc) {
  const float mx = fmaxf(M, M2);
  S = (M == -INFINITY ? 0.f : S * exp2f((M - mx) * sc)) +
      (M2 == -INFINITY ? 0.f : S2 * exp2f((M2 - mx) * sc));
  M = mx;
}

template <int D, int I>
__global__ void __launch_bounds__(kFThreads) score_lse_f32_kernel(
    const float* q_obs, const float* K, int n_ctx, int n_obs, int rtiles,
    int csize, float sc, float* lse2) {
  using L = F32Layout<D, I>;
  extern __shared__ __align__(16) float fsm[];
  __shared__ float2 part[2][L::kRows];  // the two warp columns' parts of a row
  __shared__ float2 lead[8][L::kRows];  // the CTAs' parts, in CTA 0
  float* qs = fsm;
  float* ks = fsm + L::kQ;  // [2][kK]
  const int rank = csize > 1 ? (int)cluster_rank() : 0;
  if (csize > 1) cluster_arrive_started();
  const int rt = blockIdx.x / csize, unit = rt / rtiles, r0 = (rt - unit * rtiles) * L::kRows;
  const int nk_all = (n_ctx + kFKeys - 1) / kFKeys;
  const int k0 = (int)((long long)rank * nk_all / csize);
  const int nk = (int)((long long)(rank + 1) * nk_all / csize) - k0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = (warp >> 1) * 4 * I + (lane >> 3);
  const int col = (warp & 1) * 64 + (lane & 7);
  const float* Ku = K + (size_t)unit * n_ctx * D;
  // a programmatic dependent of whatever precedes it: nothing is read before
  // this, and pass 2 goes only after it
  grid_dependency_wait();
  grid_launch_dependents();
  f32_copy_rows<D, L::kRows>(qs, q_obs + (size_t)unit * n_obs * D, r0, n_obs);
  if (nk > 0) f32_copy_rows<D, kFKeys>(ks, Ku, k0 * kFKeys, n_ctx);
  cp_async_commit();
  float m[I], s[I];
#pragma unroll
  for (int i = 0; i < I; ++i) {
    m[i] = -INFINITY;
    s[i] = 0.f;
  }
  for (int t = 0; t < nk; ++t) {
    if (t + 1 < nk)
      f32_copy_rows<D, kFKeys>(ks + ((t + 1) & 1) * L::kK, Ku, (k0 + t + 1) * kFKeys, n_ctx);
    cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();
    float x[I][8];
    f32_tile<D, I>(qs + row * L::kStride, ks + (t & 1) * L::kK + col * L::kStride, x);
    const int left = n_ctx - (k0 + t) * kFKeys - col;  // key col + 8 j is inside while 8 j < left
#pragma unroll
    for (int i = 0; i < I; ++i) {
      float mx = m[i];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (8 * j >= left) x[i][j] = -INFINITY;
        mx = fmaxf(mx, x[i][j]);
      }
      if (mx == -INFINITY) continue;  // no key of this thread yet
      float sum = 0.f;
#pragma unroll
      for (int j = 0; j < 8; ++j) sum += exp2f((x[i][j] - mx) * sc);
      s[i] = s[i] * exp2f((m[i] - mx) * sc) + sum;
      m[i] = mx;
    }
    __syncthreads();  // this buffer is copied into next
  }
  cp_async_wait<0>();
#pragma unroll
  for (int i = 0; i < I; ++i) {
#pragma unroll
    for (int o = 1; o <= 4; o <<= 1) {
      const float mo = __shfl_xor_sync(0xffffffffu, m[i], o);
      const float so = __shfl_xor_sync(0xffffffffu, s[i], o);
      lse_merge(m[i], s[i], mo, so, sc);
    }
    if ((lane & 7) == 0) part[warp & 1][row + 4 * i] = make_float2(m[i], s[i]);
  }
  __syncthreads();
  const int r = threadIdx.x;
  float M = -INFINITY, S = 0.f;
  if (r < L::kRows) {
    M = part[0][r].x;
    S = part[0][r].y;
    lse_merge(M, S, part[1][r].x, part[1][r].y, sc);
  }
  if (csize > 1) {
    cluster_wait_acquire();  // CTA 0 runs
    if (r < L::kRows) {
      const uint32_t dst = cluster_map(smem_u32(&lead[rank][r]), 0);
      asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(dst), "f"(M), "f"(S)
                   : "memory");
    }
    cluster_barrier();
    if (rank != 0) return;
    if (r < L::kRows) {
      M = lead[0][r].x;
      S = lead[0][r].y;
      for (int c = 1; c < csize; ++c) lse_merge(M, S, lead[c][r].x, lead[c][r].y, sc);
    }
  }
  if (r < L::kRows && r0 + r < n_obs) lse2[(size_t)unit * n_obs + r0 + r] = M * sc + log2f(S);
}

template <int D, int I>
__global__ void __launch_bounds__(kFThreads) score_col_f32_kernel(
    const float* q_obs, const float* K, int n_ctx, int n_obs, int ktiles,
    float sc, const float* lse2, float* scores) {
  using L = F32Layout<D, I>;
  extern __shared__ __align__(16) float fsm[];
  __shared__ float part[2][kFKeys];  // the two warp rows' parts of a key's sum
  float* ks = fsm;
  float* qs = fsm + L::kK;  // [2][kQ]
  const int unit = blockIdx.x / ktiles, j0 = (blockIdx.x - unit * ktiles) * kFKeys;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = (warp >> 1) * 4 * I + (lane >> 3);
  const int col = (warp & 1) * 64 + (lane & 7);
  const float* Qu = q_obs + (size_t)unit * n_obs * D;
  const float* lu = lse2 + (size_t)unit * n_obs;
  const int nr = (n_obs + L::kRows - 1) / L::kRows;
  // the inputs were complete when pass 1 began
  f32_copy_rows<D, kFKeys>(ks, K + (size_t)unit * n_ctx * D, j0, n_ctx);
  f32_copy_rows<D, L::kRows>(qs, Qu, 0, n_obs);
  cp_async_commit();
  grid_dependency_wait();  // pass 1's log-sum-exps (and nothing is written before)
  float sum[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) sum[j] = 0.f;
  for (int t = 0; t < nr; ++t) {
    if (t + 1 < nr) f32_copy_rows<D, L::kRows>(qs + ((t + 1) & 1) * L::kQ, Qu, (t + 1) * L::kRows, n_obs);
    cp_async_commit();
    float ls[I];
#pragma unroll
    for (int i = 0; i < I; ++i) {
      const int r = t * L::kRows + row + 4 * i;
      ls[i] = r < n_obs ? lu[r] : INFINITY;
    }
    cp_async_wait<1>();
    __syncthreads();
    float x[I][8];
    f32_tile<D, I>(qs + (t & 1) * L::kQ + row * L::kStride, ks + col * L::kStride, x);
#pragma unroll
    for (int i = 0; i < I; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) sum[j] += exp2f(fmaf(x[i][j], sc, -ls[i]));
    __syncthreads();  // this buffer is copied into next
  }
  cp_async_wait<0>();
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    sum[j] += __shfl_xor_sync(0xffffffffu, sum[j], 8);
    sum[j] += __shfl_xor_sync(0xffffffffu, sum[j], 16);
    if (lane < 8) part[warp >> 1][col + 8 * j] = sum[j];
  }
  __syncthreads();
  const int c = threadIdx.x;
  if (c < kFKeys && j0 + c < n_ctx)
    scores[(size_t)unit * n_ctx + j0 + c] = part[0][c] + part[1][c];
}

// Launch as a programmatic dependent of what precedes it, on clusters of `cluster`.
template <typename Kernel, typename... Args>
static ebd_status launch_f32(Kernel kernel, long long grid, int cluster, int smem, cudaStream_t s,
                             Args... args) {
  if (grid > 0x7fffffffLL) return EBD_ERR_UNSUPPORTED;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
      cudaSuccess)
    return EBD_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kFThreads);
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
  return cuda_status(cudaLaunchKernelEx(&cfg, kernel, args...));
}

// Pass 1 with 8 I rows per tile: its cost in microseconds (waves x (start-up +
// key tiles at `tile_us`)) with the best split of the keys over C CTAs.
template <int D, int I>
static double plan_lse_f32(int units, int n_ctx, int n_obs, double tile_us, int& C) {
  const long long rts = (long long)units * ((n_obs + 8 * I - 1) / (8 * I));
  const int ktiles = (n_ctx + kFKeys - 1) / kFKeys;
  double best = 0.;
  for (int lg = 0; lg < 4; ++lg) {
    const int c = 1 << lg;
    if (lg > 0 && c > ktiles) break;
    // (at d = 64 two CTAs share an SM)
    constexpr int kSmem = F32Layout<D, I>::kLseBytes;
    const long long fit = resident_clusters<score_lse_f32_kernel<D, I>>(lg, kFThreads, kSmem, kSmem);
    const double cost = (double)((rts + fit - 1) / fit) * (3. + tile_us * ((ktiles + c - 1) / c));
    if (lg == 0 || cost < best) {
      best = cost;
      C = c;
    }
  }
  return best;
}

template <int D, int I>
static ebd_status launch_lse_f32(int units, int n_ctx, int n_obs, int C, const float* q,
                                 const float* k, float sc, float* lse, cudaStream_t s) {
  using L = F32Layout<D, I>;
  const int rtiles = (n_obs + L::kRows - 1) / L::kRows;
  const long long rts = (long long)units * rtiles;
  ebd_status st = launch_f32(score_lse_f32_kernel<D, I>, rts * C, C, L::kLseBytes, s, q, k, n_ctx,
                             n_obs, rtiles, C, sc, lse);
  if (st != EBD_OK && C > 1) {  // the cluster could not be placed: one CTA per row tile
    (void)cudaGetLastError();
    st = launch_f32(score_lse_f32_kernel<D, I>, rts, 1, L::kLseBytes, s, q, k, n_ctx, n_obs,
                    rtiles, 1, sc, lse);
  }
  return st;
}

template <int D>
static ebd_status launch_score_f32(int units, int n_ctx, int n_obs, const void* q_obs,
                                   const void* K, float* scores, float* lse, cudaStream_t s) {
  const float* q = (const float*)q_obs;
  const float* k = (const float*)K;
  const float sc = kLog2e / sqrtf((float)D);
  // per key tile at d = 128; half of it at 64
  int c8 = 1, c4 = 1;
  const double t8 = plan_lse_f32<D, 8>(units, n_ctx, n_obs, 5.2 * D / 128, c8);
  const double t4 = plan_lse_f32<D, 4>(units, n_ctx, n_obs, 3.2 * D / 128, c4);
  ebd_status st = t4 < t8 ? launch_lse_f32<D, 4>(units, n_ctx, n_obs, c4, q, k, sc, lse, s)
                          : launch_lse_f32<D, 8>(units, n_ctx, n_obs, c8, q, k, sc, lse, s);
  if (st != EBD_OK) return st;
  const int ktiles = (n_ctx + kFKeys - 1) / kFKeys;
  return launch_f32(score_col_f32_kernel<D, 8>, (long long)units * ktiles, 1,
                    F32Layout<D, 8>::kColBytes, s, q, k, n_ctx, n_obs, ktiles, sc,
                    (const float*)lse, scores);
}

template <typename T, int D>
static ebd_status launch_score_t(int units, int n_ctx, int n_obs, const void* q_obs,
                                 const void* K, float* scores, float* lse, cudaStream_t s) {
  dim3 g1(units, (n_obs + kLseWarps - 1) / kLseWarps);
  score_lse_kernel<T, D><<<g1, kLseWarps * 32, 0, s>>>((const T*)q_obs, (const T*)K, n_ctx, n_obs,
                                                       lse);
  ebd_status st = launch_status();
  if (st != EBD_OK) return st;
  const size_t smem = (size_t)(kColThreads * (D + 1) + kColRows * D + kColRows) * sizeof(float);
  if (cudaFuncSetAttribute(score_col_kernel<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)smem) != cudaSuccess)
    return EBD_ERR_CUDA;
  dim3 g2(units, (n_ctx + kColThreads - 1) / kColThreads);
  score_col_kernel<T, D><<<g2, kColThreads, smem, s>>>((const T*)q_obs, (const T*)K, n_ctx, n_obs,
                                                       lse, scores);
  return launch_status();
}

ebd_status launch_score(ebd_dtype dtype, int batch, int n_kv_heads, int head_dim, int n_ctx,
                        int n_obs, const void* q_obs, const void* K, float* scores,
                        float* lse_ws, int32_t* dev_status, cudaStream_t s) {
  const int units = batch * n_kv_heads;
  if (units > 0x7fffffff || n_obs > 4096 || n_obs < 1) return EBD_ERR_UNSUPPORTED;
  if (score_tc_supported(dtype, head_dim, n_obs, q_obs, K))
    return launch_score_tc(units, head_dim, n_ctx, n_obs, q_obs, K, scores, lse_ws, dev_status, s);
  if ((n_obs + kLseWarps - 1) / kLseWarps > 65535 || (n_ctx + kColThreads - 1) / kColThreads > 65535)
    return EBD_ERR_UNSUPPORTED;
  if (dtype == EBD_BF16) {
    if (head_dim == 128) return launch_score_t<__nv_bfloat16, 128>(units, n_ctx, n_obs, q_obs, K, scores, lse_ws, s);
    if (head_dim == 64) return launch_score_t<__nv_bfloat16, 64>(units, n_ctx, n_obs, q_obs, K, scores, lse_ws, s);
  } else if (dtype == EBD_F32) {
    if (aligned16(q_obs) && aligned16(K)) {
      if (head_dim == 128) return launch_score_f32<128>(units, n_ctx, n_obs, q_obs, K, scores, lse_ws, s);
      if (head_dim == 64) return launch_score_f32<64>(units, n_ctx, n_obs, q_obs, K, scores, lse_ws, s);
    }
    if (head_dim == 128) return launch_score_t<float, 128>(units, n_ctx, n_obs, q_obs, K, scores, lse_ws, s);
    if (head_dim == 64) return launch_score_t<float, 64>(units, n_ctx, n_obs, q_obs, K, scores, lse_ws, s);
  }
  return EBD_ERR_UNSUPPORTED;
}

}  // namespace ebd

using namespace ebd;

extern "C" size_t ebd_score_workspace_bytes(int32_t batch, int32_t n_kv_heads, int32_t n_obs) {
  if (batch < 1 || n_kv_heads < 1 || n_obs < 1) return 0;
  return align_up((size_t)batch * n_kv_heads * n_obs * sizeof(float), 256);
}

extern "C" ebd_status ebd_score(ebd_dtype dtype, int32_t batch, int32_t n_kv_heads,
                                int32_t head_dim, int32_t n_ctx, int32_t n_obs,
                                const void* q_obs, const void* K, float* scores, void* workspace,
                                size_t ws_bytes, void* stream) {
  if (batch < 1 || n_kv_heads < 1 || n_ctx < 1 || n_obs < 1 || !q_obs || !K || !scores)
    return EBD_ERR_INVALID;
  if (dtype != EBD_F32 && dtype != EBD_BF16) return EBD_ERR_INVALID;
  if (!workspace || ws_bytes < ebd_score_workspace_bytes(batch, n_kv_heads, n_obs))
    return EBD_ERR_CAPACITY;
  return launch_score(dtype, batch, n_kv_heads, head_dim, n_ctx, n_obs, q_obs, K, scores,
                      (float*)workspace, nullptr, (cudaStream_t)stream);
}
