// CUDA-core decode of a float32 compact cache, and the second pass over any
// compact cache in float32: per-token variance contributions, or the exact range
// term (Eq. 3, Theorem 2, Eq. 4; head_dim 64/128, at most 8 query heads).
//
// A CTA of four warps takes a run of 32-token tiles of one unit, streamed by
// 16-byte cp.async into two buffers of K and V (rows padded by 16 bytes, so that
// 8 consecutive rows fall on different banks).
//
// Decode, per tile: a lane is a token and forms its logits with one or two
// heads' queries (read once for all lanes) and a quarter of ||v - c||^2; a lane
// is a token of one head and turns its logit into (w, u = (1 - pi) w^2), with
// its own sums of w, u, u ||v - c||^2 and maxima, added over the lanes once at the
// end; a thread is a channel and adds (w, u) v over the tile's tokens for every
// head, two-wide.  No shuffles over channels, and one exponential per token and
// head.  One partial record per (unit, split, head), merged by
// decode_reduce_kernel.  Bound by shared-memory reads (about 50 cycles a token at
// 8 heads, d = 128; HBM brings one in 45).
//
// Second pass, per tile: a lane is a token and forms, for one or two heads,
// p = w / N_hat and ||v - y_hat||^2 from the differences.
//
// Measured, against a warp per token with its channels over the lanes: decode with
// the exact range term, 4 units x 3 heads x 28457 rows of 64 channels, 165 -> 45
// us; contributions and block scores of 104 units x 2 heads x 1741 rows of 128,
// 96 -> 48 us; a 512-token layer of 4 heads (with its eviction) 26.6 -> 16.6 us.
#include <cuda_runtime.h>
#include <math.h>

#include <type_traits>

#include "common.cuh"
#include "decode.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace ebd {

constexpr int kCoreTile = 32;
constexpr int kCoreThreads = 128;
constexpr int kCoreWarps = kCoreThreads / 32;
constexpr int kCoreHeads = 8;
constexpr int kCoreCtasPerSm = 3;

// Bytes of a padded row, and of one tile of K or V.
template <typename T, int D>
constexpr int core_row() { return D * (int)sizeof(T) + 16; }
template <typename T, int D>
constexpr int core_tile() { return kCoreTile * core_row<T, D>(); }

// Rows [t, t + 32) below `end` of K, V and log(1/pi) to one buffer (zeros past
// them); the caller commits the group.
template <typename T, int D>
__device__ __forceinline__ void core_copy(unsigned char* ks, unsigned char* vs, float* lws,
                                          const T* K, const T* V, const float* lw, int t,
                                          int end) {
  constexpr int CPR = D * (int)sizeof(T) / 16;
#pragma unroll
  for (int i = 0; i < kCoreTile * CPR / kCoreThreads; ++i) {
    const int c = threadIdx.x + i * kCoreThreads;
    const int r = c / CPR, ch = c - r * CPR;
    const bool live = t + r < end;
    const size_t src = (size_t)(live ? t + r : 0) * D + ch * (16 / sizeof(T));
    cp_async16_zfill(ks + r * core_row<T, D>() + 16 * ch, K + src, live);
    cp_async16_zfill(vs + r * core_row<T, D>() + 16 * ch, V + src, live);
  }
  if (threadIdx.x < kCoreTile) cp_async4(lws + threadIdx.x, lw + min(t + (int)threadIdx.x, end - 1));
}

// 4 floats from 16 bytes of float32, 8 from 16 of bf16.
__device__ __forceinline__ void core_load(const unsigned char* p, float (&x)[4], float) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
}
__device__ __forceinline__ void core_load(const unsigned char* p, float (&x)[8], __nv_bfloat16) {
  const uint4 v = *reinterpret_cast<const uint4*>(p);
  const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    x[2 * i] = bf16_lo(u[i]);
    x[2 * i + 1] = bf16_hi(u[i]);
  }
}

// Sum of eight pairs, as a tree.
__device__ __forceinline__ float tree8(const float2 (&x)[8]) {
  const float2 a = __fadd2_rn(__fadd2_rn(x[0], x[1]), __fadd2_rn(x[2], x[3]));
  const float2 b = __fadd2_rn(__fadd2_rn(x[4], x[5]), __fadd2_rn(x[6], x[7]));
  const float2 s = __fadd2_rn(a, b);
  return s.x + s.y;
}

// GM: heads held (a power of two >= the slice's).
template <int D, int GM>
__global__ void __launch_bounds__(kCoreThreads) decode_f32_kernel(DecodeArgs a) {
  constexpr int REC = rec_floats(D), TILE = core_tile<float, D>(), ROW = core_row<float, D>();
  constexpr int HP = (GM + kCoreWarps - 1) / kCoreWarps;  // heads of a warp: w, w + 4
  constexpr int TP = kCoreThreads / D;                    // threads of a channel
  extern __shared__ __align__(16) unsigned char csm[];
  unsigned char* ks = csm;             // [2][TILE]
  unsigned char* vs = csm + 2 * TILE;  // [2][TILE]
  __shared__ __align__(16) float qs[GM][D], cs[D];
  __shared__ float lws[2][kCoreTile], xs[GM][kCoreTile], vcp[kCoreWarps][kCoreTile];
  __shared__ __align__(16) float2 wu[kCoreTile][GM];
  __shared__ float fac[GM];
  const int unit = blockIdx.y, split = blockIdx.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int G = a.group;
  grid_dependency_wait();
  grid_launch_dependents();
  const int n = min(max(a.n_kept[unit], 0), a.cap);
  const int T = (n + kCoreTile - 1) / kCoreTile;
  const int tb = (int)((long long)split * T / a.splits);
  const int te = (int)((long long)(split + 1) * T / a.splits);
  const float* K = (const float*)a.Kc + (size_t)unit * a.cap * D;
  const float* V = (const float*)a.Vc + (size_t)unit * a.cap * D;
  const float* lw = a.logw + (size_t)unit * a.cap;
  if (tb < te) core_copy<float, D>(ks, vs, lws[0], K, V, lw, tb * kCoreTile, n);
  cp_async_commit();
  const float scale = rsqrtf((float)D);
  const float* Q = (const float*)a.Q + (size_t)unit * a.gstride * D;
  for (int i = tid; i < GM * D; i += kCoreThreads) qs[i / D][i % D] = i / D < G ? Q[i] * scale : 0.f;
  const int cr = centre_row(n);
  for (int i = tid; i < D; i += kCoreThreads) cs[i] = cr < 0 ? 0.f : V[(size_t)cr * D + i];

  float M[HP], l[HP], U[HP], A2[HP], cmax[HP], umax[HP];
#pragma unroll
  for (int h = 0; h < HP; ++h) {
    M[h] = -INFINITY;
    l[h] = U[h] = A2[h] = cmax[h] = umax[h] = 0.f;
  }
  float2 acc[GM];  // o and A1 of this thread's channel (TP > 1: of its share of the tokens)
#pragma unroll
  for (int g = 0; g < GM; ++g) acc[g] = make_float2(0.f, 0.f);
  const int ch = tid % D, tpart = tid / D;

  for (int t = tb; t < te; ++t) {
    const int s = (t - tb) & 1;
    if (t + 1 < te)
      core_copy<float, D>(ks + (s ^ 1) * TILE, vs + (s ^ 1) * TILE, lws[s ^ 1], K, V, lw,
                          (t + 1) * kCoreTile, n);
    cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();
    {  // logits, and a quarter of ||v - c||^2
      const unsigned char* kr = ks + s * TILE + lane * ROW;
      // a logit in sums of four channels each (16 at a time), added as a tree
      float xt[HP];
#pragma unroll
      for (int h = 0; h < HP; ++h) xt[h] = 0.f;
      if (warp < G) {
#pragma unroll 1
        for (int c0 = 0; c0 < D; c0 += 64) {
          float2 x[HP][8];
#pragma unroll
          for (int h = 0; h < HP; ++h)
#pragma unroll
            for (int i = 0; i < 8; ++i) x[h][i] = make_float2(0.f, 0.f);
#pragma unroll 2
          for (int e0 = c0; e0 < c0 + 64; e0 += 16) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int e = e0 + 4 * j;
              const float4 kv = *reinterpret_cast<const float4*>(kr + 4 * e);
#pragma unroll
              for (int h = 0; h < HP; ++h) {
                const float4 qv = *reinterpret_cast<const float4*>(&qs[(warp + 4 * h) % GM][e]);
                x[h][2 * j] =
                    __ffma2_rn(make_float2(kv.x, kv.y), make_float2(qv.x, qv.y), x[h][2 * j]);
                x[h][2 * j + 1] =
                    __ffma2_rn(make_float2(kv.z, kv.w), make_float2(qv.z, qv.w), x[h][2 * j + 1]);
              }
            }
          }
#pragma unroll
          for (int h = 0; h < HP; ++h) xt[h] += tree8(x[h]);
        }
#pragma unroll
        for (int h = 0; h < HP; ++h)
          if (warp + 4 * h < G) xs[warp + 4 * h][lane] = xt[h];
      }
      const unsigned char* vr = vs + s * TILE + lane * ROW;
      float2 vc = make_float2(0.f, 0.f);
#pragma unroll
      for (int e = 0; e < D / 4; e += 4) {
        const float4 vv = *reinterpret_cast<const float4*>(vr + 4 * (warp * (D / 4) + e));
        const float4 cv = *reinterpret_cast<const float4*>(&cs[warp * (D / 4) + e]);
        const float2 d0 = make_float2(vv.x - cv.x, vv.y - cv.y);
        const float2 d1 = make_float2(vv.z - cv.z, vv.w - cv.w);
        vc = __ffma2_rn(d0, d0, __ffma2_rn(d1, d1, vc));
      }
      vcp[warp][lane] = vc.x + vc.y;
    }
    __syncthreads();
    {  // weights: lane = token
      const bool live = t * kCoreTile + lane < n;
      const float lwt = lws[s][lane];
      const float omp = live ? -expm1f(-lwt) : 0.f;  // 1 - pi
      const float sq = sqrtf(omp);
      const float vc2 = (vcp[0][lane] + vcp[1][lane]) + (vcp[2][lane] + vcp[3][lane]);
      const float vn = sqrtf(vc2);
#pragma unroll
      for (int h = 0; h < HP; ++h) {
        const int g = warp + 4 * h;
        if (g >= G) break;
        const float x = live ? xs[g][lane] + lwt : -INFINITY;
        const float mx = warp_max(x);
        float f = 1.f;
        if (mx > M[h]) {
          f = expf(M[h] - mx);
          const float f2 = f * f;
          l[h] *= f;
          U[h] *= f2;
          A2[h] *= f2;
          cmax[h] *= f;
          umax[h] *= f;
          M[h] = mx;
        }
        if (lane == 0) fac[g] = f;
        const float w = live ? expf((xs[g][lane] - M[h]) + lwt) : 0.f;
        const float u = omp * w * w, su = sq * w;
        l[h] += w;
        U[h] += u;
        A2[h] = fmaf(u, vc2, A2[h]);
        cmax[h] = fmaxf(cmax[h], su * vn);
        umax[h] = fmaxf(umax[h], su);
        wu[lane][g] = make_float2(w, u);
      }
    }
    __syncthreads();
#pragma unroll
    for (int g = 0; g < GM; ++g) {
      if (g >= G) break;
      const float f = fac[g];
      acc[g].x *= f;
      acc[g].y *= f * f;
    }
    const unsigned char* vcol = vs + s * TILE + 4 * ch;
#pragma unroll 8
    for (int r = tpart; r < kCoreTile; r += TP) {
      const float v = *reinterpret_cast<const float*>(vcol + r * ROW);
#pragma unroll
      for (int g = 0; g < GM; ++g) acc[g] = __ffma2_rn(wu[r][g], make_float2(v, v), acc[g]);
    }
    __syncthreads();  // this buffer is copied into next
  }
  cp_async_wait<0>();
  float* out = a.part + ((size_t)unit * a.splits + split) * (size_t)G * REC;
#pragma unroll
  for (int h = 0; h < HP; ++h) {
    const int g = warp + 4 * h;
    if (g >= G) break;
    const float ls = warp_sum(l[h]), Us = warp_sum(U[h]), As = warp_sum(A2[h]);
    const float cm = warp_max(cmax[h]), um = warp_max(umax[h]);
    if (lane == 0) {
      float* r = out + (size_t)g * REC;
      r[kRecM] = M[h];
      r[kRecL] = ls;
      r[kRecU] = Us;
      r[kRecA2] = As;
      r[kRecCmax] = cm;
      r[kRecUmax] = um;
    }
  }
  if constexpr (TP > 1) {  // the second half of the tokens, added by the first's threads
    float2* half = reinterpret_cast<float2*>(csm);  // [GM][D]
    __syncthreads();
    if (tpart == 1)
#pragma unroll
      for (int g = 0; g < GM; ++g) half[g * D + ch] = acc[g];
    __syncthreads();
    if (tpart == 0)
#pragma unroll
      for (int g = 0; g < GM; ++g) acc[g] = __fadd2_rn(acc[g], half[g * D + ch]);
  }
  if (tpart == 0) {
#pragma unroll
    for (int g = 0; g < GM; ++g) {
      if (g >= G) break;
      out[(size_t)g * REC + kRecHead + ch] = acc[g].x;
      out[(size_t)g * REC + kRecHead + D + ch] = acc[g].y;
    }
  }
}

struct SecondArgs {
  const void* Q;
  const void* Kc;
  const void* Vc;
  const float* logw;
  const int32_t* n_kept;
  const float* y;
  const float* lse;  // RANGE: l
  const float* m;    // RANGE: M (HeadNorm)
  float* out;  // contributions [units * gstride, cap], or b_t [units * gstride] (maximum)
  int cap;
  int group;
  int gstride;
  int splits;
};

// The second pass: RANGE false, contrib = (1 - pi) p^2 ||v - y_hat||^2 of every row
// (0 for certain rows and rows at or past n_kept); RANGE true, the maximum of
// its square root over the rows into out.
template <typename T, int D, int GM, bool RANGE>
__global__ void __launch_bounds__(kCoreThreads) second_pass_kernel(SecondArgs a) {
  constexpr int TILE = core_tile<T, D>(), ROW = core_row<T, D>(), VEC = 16 / (int)sizeof(T);
  constexpr int HP = (GM + kCoreWarps - 1) / kCoreWarps;
  extern __shared__ __align__(16) unsigned char csm[];
  unsigned char* ks = csm;
  unsigned char* vs = csm + 2 * TILE;
  __shared__ __align__(16) float qs[GM][D], ys[GM][D];
  __shared__ float lws[2][kCoreTile];
  const int unit = blockIdx.y, split = blockIdx.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int G = a.group;
  grid_dependency_wait();
  grid_launch_dependents();
  const int n = min(max(a.n_kept[unit], 0), a.cap);
  const int tiles = (n + kCoreTile - 1) / kCoreTile;
  const int tb = (int)((long long)split * tiles / a.splits);
  const int te = (int)((long long)(split + 1) * tiles / a.splits);
  const T* K = (const T*)a.Kc + (size_t)unit * a.cap * D;
  const T* V = (const T*)a.Vc + (size_t)unit * a.cap * D;
  const float* lw = a.logw + (size_t)unit * a.cap;
  const size_t hq0 = (size_t)unit * a.gstride;
  if (tb < te) core_copy<T, D>(ks, vs, lws[0], K, V, lw, tb * kCoreTile, n);
  cp_async_commit();
  const float scale = rsqrtf((float)D);
  const T* Q = (const T*)a.Q + hq0 * D;
  for (int i = tid; i < GM * D; i += kCoreThreads) {
    const bool in = i / D < G;
    qs[i / D][i % D] = in ? to_f32(Q[i]) * scale : 0.f;
    ys[i / D][i % D] = in ? a.y[hq0 * D + i] : 0.f;
  }
  float ls[HP], ln[HP], best[HP];  // log N_hat, or (RANGE) M and l
#pragma unroll
  for (int h = 0; h < HP; ++h) {
    const bool in = warp + 4 * h < G;
    ls[h] = in ? (RANGE ? a.m : a.lse)[hq0 + warp + 4 * h] : 0.f;
    ln[h] = RANGE && in ? a.lse[hq0 + warp + 4 * h] : 1.f;
    best[h] = 0.f;
  }
  if constexpr (!RANGE)  // rows at or past n_kept
    for (int g = 0; g < G; ++g)
      for (int i = n + split * kCoreThreads + tid; i < a.cap; i += a.splits * kCoreThreads)
        a.out[(hq0 + g) * a.cap + i] = 0.f;
  for (int t = tb; t < te; ++t) {
    const int s = (t - tb) & 1;
    if (t + 1 < te)
      core_copy<T, D>(ks + (s ^ 1) * TILE, vs + (s ^ 1) * TILE, lws[s ^ 1], K, V, lw,
                      (t + 1) * kCoreTile, n);
    cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();
    if (warp < G) {
      const unsigned char* kr = ks + s * TILE + lane * ROW;
      const unsigned char* vr = vs + s * TILE + lane * ROW;
      // in sums of four channels each, as in the decode
      float xt[HP], dt[HP];
#pragma unroll
      for (int h = 0; h < HP; ++h) xt[h] = dt[h] = 0.f;
#pragma unroll 1
      for (int c0 = 0; c0 < D; c0 += 64) {
        float2 x[HP][8], d2[HP][8];
#pragma unroll
        for (int h = 0; h < HP; ++h)
#pragma unroll
          for (int i = 0; i < 8; ++i) x[h][i] = d2[h][i] = make_float2(0.f, 0.f);
#pragma unroll 1
        for (int e0 = c0; e0 < c0 + 64; e0 += 16) {
#pragma unroll
          for (int e = e0; e < e0 + 16; e += VEC) {
            float kv[VEC], vv[VEC];
            core_load(kr + e * (int)sizeof(T), kv, T());
            core_load(vr + e * (int)sizeof(T), vv, T());
#pragma unroll
            for (int h = 0; h < HP; ++h)
#pragma unroll
              for (int i = 0; i < VEC; i += 4) {
                const int j = (e - e0 + i) / 2;
                const float4 qv = *reinterpret_cast<const float4*>(&qs[(warp + 4 * h) % GM][e + i]);
                const float4 yv = *reinterpret_cast<const float4*>(&ys[(warp + 4 * h) % GM][e + i]);
                x[h][j] = __ffma2_rn(make_float2(kv[i], kv[i + 1]), make_float2(qv.x, qv.y), x[h][j]);
                x[h][j + 1] =
                    __ffma2_rn(make_float2(kv[i + 2], kv[i + 3]), make_float2(qv.z, qv.w), x[h][j + 1]);
                const float2 a0 = make_float2(vv[i] - yv.x, vv[i + 1] - yv.y);
                const float2 a1 = make_float2(vv[i + 2] - yv.z, vv[i + 3] - yv.w);
                d2[h][j] = __ffma2_rn(a0, a0, d2[h][j]);
                d2[h][j + 1] = __ffma2_rn(a1, a1, d2[h][j + 1]);
              }
          }
        }
#pragma unroll
        for (int h = 0; h < HP; ++h) {
          xt[h] += tree8(x[h]);
          dt[h] += tree8(d2[h]);
        }
      }
      const int row = t * kCoreTile + lane;
      const float lwt = row < n ? lws[s][lane] : 0.f;
      const bool tail = lwt > 0.f;  // pi = 1: not in the tail sample
      const float omp = tail ? -expm1f(-lwt) : 0.f;
#pragma unroll
      for (int h = 0; h < HP; ++h) {
        const int g = warp + 4 * h;
        if (g >= G) break;
        const float p = expf((xt[h] - ls[h]) + lwt);  // w / N_hat (RANGE: w)
        const float dist = dt[h];
        if constexpr (RANGE) {
          if (tail) best[h] = fmaxf(best[h], sqrtf(omp) * (p / ln[h]) * sqrtf(dist));
        } else {
          if (row < n) a.out[(hq0 + g) * a.cap + row] = tail ? omp * p * p * dist : 0.f;
        }
      }
    }
    __syncthreads();  // this buffer is copied into next
  }
  cp_async_wait<0>();
  if constexpr (RANGE) {
#pragma unroll
    for (int h = 0; h < HP; ++h) {
      const int g = warp + 4 * h;
      if (g >= G) break;
      const float m = warp_max(best[h]);
      // non-negative floats order like their bit patterns
      if (lane == 0 && m > 0.f) atomicMax((unsigned int*)&a.out[hq0 + g], __float_as_uint(m));
    }
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
// CTAs per unit: one wave of kCoreCtasPerSm CTAs per SM, each at least a tile.
static int core_splits(int units, int cap, int most) {
  const int tiles = (cap + kCoreTile - 1) / kCoreTile;
  int s = kCoreCtasPerSm * sm_count() / units;
  if (s > tiles) s = tiles;
  if (s > most) s = most;
  return s < 1 ? 1 : s;
}

template <typename Kernel, typename A>
static ebd_status launch_core(Kernel kernel, int units, int tile_bytes, const A& a, cudaStream_t s) {
  const int smem = 4 * tile_bytes;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
      cudaSuccess)
    return EBD_ERR_CUDA;
  return launch_dependent(kernel, dim3((unsigned)a.splits, (unsigned)units), kCoreThreads, smem, s,
                          a);
}

// f(integral_constant GM) for the smallest of 1, 2, 4, 8 that holds `group` heads.
template <typename F>
static ebd_status with_heads(int group, F f) {
  if (group <= 1) return f(std::integral_constant<int, 1>{});
  if (group <= 2) return f(std::integral_constant<int, 2>{});
  if (group <= 4) return f(std::integral_constant<int, 4>{});
  return f(std::integral_constant<int, 8>{});
}

bool decode_f32_usable(const DecodeArgs& a) {
  return aligned16(a.Kc) && aligned16(a.Vc) && a.group <= kCoreHeads;
}

ebd_status launch_decode_f32(int head_dim, DecodeArgs& a, int units, cudaStream_t s) {
  a.splits = core_splits(units, a.cap, a.splits);
  return with_heads(a.group, [&](auto gm) {
    constexpr int GM = decltype(gm)::value;
    return head_dim == 128
               ? launch_core(decode_f32_kernel<128, GM>, units, core_tile<float, 128>(), a, s)
               : launch_core(decode_f32_kernel<64, GM>, units, core_tile<float, 64>(), a, s);
  });
}

template <typename T, bool RANGE>
static ebd_status launch_second(int head_dim, SecondArgs& a, int units, cudaStream_t s) {
  a.splits = core_splits(units, a.cap, 65535);
  return with_heads(a.group, [&](auto gm) {
    constexpr int GM = decltype(gm)::value;
    return head_dim == 128 ? launch_core(second_pass_kernel<T, 128, GM, RANGE>, units,
                                         core_tile<T, 128>(), a, s)
                           : launch_core(second_pass_kernel<T, 64, GM, RANGE>, units,
                                         core_tile<T, 64>(), a, s);
  });
}

ebd_status launch_range_f32(int head_dim, const DecodeArgs& d, int units, cudaStream_t s) {
  SecondArgs a = {d.Q, d.Kc, d.Vc, d.logw, d.n_kept, d.y, d.lse, d.radius, d.b_t, d.cap,
                  d.group, d.gstride, 1};
  return launch_second<float, true>(head_dim, a, units, s);
}

bool contributions_core_usable(const void* K_c, const void* V_c, int group) {
  return aligned16(K_c) && aligned16(V_c) && group <= kCoreHeads;
}

ebd_status launch_contributions_core(ebd_dtype dtype, int head_dim, int units, int group, int cap,
                                     const void* Q, const void* K_c, const void* V_c,
                                     const float* logw_c, const int32_t* n_kept, const float* y,
                                     const float* lse, float* contrib, cudaStream_t s) {
  SecondArgs a = {Q, K_c, V_c, logw_c, n_kept, y, lse, nullptr, contrib, cap, group, group, 1};
  return dtype == EBD_F32 ? launch_second<float, false>(head_dim, a, units, s)
                          : launch_second<__nv_bfloat16, false>(head_dim, a, units, s);
}

}  // namespace ebd
