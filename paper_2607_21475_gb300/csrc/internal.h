// Host-side declarations shared by the translation units of libebd.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <atomic>

#include "../../include/ebd.h"

namespace ebd {

// Number of SMs of the current device (cached per device).
int sm_count();

inline ebd_status cuda_status(cudaError_t e) { return e == cudaSuccess ? EBD_OK : EBD_ERR_CUDA; }

// Last launch error of this thread, mapped to a status (clears the error).
inline ebd_status launch_status() { return cuda_status(cudaGetLastError()); }

// Dynamic shared memory that launches of `kernel` may ask for.  The limit is the
// process's, not the launch's: every call for a kernel passes the same number, its
// largest layout, so that no thread lowers it between another's call and launch.
template <typename Kernel>
ebd_status allow_smem(Kernel kernel, int most) {
  return cuda_status(
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
}

// Clusters of 2^lg CTAs (lg < 4) of Kernel that the current device holds at a time.  A
// cluster lies within one GPC, so for the larger ones that is fewer than SMs / 2^lg
// (152 SMs hold 15 clusters of 8 whose CTAs take an SM each).  Asked once per
// device and kernel; `smem`: dynamic shared memory of a CTA, `most`: allow_smem's.
template <auto Kernel>
int resident_clusters(int lg, int threads, int smem, int most) {
  static std::atomic<int> cached[64][4];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return sm_count() >> lg;
  int n = cached[dev][lg].load(std::memory_order_relaxed);
  if (n > 0) return n;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1u << lg);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1u << lg;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (allow_smem(Kernel, most) != EBD_OK ||
      cudaOccupancyMaxActiveClusters(&n, Kernel, &cfg) != cudaSuccess || n < 1) {
    (void)cudaGetLastError();
    n = sm_count() >> lg;
  }
  cached[dev][lg].store(n, std::memory_order_relaxed);
  return n;
}

// Launch as a programmatic dependent of what precedes it in the stream (the
// kernel waits for that before it reads or writes memory).
template <typename... Params, typename... Args>
ebd_status launch_dependent(void (*kernel)(Params...), dim3 grid, int threads, size_t smem,
                            cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cuda_status(cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...));
}

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Design validation shared by the eviction entry points (evict.cu).
ebd_status check_design(const ebd_design* d);

// E1-E4a for every unit (evict.cu): certainty set, pi, draws, index
// compaction.  n_len (nullable, device [units]) gives each unit's context
// length when it is below the row stride d->n_ctx of `scores`.
ebd_status launch_select(const ebd_design* d, const float* scores, const int32_t* n_len,
                         float* pi, uint8_t* mask, int32_t* idx_c, float* logw_c, int32_t* n_kept,
                         int cap, int32_t* dev_status, cudaStream_t stream);

// E4b for every unit (evict.cu): rows K[idx_c[p]], V[idx_c[p]] (row stride
// d->n_ctx) to K_c[p], V_c[p] for p < min(n_kept, cap); rows whose index lies
// outside [0, n_ctx) are skipped.
ebd_status launch_gather(const ebd_design* d, ebd_dtype dtype, const void* K, const void* V,
                         const int32_t* idx_c, const int32_t* n_kept, int cap, void* K_c,
                         void* V_c, cudaStream_t s);

// The same for the units [unit0, unit0 + n_units) only.  `ctas_per_unit`:
// the cluster size of the shared-memory select (0: chosen for this launch's
// units; a caller that splits one request into several launches passes the
// size chosen for the whole request, so each unit is split the same way).
// `dependent`: launched as a programmatic dependent of the work before it.
ebd_status launch_select_range(const ebd_design* d, const float* scores, const int32_t* n_len,
                               float* pi, uint8_t* mask, int32_t* idx_c, float* logw_c,
                               int32_t* n_kept, int cap, int32_t* dev_status, int unit0,
                               int n_units, cudaStream_t stream, int ctas_per_unit,
                               bool dependent);

// CTAs per unit of the shared-memory select for `units` units of n_ctx
// tokens (0 when the context is too long for a cluster).
int select_cluster_size(int n_ctx, int units);
ebd_status launch_gather_range(const ebd_design* d, ebd_dtype dtype, const void* K,
                               const void* V, const int32_t* idx_c, const int32_t* n_kept,
                               int cap, void* K_c, void* V_c, int unit0, int n_units,
                               cudaStream_t s);

bool aligned16(const void* p);

// Address under which kernels read a caller's buffer: device or managed memory
// as is, page-locked host memory through its device mapping (read over the
// host link); nullptr for memory the device cannot address (evict.cu).
const void* device_address(const void* p);
bool is_device_memory(const void* p);

// E0: accumulated attention scores into `scores` using `workspace` for the
// per-row log-sum-exp.  Arguments validated by the caller; dev_status nullable.
ebd_status launch_score(ebd_dtype dtype, int batch, int n_kv_heads, int head_dim, int n_ctx,
                        int n_obs, const void* q_obs, const void* K, float* scores,
                        float* lse_ws, int32_t* dev_status, cudaStream_t stream);

// E0 on tcgen05 with tensor-memory accumulators (score_tc.cu): bf16,
// head_dim 64/128, 16-byte aligned inputs.
bool score_tc_supported(ebd_dtype dtype, int head_dim, int n_obs, const void* q_obs,
                        const void* K);
ebd_status launch_score_tc(int units, int head_dim, int n_ctx, int n_obs, const void* q_obs,
                           const void* K, float* scores, float* lse, int32_t* dev_status,
                           cudaStream_t s);

}  // namespace ebd
