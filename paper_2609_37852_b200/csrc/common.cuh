// Declarations shared by the kernels' translation units and the C-ABI layer.
#pragma once
#include <atomic>
#include <cstddef>
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

#include "../../include/attn_fp8.h"

namespace attnfp8 {

// Records a message for attn_fp8_last_error() and returns `code`.
attn_status_t fail(attn_status_t code, const char* fmt, ...);

// The current device's ordinal and SM count; fails when it is not compute capability 10.x.  What the runtime
// says of a device is kept per ordinal: asked for on every call it was a quarter of a small call's host time.
attn_status_t current_device(int* dev, int* sms);

// The id of the calling thread's context, never used again in the life of the process (a context that follows a reset has
// another); 0 where the thread has none yet.
uint64_t context_id();
constexpr int kMaxDevices = 64;

// Lets `kernel` ask for up to `bytes` of dynamic shared memory.  The limit belongs to a context: it is raised again where a
// device's context is not the one of the call before, and one runtime call per launch is saved otherwise.  Gives the
// device's SM count as well.
template <auto kernel>
attn_status_t allow_smem(size_t bytes, const char* who, int* sms) {
  static std::atomic<uint64_t> raised[kMaxDevices];   // per device ordinal: the context in which the limit is raised
  int dev = 0;
  const attn_status_t st = current_device(&dev, sms);
  if (st != ATTN_OK) return st;
  const uint64_t id = context_id();
  if (id && dev < kMaxDevices && raised[dev].load(std::memory_order_acquire) == id) return ATTN_OK;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
  if (e != cudaSuccess) {
    cudaGetLastError();
    return fail(ATTN_ERR_CUDA, "%s: cudaFuncSetAttribute: %s", who, cudaGetErrorString(e));
  }
  if (id && dev < kMaxDevices) raised[dev].store(id, std::memory_order_release);
  return ATTN_OK;
}

// Launches `kernel` so that it may start while the kernel ahead of it in the stream is finishing (programmatic
// stream serialisation): a kernel of the library sets itself up, executes griddepcontrol.wait before its first
// access to global memory, and lets the next one start as soon as that has returned.  What overlaps is the
// launch, barrier initialisation, tensor-memory allocation and descriptor fetch of one kernel and the tail of the
// one ahead: a step of one head of 256 tokens went from 32.5 to 28 us, a padded forward of 24 heads of 1111 tokens
// (five launches) from 69 to 62 us, an encoder step from 133 to 122 us.  `cluster`: CTAs per cluster along x.
template <class... Params, class... Args>
cudaError_t launch_kernel(void (*kernel)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t stream, int cluster, bool overlapped,
                          Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  if (overlapped) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs].val.clusterDim.x = cluster; attr[cfg.numAttrs].val.clusterDim.y = 1; attr[cfg.numAttrs++].val.clusterDim.z = 1;
  }
  cfg.attrs = attr;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
  if (e != cudaSuccess) cudaGetLastError();            // reported here, and not again by the next call that asks
  return e;
}
template <class... Params, class... Args>
cudaError_t launch_overlapped(void (*kernel)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t stream, int cluster,
                              Args&&... args) {
  return launch_kernel(kernel, grid, threads, smem, stream, cluster, true, static_cast<Args&&>(args)...);
}

// Bytes at the head of every workspace reserved for the device status word.
constexpr size_t kWorkspaceHeaderBytes = ATTN_STATUS_WORKSPACE_BYTES;

// The ticket counter of the persistent dQ kernel: bytes 16..19 of the workspace header, whose first word is `status`.
inline int* ticket_counter(int* status) { return status + 4; }

// Whether rows of a multiple of 32 bytes from `p` on can be stored a sector at a time (pointers are 16-byte aligned).
inline bool starts_sector(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 31) == 0; }

// cuTensorMapEncodeTiled fetched through the runtime (no link-time dependency on libcuda).
// Encodes a 2-D uint8 tensor [rows, row_bytes] (row pitch == row_bytes) with a
// (box_rows x 128-byte) box and the 128-byte swizzle.
attn_status_t encode_tmap_u8_sw128(CUtensorMap* out, const void* base, uint64_t row_bytes, uint64_t rows,
                                   uint32_t box_rows);

struct AttnShape {
  int B, N, Hq, Hkv, dqk, dv, causal;   // N: query rows (the length of Q, dO, O, dQ, LSE, delta)
  float scale;
  int eb;   // bytes per operand element: 1 = E4M3 codes with E8M0 block scales, 2 = BF16 without scales
  int ebv;  // the same for the row copies of dO and V, the operands of dP alone (2 with eb == 1: protected dP)
  int Nk;   // keys (the length of K, V, dK, dV); == N unless the caller holds a shard of the queries
  int q0t;  // 128-row tile index of query row 0 in the key sequence: key j is visible to query i iff j <= 128 * q0t + i
  int kv_lim;  // last real key inside the last key tile (127: the tile is full); read without the causal mask only
};

// Kernel launchers (each validates nothing: the C-ABI layer has done so).
attn_status_t launch_quantize_fused(const attn_quantize_job_t& job, const float* cos, const float* sin, float scale,
                                    float* mean, int* status, cudaStream_t stream);
attn_status_t launch_token_mean(const void* src, int slabs, int N, int d, const float* cos, const float* sin,
                                float* mean, cudaStream_t stream);
attn_status_t launch_quantize_batch(const attn_quantize_job_t* jobs, int n_jobs, int* status, cudaStream_t stream);
attn_status_t launch_bf16_copies(const void* src, int src_dtype, int B, int H, int N, int d, void* row_out, void* col_out,
                                 cudaStream_t stream);
attn_status_t launch_copy_batch(const attn_copy_job_t* jobs, int n, cudaStream_t stream);
attn_status_t launch_pad_tokens(const void* src, long long slabs, long long row_bytes, int n, int n_out, void* dst, cudaStream_t stream);
attn_status_t launch_fwd(const AttnShape& s, attn_qtensor_t q, attn_qtensor_t k, attn_qtensor_t v, void* o,
                         float* lse, int* status, cudaStream_t stream);
attn_status_t launch_fwd_interleaved(const AttnShape& s, attn_qtensor_t q, attn_qtensor_t k, attn_qtensor_t v, void* o,
                                     float* lse, int* status, cudaStream_t stream);
attn_status_t launch_bwd_delta(const AttnShape& s, attn_qtensor_t q, attn_qtensor_t k, attn_qtensor_t v,
                               attn_qtensor_t dO, const float* lse, float* delta, int* status, cudaStream_t stream);
attn_status_t launch_stale_delta(const AttnShape& s, const void* dO_bf16, const void* o_bf16, float* delta,
                                 cudaStream_t stream);
attn_status_t launch_consistent_delta(const AttnShape& s, attn_qtensor_t dO, const void* o_bf16, float* delta,
                                      cudaStream_t stream);
attn_status_t launch_bwd_dq(const AttnShape& s, attn_qtensor_t q, attn_qtensor_t k, attn_qtensor_t v,
                            attn_qtensor_t dO, const float* lse, const float* delta, void* dq, float* rowsum,
                            float* rowabs, float* post_rowsum, float* post_rowabs, int* status, cudaStream_t stream,
                            bool behind_dkdv = false, float* p_abs_dp = nullptr);
attn_status_t launch_bwd_dkdv(const AttnShape& s, attn_qtensor_t q, attn_qtensor_t k, attn_qtensor_t v,
                              attn_qtensor_t dO, const float* lse, const float* delta, void* dk, void* dv,
                              int* status, cudaStream_t stream, bool clear_tickets);

attn_status_t measure_mma_peak(double* tflops_out, int* status, cudaStream_t stream);
attn_status_t measure_dq_reduction(const AttnShape& s, float* dq_f32, double* ms_out, double* bytes_out, cudaStream_t stream);

inline size_t scale_tiles_per_slab(int64_t rows, int64_t cols) {
  return static_cast<size_t>((rows + 127) / 128) * static_cast<size_t>((cols / 32 + 3) / 4);
}

}  // namespace attnfp8
