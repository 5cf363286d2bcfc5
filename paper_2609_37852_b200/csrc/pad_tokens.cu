// Zero rows appended to the token dimension, for sequences whose length is no multiple of the 128-token tile.
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace attnfp8 {
namespace {

constexpr int kThreads = 256;
constexpr int kPerThread = 4;                         // 16-byte pieces in flight per thread

// A contiguous slab [n rows] becomes a slab [n_out rows]: the first `have` 16-byte pieces are copied, the rest of
// `want` is zero.  Memory-bound; torch's fill followed by a strided copy wrote the real rows twice and moved BF16
// values two bytes at a time: three tensors of 64, 16 and 16 slabs of 1111 x 128 BF16 values took 44.7 us, 10.9 us
// here (56 MB: 5.1 TB/s).
__global__ void __launch_bounds__(kThreads) pad_kernel(const uint4* src, uint4* dst, uint32_t have,
                                                       uint32_t want, uint32_t blocks_per_slab) {
  const size_t slab = blockIdx.x / blocks_per_slab;
  const uint32_t i0 = (blockIdx.x % blocks_per_slab) * (kThreads * kPerThread) + threadIdx.x;
  sm100::griddep_begin();
  uint4 v[kPerThread];
#pragma unroll
  for (int k = 0; k < kPerThread; ++k) {
    const uint32_t i = i0 + k * kThreads;
    v[k] = i < have ? src[slab * have + i] : make_uint4(0u, 0u, 0u, 0u);
  }
#pragma unroll
  for (int k = 0; k < kPerThread; ++k) {
    const uint32_t i = i0 + k * kThreads;
    if (i < want) dst[slab * want + i] = v[k];
  }
}

}  // namespace

attn_status_t launch_pad_tokens(const void* src, long long slabs, long long row_bytes, int n, int n_out, void* dst, cudaStream_t stream) {
  const long long have = row_bytes / 16 * n, want = row_bytes / 16 * n_out;
  const long long per_slab = (want + kThreads * kPerThread - 1) / (kThreads * kPerThread), blocks = per_slab * slabs;
  if (want > 0x7fffffffLL || blocks > 0x7fffffffLL) return fail(ATTN_ERR_UNSUPPORTED, "pad_tokens: %lld blocks exceed 2^31 - 1", blocks);
  const cudaError_t e = launch_overlapped(pad_kernel, dim3(static_cast<unsigned>(blocks)), kThreads, 0, stream, 1,
                                          static_cast<const uint4*>(src), static_cast<uint4*>(dst), static_cast<uint32_t>(have),
                                          static_cast<uint32_t>(want), static_cast<uint32_t>(per_slab));
  if (e != cudaSuccess) return fail(ATTN_ERR_CUDA, "pad_tokens: launch: %s", cudaGetErrorString(e));
  return ATTN_OK;
}

}  // namespace attnfp8
