// Several pitched copies in one launch: the byte tensors of the chunks of a sequence, put together.
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace attnfp8 {
namespace {

constexpr int kThreads = 256;
constexpr int kPerThread = 4;                         // 16-byte pieces in flight per thread

struct CopyBatch {
  attn_copy_job_t job[ATTN_COPY_MAX_JOBS];
  int first_block[ATTN_COPY_MAX_JOBS + 1];
  int n;
};

// Memory-bound and, at the sizes of a sequence shard, launch-bound: 16 to 32 segments of 16 KB to 4 MB, which as one
// torch.cat per byte tensor took 14 launches and 150 us of host time in a step of 512 to 1024 queries.
__global__ void __launch_bounds__(kThreads) copy_kernel(const __grid_constant__ CopyBatch p) {
  int j = 0;
  while (j + 1 < p.n && static_cast<int>(blockIdx.x) >= p.first_block[j + 1]) ++j;
  const attn_copy_job_t& c = p.job[j];
  const uint32_t per_row = static_cast<uint32_t>(c.row_bytes / 16);
  const size_t pieces = static_cast<size_t>(c.rows) * per_row;
  const size_t i0 = static_cast<size_t>(static_cast<int>(blockIdx.x) - p.first_block[j]) * (kThreads * kPerThread) + threadIdx.x;
  sm100::griddep_begin();
  uint4 v[kPerThread];
#pragma unroll
  for (int k = 0; k < kPerThread; ++k) {
    const size_t i = i0 + k * kThreads;
    if (i < pieces) v[k] = reinterpret_cast<const uint4*>(c.src)[i];
  }
#pragma unroll
  for (int k = 0; k < kPerThread; ++k) {
    const size_t i = i0 + k * kThreads;
    if (i < pieces) *reinterpret_cast<uint4*>(static_cast<uint8_t*>(c.dst) + i / per_row * c.dst_pitch + i % per_row * 16) = v[k];
  }
}

}  // namespace

attn_status_t launch_copy_batch(const attn_copy_job_t* jobs, int n, cudaStream_t stream) {
  CopyBatch p;
  p.n = n;
  long long blocks = 0;
  for (int j = 0; j < n; ++j) {
    p.job[j] = jobs[j];
    p.first_block[j] = static_cast<int>(blocks);
    blocks += (jobs[j].rows * (jobs[j].row_bytes / 16) + kThreads * kPerThread - 1) / (kThreads * kPerThread);
    if (blocks > 0x7fffffffLL) return fail(ATTN_ERR_UNSUPPORTED, "copy batch: %lld blocks exceed 2^31 - 1", blocks);
  }
  p.first_block[n] = static_cast<int>(blocks);
  const cudaError_t e = launch_overlapped(copy_kernel, dim3(static_cast<unsigned>(blocks)), kThreads, 0, stream, 1, p);
  if (e != cudaSuccess) return fail(ATTN_ERR_CUDA, "copy batch: launch: %s", cudaGetErrorString(e));
  return ATTN_OK;
}

}  // namespace attnfp8
