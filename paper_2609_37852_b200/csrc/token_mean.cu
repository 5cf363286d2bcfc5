// The token mean that key centering subtracts.  The quantiser, with and without the producer steps in
// front, lives in quantize_batch.cu.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include "common.cuh"
#include "mxfp8_device.cuh"
#include "sm100_ptx.cuh"

namespace attnfp8 {
namespace {

namespace cg = cooperative_groups;

// Four consecutive values as FP32.
__device__ __forceinline__ void load4(const __nv_bfloat16* p, float* x) {
  const uint2 raw = *reinterpret_cast<const uint2*>(p);
  x[0] = __uint_as_float(raw.x << 16); x[1] = __uint_as_float(raw.x & 0xFFFF0000u);
  x[2] = __uint_as_float(raw.y << 16); x[3] = __uint_as_float(raw.y & 0xFFFF0000u);
}
__device__ __forceinline__ void load4(const float* p, float* x) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
}

// FP32 mean over tokens of the (rotated, BF16-rounded) tensor, per (batch, head, channel).  The
// terms are BF16 values, so a double-precision sum is exact whatever its order while the largest
// magnitude is at most 2^45 / N times the smallest, and the result is then the correctly rounded quotient; beyond that the order of the sum, which follows from the shape and the number of SMs, keeps it reproducible.
//
// Memory-bound work (the key tensor once, the tables from L2) on few slabs: a grouped-query layer has 4 to
// 8, so a slab is shared by a cluster of up to eight CTAs, each summing a range of the tokens with vector
// loads; the first CTA adds the others' sums from their shared memory.  With rotary embedding, BF16:
// 4 x 4096 x 128 values 135 -> 13 us, 48 x 2816 x 128 97 -> 24 us against one CTA per slab with scalar loads
// (four pairs per thread and 64 registers: with eight pairs and 88 registers the second took 40 us).
constexpr int kMaxCluster = 8;
constexpr int kMeanThreads = 512;

template <typename T>
__global__ void __launch_bounds__(kMeanThreads, 2) token_mean_kernel(const T* src, int N, int d, const float* cos,
                                                                     const float* sin, float* mean) {
  extern __shared__ __align__(16) uint8_t smem[];
  double* part = reinterpret_cast<double*>(smem);                   // [phases][d], then the CTA's sums in row 0
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = static_cast<int>(cluster.block_rank()), ranks = static_cast<int>(cluster.num_blocks());
  const int half = d >> 1, chunks = half >> 2, phases = kMeanThreads / chunks;   // a thread sums four pairs (c, c + d / 2)
  const int ph = threadIdx.x / chunks, pc = (threadIdx.x - ph * chunks) * 4;
  const size_t slab = blockIdx.x / ranks;
  const T* g = src + slab * N * d + pc;
  const int per = N / ranks;                                         // N is a multiple of 128
  const int n0 = rank * per, n1 = rank == ranks - 1 ? N : n0 + per;
  sm100::griddep_begin();
  if (ph < phases) {
    double lo[4], hi[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) lo[k] = hi[k] = 0.0;
#pragma unroll 4
    for (int n = n0 + ph; n < n1; n += phases) {
      float x1[4], x2[4];
      load4(g + static_cast<size_t>(n) * d, x1);
      load4(g + static_cast<size_t>(n) * d + half, x2);
      if (cos != nullptr) {
        float c[4], s[4];
        load4(cos + static_cast<size_t>(n) * half + pc, c);
        load4(sin + static_cast<size_t>(n) * half + pc, s);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float r = rotate_bf16(x1[k], x2[k], c[k], s[k], false);
          x2[k] = rotate_bf16(x2[k], x1[k], c[k], s[k], true);
          x1[k] = r;
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        lo[k] += static_cast<double>(x1[k]);
        hi[k] += static_cast<double>(x2[k]);
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      part[ph * d + pc + k] = lo[k];
      part[ph * d + half + pc + k] = hi[k];
    }
  }
  __syncthreads();
  const int c = threadIdx.x;                                         // d <= 256: one channel per thread
  if (c < d) {
    double sum = 0.0;
    for (int i = 0; i < phases; ++i) sum += part[i * d + c];
    part[c] = sum;                                                   // only this thread reads column c
  }
  cluster.sync();
  if (rank == 0 && c < d) {
    double sum = part[c];
    for (int r = 1; r < ranks; ++r) sum += *cluster.map_shared_rank(part + c, r);
    mean[slab * d + c] = static_cast<float>(sum / static_cast<double>(N));
  }
  cluster.sync();                                                    // the sums stay until they have been read
}

template <typename T>
attn_status_t launch_mean_t(const void* src, int slabs, int N, int d, const float* cos, const float* sin, float* mean,
                            cudaStream_t stream) {
  // enough CTAs for two on every SM, no fewer than 128 tokens each
  int dev = 0, sms = 0, ranks = 1;
  const attn_status_t st = current_device(&dev, &sms);
  if (st != ATTN_OK) return st;
  while (ranks < kMaxCluster && slabs * ranks < 2 * sms && 2 * ranks <= N / 128) ranks *= 2;
  const int chunks = d / 8;
  const size_t smem = static_cast<size_t>(kMeanThreads / chunks) * d * sizeof(double);   // 32 KB
  const cudaError_t e = launch_overlapped(token_mean_kernel<T>, dim3(static_cast<unsigned>(slabs) * ranks), kMeanThreads, smem, stream,
                                          ranks, static_cast<const T*>(src), N, d, cos, sin, mean);
  if (e != cudaSuccess) return fail(ATTN_ERR_CUDA, "token mean: launch: %s", cudaGetErrorString(e));
  return ATTN_OK;
}

}  // namespace

attn_status_t launch_token_mean(const void* src, int src_dtype, int slabs, int N, int d, const float* cos, const float* sin,
                                float* mean, cudaStream_t stream) {
  if (src_dtype == ATTN_SRC_BF16) return launch_mean_t<__nv_bfloat16>(src, slabs, N, d, cos, sin, mean, stream);
  return launch_mean_t<float>(src, slabs, N, d, cos, sin, mean, stream);
}

}  // namespace attnfp8
