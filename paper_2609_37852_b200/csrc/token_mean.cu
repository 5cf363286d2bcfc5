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

// FP32 mean over tokens of the (rotated, BF16-rounded) tensor, per (batch, head, channel).  The source is BF16 (centering of
// FP32 sources is refused), so the terms are BF16 values, and a double-precision sum is exact whatever its order while the
// largest magnitude is at most 2^45 / N times the smallest: the result is then the correctly rounded quotient.  Beyond that
// the order of the sum, which follows from the shape and the number of SMs, keeps it reproducible.
//
// Memory-bound work (the key tensor once, the tables from L2) on few slabs: a grouped-query layer has 4 to
// 8, so a slab is shared by a cluster of up to eight CTAs, each summing a range of the tokens with vector
// loads; the first CTA adds the others' sums from their shared memory.  With rotary embedding, BF16:
// 4 x 4096 x 128 values 135 -> 13 us, 48 x 2816 x 128 97 -> 24 us against one CTA per slab with scalar loads
// (four pairs per thread and 64 registers: with eight pairs and 88 registers the second took 40 us).
// Where the CTAs fill no more than half of the SMs (kFew), the latency of a thread's loads is all that counts: it then takes
// 128 registers and loads four tokens ahead of the arithmetic.  Mean and quantiser, before and so: 4 x 4096 x 128 18.4, 16.1
// us; 8 x 8192 x 128 41.1, 27.6; 4 x 8192 x 192 47.7, 30.9; 4 x 16384 x 128 without rotation 35.1, 22.2.  With more CTAs, one
// on an SM is too few and clusters of eight wait for one another: 16 x 8192 x 192 86.0, 88.3; 18 x 2048 x 128 19.2, 19.5.
constexpr int kMaxCluster = 8;
constexpr int kMeanThreads = 512;
constexpr int kAhead = 4;                                            // tokens of a thread loaded ahead of the arithmetic

// Four consecutive values as FP32: of the source, and of the rotary tables.
__device__ __forceinline__ void widen4(const uint2& raw, float* x) {
  x[0] = __uint_as_float(raw.x << 16); x[1] = __uint_as_float(raw.x & 0xFFFF0000u);
  x[2] = __uint_as_float(raw.y << 16); x[3] = __uint_as_float(raw.y & 0xFFFF0000u);
}
__device__ __forceinline__ void widen4(const float4& raw, float* x) {
  x[0] = raw.x; x[1] = raw.y; x[2] = raw.z; x[3] = raw.w;
}

__device__ __forceinline__ void load4(const __nv_bfloat16* p, float* x) { widen4(*reinterpret_cast<const uint2*>(p), x); }
__device__ __forceinline__ void load4(const float* p, float* x) { widen4(*reinterpret_cast<const float4*>(p), x); }

template <bool kFew>
__global__ void __launch_bounds__(kMeanThreads, kFew ? 1 : 2) token_mean_kernel(const __nv_bfloat16* src, int N, int d, const float* cos,
                                                                     const float* sin, float* mean) {
  extern __shared__ __align__(16) uint8_t smem[];
  double* part = reinterpret_cast<double*>(smem);                   // [phases][d], then the CTA's sums in row 0
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = static_cast<int>(cluster.block_rank()), ranks = static_cast<int>(cluster.num_blocks());
  const int half = d >> 1, chunks = half >> 2, phases = kMeanThreads / chunks;   // a thread sums four pairs (c, c + d / 2)
  const int ph = threadIdx.x / chunks, pc = (threadIdx.x - ph * chunks) * 4;
  const size_t slab = blockIdx.x / ranks;
  const __nv_bfloat16* g = src + slab * N * d + pc;
  const int per = N / ranks;                                         // N is a multiple of 128
  const int n0 = rank * per, n1 = rank == ranks - 1 ? N : n0 + per;
  sm100::griddep_begin();
  if (ph < phases) {
    double lo[4], hi[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) lo[k] = hi[k] = 0.0;
    int n = n0 + ph;
    if constexpr (kFew) {
      // (the other loop has its own copy: one for both took mean and quantiser of 16 x 8192 x 192 from 86.1 to 89.4 us)
      auto add = [&](float* x1, float* x2, const float* c, const float* s) {
        if (cos != nullptr) {
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
      };
      for (; n + (kAhead - 1) * phases < n1; n += kAhead * phases) {
        uint2 r1[kAhead], r2[kAhead];
        float4 c4[kAhead], s4[kAhead];
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
          const size_t m = n + i * phases;
          r1[i] = *reinterpret_cast<const uint2*>(g + m * d);
          r2[i] = *reinterpret_cast<const uint2*>(g + m * d + half);
          if (cos != nullptr) {
            c4[i] = *reinterpret_cast<const float4*>(cos + m * half + pc);
            s4[i] = *reinterpret_cast<const float4*>(sin + m * half + pc);
          }
        }
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
          float x1[4], x2[4], c[4], s[4];
          widen4(r1[i], x1); widen4(r2[i], x2);
          if (cos != nullptr) { widen4(c4[i], c); widen4(s4[i], s); }
          add(x1, x2, c, s);
        }
      }
    }
#pragma unroll 4
    for (; n < n1; n += phases) {
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
#pragma unroll (kFew ? 8 : 4)
    for (int i = 0; i < phases; ++i) sum += part[i * d + c];
    part[c] = sum;                                                   // only this thread reads column c
  }
  cluster.sync();
  if (rank == 0 && c < d) {
    double sum = part[c];
#pragma unroll
    for (int r = 1; r < kMaxCluster; ++r)
      if (r < ranks) sum += *cluster.map_shared_rank(part + c, r);
    mean[slab * d + c] = static_cast<float>(sum / static_cast<double>(N));
  }
  cluster.sync();                                                    // the sums stay until they have been read
}

}  // namespace

attn_status_t launch_token_mean(const void* src, int slabs, int N, int d, const float* cos, const float* sin, float* mean,
                                cudaStream_t stream) {
  // enough CTAs for two on every SM, no fewer than 128 tokens each
  int dev = 0, sms = 0, ranks = 1;
  const attn_status_t st = current_device(&dev, &sms);
  if (st != ATTN_OK) return st;
  while (ranks < kMaxCluster && slabs * ranks < 2 * sms && 2 * ranks <= N / 128) ranks *= 2;
  const int chunks = d / 8;
  const size_t smem = static_cast<size_t>(kMeanThreads / chunks) * d * sizeof(double);   // 32 KB
  const bool few = 2 * slabs * ranks <= sms;
  const cudaError_t e = launch_overlapped(few ? token_mean_kernel<true> : token_mean_kernel<false>, dim3(static_cast<unsigned>(slabs) * ranks),
                                          kMeanThreads, smem, stream, ranks, static_cast<const __nv_bfloat16*>(src), N, d, cos, sin, mean);
  if (e != cudaSuccess) return fail(ATTN_ERR_CUDA, "token mean: launch: %s", cudaGetErrorString(e));
  return ATTN_OK;
}

}  // namespace attnfp8
