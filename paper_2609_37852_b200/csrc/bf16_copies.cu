// Operands of BF16 mode: the tensors themselves, rounded to BF16, in both orientations.
#include <cuda_bf16.h>

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace attnfp8 {
namespace {

constexpr int kThreads = 256;
constexpr int kTokens = 64;

// Eight consecutive values as four words of two BF16 values.
__device__ __forceinline__ uint4 load8(const __nv_bfloat16* p) { return *reinterpret_cast<const uint4*>(p); }
__device__ __forceinline__ uint4 load8(const float* p) {
  const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
  return make_uint4(sm100::cvt_bf16x2(a.x, a.y), sm100::cvt_bf16x2(a.z, a.w), sm100::cvt_bf16x2(b.x, b.y), sm100::cvt_bf16x2(b.z, b.w));
}

// Groups of eight values that a thread loads ahead of its first store, and CTAs per SM that the registers have to allow.
// FP32 values take twice the registers on their way; up to head dim 128 they are held to those of eight CTAs, and 32 and 96
// have kernels of their own.  Without, one
// call on 32 heads x 4096 that writes both took 13.7 us at 96 and 19.9 at 128, now 12.4 and 19.4, and the transposed copy of 128
// heads x 8192 x 32 38.8, now 29.8.
template <typename T, int kD>
constexpr int kAhead = kD ? kTokens * kD / 8 / kThreads : 4;
template <typename T, int kD>
constexpr int kCtas = sizeof(T) == 4 && kD && kD <= 128 ? 8 : 0;        // (0: no demand)

// Memory-bound: each value read once and written once or twice.  One CTA transposes 64 tokens x d channels
// through shared memory, 16 bytes per access on both sides: a thread loads eight channels of a token, and
// stores eight tokens of two neighbouring channels, eight threads of a warp covering one 128-byte line of
// a channel.  The 16-byte groups of token t sit at group ^ (t / 8), so that the words the lanes of a warp
// read (eight token groups x four channel pairs) fall into 32 different banks.  The four operands of a
// layer with 2 x (16 + 4 + 4 + 16) heads of 4096 x 128 BF16 values: 54 us with 4-byte accesses and strided
// 2-byte shared-memory reads, 35.2 us with the loads and stores of this loop in turn, 32.4 us with every load of a thread
// ahead of its first store (168 MB: 5.2 TB/s, 0.79 of the measured copy bandwidth).
// kD is the head dim where it is one of the usual ones, which makes the index arithmetic constant and the loop one pass;
// others (0: the run-time value) take passes of four groups a thread.  Four calls each, before and now: 8 x 12 heads x 1024 x
// 64 23.3, 19.5 us; 16 x 8192 at (192, 128) 67.2, 56.9; 8/2 x 8192 x 256 43.9, 34.6; FP32 16/4 x 4096 x 256 76.2, 63.5; by the
// general kernel 2 x 16/4 x 4096 x 96 30.4, 25.7 and 16 x 4096 at (160, 32) 22.0, 22.0.
template <typename T, int kD>
__global__ void __launch_bounds__(kThreads, kCtas<T, kD>) bf16_copies_kernel(const T* src, int N, int d_rt, __nv_bfloat16* row_out,
                                                               __nv_bfloat16* col_out) {
  constexpr int kBatch = kAhead<T, kD>;
  static_assert(kD == 0 || kTokens * kD / 8 % (kBatch * kThreads) == 0, "a thread's groups fill the tile");
  const int d = kD ? kD : d_rt;
  extern __shared__ __align__(16) uint8_t smem[];
  uint4* tile = reinterpret_cast<uint4*>(smem);                       // [64][d / 8]
  const uint32_t* words = reinterpret_cast<const uint32_t*>(smem);
  const int groups = d >> 3;
  const int mask = (groups & 7) ? 3 : 7;                              // d is a multiple of 32
  const size_t slab = blockIdx.y;
  const size_t tok0 = static_cast<size_t>(blockIdx.x) * kTokens;
  const size_t first = (slab * N + tok0) * d;
  sm100::griddep_begin();
  const int total = kTokens * groups;
  for (int i0 = threadIdx.x; i0 < total; i0 += kBatch * kThreads) {
    uint4 v[kBatch];
#pragma unroll
    for (int k = 0; k < kBatch; ++k)
      if (kD || i0 + k * kThreads < total) v[k] = load8(src + first + static_cast<size_t>(i0 + k * kThreads) * 8);
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const int i = i0 + k * kThreads;
      if (!kD && i >= total) break;
      const int tok = i / groups, ch = i - tok * groups;
      tile[tok * groups + (ch ^ ((tok >> 3) & mask))] = v[k];
      if (row_out) *reinterpret_cast<uint4*>(row_out + first + static_cast<size_t>(i) * 8) = v[k];
    }
  }
  if (!col_out) return;
  __syncthreads();
  const int lane = threadIdx.x & 31, tg = lane & 7, cw = lane >> 3;   // token group, channel pair of the 16-byte group
  for (int ch = threadIdx.x >> 5; ch < groups; ch += kThreads / 32) {
    uint32_t w[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) w[t] = words[((8 * tg + t) * groups + (ch ^ (tg & mask))) * 4 + cw];
    uint32_t lo[4], hi[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      lo[k] = __byte_perm(w[2 * k], w[2 * k + 1], 0x5410);
      hi[k] = __byte_perm(w[2 * k], w[2 * k + 1], 0x7632);
    }
    __nv_bfloat16* dst = col_out + (slab * d + 8 * ch + 2 * cw) * N + tok0 + 8 * tg;
    *reinterpret_cast<uint4*>(dst) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    *reinterpret_cast<uint4*>(dst + N) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
  }
}

template <typename T, int kD>
attn_status_t launch_copies_d(const void* src, int B, int H, int N, int d, void* row_out, void* col_out,
                              cudaStream_t stream) {
  const size_t smem = static_cast<size_t>(kTokens) * d * sizeof(__nv_bfloat16);        // at most 32 KB
  dim3 grid(N / kTokens, B * H);
  const cudaError_t e = launch_overlapped(bf16_copies_kernel<T, kD>, grid, kThreads, smem, stream, 1, static_cast<const T*>(src), N, d,
                                          static_cast<__nv_bfloat16*>(row_out), static_cast<__nv_bfloat16*>(col_out));
  if (e != cudaSuccess) return fail(ATTN_ERR_CUDA, "bf16 copies: launch: %s", cudaGetErrorString(e));
  return ATTN_OK;
}

template <typename T>
attn_status_t launch_copies_t(const void* src, int B, int H, int N, int d, void* row_out, void* col_out, cudaStream_t stream) {
  if constexpr (sizeof(T) == 4) {
    if (d == 32) return launch_copies_d<T, 32>(src, B, H, N, d, row_out, col_out, stream);
    if (d == 96) return launch_copies_d<T, 96>(src, B, H, N, d, row_out, col_out, stream);
  }
  switch (d) {
    case 64: return launch_copies_d<T, 64>(src, B, H, N, d, row_out, col_out, stream);
    case 128: return launch_copies_d<T, 128>(src, B, H, N, d, row_out, col_out, stream);
    case 192: return launch_copies_d<T, 192>(src, B, H, N, d, row_out, col_out, stream);
    case 256: return launch_copies_d<T, 256>(src, B, H, N, d, row_out, col_out, stream);
    default: return launch_copies_d<T, 0>(src, B, H, N, d, row_out, col_out, stream);
  }
}

}  // namespace

attn_status_t launch_bf16_copies(const void* src, int src_dtype, int B, int H, int N, int d, void* row_out, void* col_out,
                                 cudaStream_t stream) {
  if (src_dtype == ATTN_SRC_BF16) return launch_copies_t<__nv_bfloat16>(src, B, H, N, d, row_out, col_out, stream);
  return launch_copies_t<float>(src, B, H, N, d, row_out, col_out, stream);
}

}  // namespace attnfp8
