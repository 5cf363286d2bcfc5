// Block-scaling quantiser: E4M3 codes with one E8M0 scale per 32 consecutive elements, written
// in both orientations (blocks along channels; blocks along tokens, stored transposed), for one
// tensor or for several in one launch (the four operands of a step: Q, K, V, dO), and for one tensor
// with the producer steps in front (rotary embedding, key centering, scale folding).
//
// The tiles (128 tokens x d channels, contiguous in the source) of all tensors form one list.  A
// persistent grid (two CTAs per SM) walks it; each CTA keeps a ring of two source tiles in shared
// memory (one where two would cost the second CTA), filled by bulk asynchronous copies (one
// instruction per tile, completion counted on an mbarrier), so that the next tile is in flight
// while the current one is quantised: the short tails and ramps of four separate launches
// disappear and every SM always has loads outstanding.
// Pass 1 walks the tile along channels (row copy), pass 2 along tokens (column copy).
//
// Bound by memory, nearly: Q, K, V, dO of 80 heads x 8192 x 128 in BF16 (341 MB) take 56.1 us, 6.1 TB/s or 0.93 of the measured
// copy rate; before, with 8 values a thread in pass 1 and the transposed codes staged in shared memory and copied out
// behind a third barrier, 63.3 (40.3 M instructions, now 32 M).  40 heads x 4096 x 128: 34.9 -> 30.8; 64 heads x 8192 x 192 / 128:
// 72.8 -> 59.1; 20 heads x 8192 x 256: 36.6 -> 35.1.  (Launches of column copies only
// kept the staged codes: launch_batch_o.)  Three CTAs per SM (80 registers, so fewer loads in flight) take 67.5 us on the first.
//
// Producer steps (kProd).  A pass ahead of the other two rotates the tile in place: a rotated channel is
// a BF16 value, so it goes back into the slot it came from whatever the source type.  The FP32 steps
// (minus the token mean, times the scale) are repeated by both passes, two packed operations per pair,
// instead of parking an FP32 tile.  The kernel this replaced (one tile per CTA, scalar loads of partner
// and tables, an FP32 tile parked in shared memory) took 17.4 us on average over Q and K of a layer with
// 16 + 4 heads of 4096 x 128 BF16 values, this one 12.7 us.
#include <cuda_bf16.h>

#include "common.cuh"
#include "mxfp8_device.cuh"
#include "sm100_ptx.cuh"

namespace attnfp8 {
namespace {

using namespace sm100;

constexpr int kTokens = 128;
constexpr int kThreads = 256;
constexpr int kMaxRing = 2;
constexpr int kColPitch = kTokens + 16;

struct BatchJob {
  const void* src;
  uint8_t *row_codes, *row_scales, *col_codes, *col_scales;
  int N, d;
  int first_tile;        // index of this tensor's first tile in the list
};

// The producer of a one-tensor launch (paper Appendix "Operands, Scaling, and Accumulation").
struct Producer {
  const float *cos, *sin;  // [N, d / 2], or both null: no rotary embedding
  const float* mean;       // [B * H, d], or null: no centering
  float scale;             // 1: no scaling (an exact multiplication)
};

struct BatchParams {
  BatchJob job[ATTN_QUANTIZE_MAX_JOBS];
  int n_jobs;
  int total_tiles;
  int d_max;
  int ring;              // source tiles a CTA keeps in shared memory (1 or 2)
  int* status;
  Producer prod;         // kProd only
};

// |a| max |b| per 16-bit lane; a NaN lane yields the other operand, as fmaxf does
__device__ __forceinline__ __nv_bfloat162 absmax2(__nv_bfloat162 acc, uint32_t raw) {
  return __hmax2(acc, __habs2(*reinterpret_cast<const __nv_bfloat162*>(&raw)));
}
// the two BF16 values of a word as FP32 (exact)
__device__ __forceinline__ float2 unpack_bf16x2(uint32_t raw) {
  return make_float2(__uint_as_float(raw << 16), __uint_as_float(raw & 0xFFFF0000u));
}

// Eight consecutive values as FP32, and back (the values of a BF16 row are BF16-representable).
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float* x) {
  const uint4 raw = *reinterpret_cast<const uint4*>(p);
  const float2 a = unpack_bf16x2(raw.x), b = unpack_bf16x2(raw.y), c = unpack_bf16x2(raw.z), e = unpack_bf16x2(raw.w);
  x[0] = a.x; x[1] = a.y; x[2] = b.x; x[3] = b.y; x[4] = c.x; x[5] = c.y; x[6] = e.x; x[7] = e.y;
}
__device__ __forceinline__ void load8(const float* p, float* x) {
  const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
  x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
}
__device__ __forceinline__ void store8(__nv_bfloat16* p, const float* x) {
  *reinterpret_cast<uint4*>(p) = make_uint4(cvt_bf16x2(x[0], x[1]), cvt_bf16x2(x[2], x[3]), cvt_bf16x2(x[4], x[5]), cvt_bf16x2(x[6], x[7]));
}
__device__ __forceinline__ void store8(float* p, const float* x) {
  reinterpret_cast<float4*>(p)[0] = make_float4(x[0], x[1], x[2], x[3]);
  reinterpret_cast<float4*>(p)[1] = make_float4(x[4], x[5], x[6], x[7]);
}

// Rotary embedding of a tile in place: eight pairs (c, c + d / 2) of one token per thread and step.
template <typename T>
__device__ __forceinline__ void rotate_tile(T* tile, int d, const Producer& prod, size_t tok0, int tid) {
  const int half = d >> 1, chunks = half >> 3;
#pragma unroll 2
  for (int i = tid; i < kTokens * chunks; i += kThreads) {
    const int tok = i / chunks, pc = (i - tok * chunks) * 8;
    float c[8], s[8], lo[8], hi[8];
    load8(prod.cos + (tok0 + tok) * half + pc, c);
    load8(prod.sin + (tok0 + tok) * half + pc, s);
    T* row = tile + tok * d + pc;
    load8(row, lo);
    load8(row + half, hi);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float r = rotate_bf16(lo[k], hi[k], c[k], s[k], false);
      hi[k] = rotate_bf16(hi[k], lo[k], c[k], s[k], true);
      lo[k] = r;
    }
    store8(row, lo);
    store8(row + half, hi);
  }
  fence_proxy_async_smem();        // the slot is refilled by a bulk copy later
}

// The FP32 steps behind the rotation.  Without centering the subtrahend is +0 and without scaling the
// factor is 1: both exact.
__device__ __forceinline__ float2 affine2(float2 x, float2 neg_mean, float2 scale) { return __fmul2_rn(__fadd2_rn(x, neg_mean), scale); }
__device__ __forceinline__ float2 neg_mean2(const float* mean) {        // mean: of two neighbouring channels, or null
  if (mean == nullptr) return make_float2(-0.f, -0.f);
  const float2 m = *reinterpret_cast<const float2*>(mean);
  return make_float2(-m.x, -m.y);
}

// Both passes over one source tile in shared memory ([128 tokens][d], unpadded).  kD is the head
// dim when it is one of the built ones (0: use the run-time value).  kCol: only the second pass, its codes staged in
// s_col_codes (see launch_batch_o).
template <typename T, int kD, bool kProd, bool kCol>
__device__ __forceinline__ void quantize_tile(T* tile, int d_rt, const BatchJob& job, const Producer& prod, size_t slab,
                                              size_t tok0, uint8_t* s_row_sf, uint8_t* s_col_sf, uint8_t* s_col_codes, int tid) {
  const int d = kD ? kD : d_rt;
  const int N = job.N;
  const float* mean = kProd && prod.mean != nullptr ? prod.mean + slab * d : nullptr;
  const float2 scale2 = make_float2(prod.scale, prod.scale);
  if (kProd && prod.cos != nullptr) {
    rotate_tile(tile, d, prod, tok0, tid);
    __syncthreads();
  }
  // ---- pass 1: rows.  32 bytes per thread and step, two (BF16) or four (FP32) lanes per block of 32 channels.  Every other
  // group of four lanes takes its two 16-byte halves in the other order, so that eight lanes read from all 32 banks.
  if (!kCol && job.row_codes != nullptr) {
    uint8_t* g_codes = job.row_codes + (slab * N + tok0) * d;
    constexpr int kEl = 32 / static_cast<int>(sizeof(T)), kPr = kEl / 2;        // elements and pairs of a thread
    // With producer steps a thread keeps its channels, so that their means stay in registers: whole tokens per step, some
    // threads idle at head dim 192 (32 heads x 4096, rotated and centred, 75.4 us with the means loaded at every step, now 67.9).
    // FP32 sources, which are not centred, gain by it from head dim 128 on (rotated and scaled, row copies of 32 heads x 4096:
    // 27.7 -> 26.6 us at 128, 48.3 -> 46.7 at 192, 64.7 -> 63.2 at 256) and lose below (22.7 -> 24.3 at 96, where 4 of 256 threads idle).
    constexpr bool kFixed = kProd && (sizeof(T) == 2 ? kD != 0 : kD >= 128);
    constexpr int kLanes = kFixed ? kD / kEl : 1, kTokStep = kThreads / kLanes;
    const int steps = kFixed ? (kTokens + kTokStep - 1) / kTokStep : kTokens * d / (kEl * kThreads);
    const bool swapped = (tid >> 2) & 1;
    const int off = swapped ? kEl / 2 : 0;
    auto minus_mean = [&](int ch, int k) {            // of the pair held at place k
      return neg_mean2(mean ? mean + ch + 2 * k + (k < kPr / 2 ? off : -off) : nullptr);
    };
    float2 nm[kPr];
    if (kFixed)
#pragma unroll
      for (int k = 0; k < kPr; ++k) nm[k] = minus_mean((tid % kLanes) * kEl, k);
#pragma unroll 4
    for (int s = 0; s < steps; ++s) {
      int e0 = (s * kThreads + tid) * kEl, tok = e0 / d, ch = e0 - tok * d;
      bool mine = true;
      if (kFixed) {
        tok = s * kTokStep + tid / kLanes; ch = (tid % kLanes) * kEl;
        mine = tid < kTokStep * kLanes && tok < kTokens;
        e0 = mine ? tok * d + ch : 0;
      }
      const uint4 lo = *reinterpret_cast<const uint4*>(tile + e0 + off), hi = *reinterpret_cast<const uint4*>(tile + e0 + (kEl / 2 - off));
      const uint32_t raw[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
      float amax = 0.f;
      float2 v[kPr];
      if constexpr (sizeof(T) == 2) {
        if (!kProd) {
          const __nv_bfloat162 zero = __float2bfloat162_rn(0.f);
          __nv_bfloat162 m = absmax2(absmax2(zero, raw[0]), raw[1]), n = absmax2(absmax2(zero, raw[2]), raw[3]);
          m = absmax2(m, raw[4]); n = absmax2(n, raw[5]); m = absmax2(m, raw[6]); n = absmax2(n, raw[7]);
          m = __hmax2(m, n);
          m = __hmax2(m, __shfl_xor_sync(0xffffffffu, m, 1));
          amax = fmaxf(__low2float(m), __high2float(m));
        }
#pragma unroll
        for (int k = 0; k < kPr; ++k) v[k] = unpack_bf16x2(raw[k]);
      } else {
#pragma unroll
        for (int k = 0; k < kPr; ++k) v[k] = make_float2(__uint_as_float(raw[2 * k]), __uint_as_float(raw[2 * k + 1]));
      }
      if (kProd) {
#pragma unroll
        for (int k = 0; k < kPr; ++k) v[k] = affine2(v[k], kFixed ? nm[k] : minus_mean(ch, k), scale2);
      }
      if (kProd || sizeof(T) == 4) {
#pragma unroll
        for (int k = 0; k < kPr; ++k) amax = fmaxf(amax, fmaxf(fabsf(v[k].x), fabsf(v[k].y)));
        amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 1));
        if (sizeof(T) == 4) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 2));
      }
      uint32_t byte; float inv;
      block_scale(amax, byte, inv);
      const float2 inv2 = make_float2(inv, inv);
#pragma unroll
      for (int k = 0; k < kPr; ++k) v[k] = __fmul2_rn(v[k], inv2);
      uint32_t w[kPr / 2];
#pragma unroll
      for (int k = 0; k < kPr; k += 2) w[k / 2] = cvt_e4m3x4(v[k].x, v[k].y, v[k + 1].x, v[k + 1].y);
      if (kFixed && !mine) continue;
      if constexpr (sizeof(T) == 2)
        *reinterpret_cast<uint4*>(g_codes + e0) = swapped ? make_uint4(w[2], w[3], w[0], w[1]) : make_uint4(w[0], w[1], w[2], w[3]);
      else
        *reinterpret_cast<uint2*>(g_codes + e0) = swapped ? make_uint2(w[1], w[0]) : make_uint2(w[0], w[1]);
      if ((tid & (32 / kEl - 1)) == 0) {
        const int blk = ch >> 5;
        s_row_sf[(blk >> 2) * 512 + sf_tile_offset(tok, blk & 3)] = static_cast<uint8_t>(byte);
      }
    }
  }
  // ---- pass 2: columns.  The 32 codes of a channel and token block leave from the thread that made them, one sector of
  // the transposed copy; the other sectors of the line follow from other warps, before L2 lets go of it.
  if (job.col_codes != nullptr) {
    uint8_t* g_col = job.col_codes + slab * d * N + tok0;
    const bool sector = (reinterpret_cast<uintptr_t>(job.col_codes) & 31) == 0;
    if constexpr (sizeof(T) == 2) {
      // One pair of neighbouring channels x one block of 32 tokens per thread and step: 32-bit loads, packed maxima.
      // A tile has 2 d such items: at head dims up to 64 they fill at most half of the CTA's threads, so two lanes of a
      // warp share an item there, 16 tokens each (four BF16 tensors of 8 x 12 heads x 1024 x 64: 28.7 -> 28.0 us; at head
      // dim 192, where they fill the threads one and a half times, one of 2 x 16 x 4096 took 27.8 us shared, 27.2 not).
      constexpr int kShare = kD == 32 || kD == 64 ? 2 : 1, kTok = 32 / kShare;
      const int pairs = d >> 1;
      for (int i = tid; i < pairs * 4 * kShare; i += kThreads) {
        const int item = kShare == 1 ? i : (i >> 5) * 16 + (i & 15), part = kShare == 1 ? 0 : (i >> 4) & 1;
        const int c = (item % pairs) * 2, tb = item / pairs;
        const uint32_t* col = reinterpret_cast<const uint32_t*>(tile + (tb * 32 + part * kTok) * d + c);
        uint32_t raw[kTok];
        __nv_bfloat162 m = __float2bfloat162_rn(0.f);
        float2 amax2 = make_float2(0.f, 0.f);
        const float2 nm = kProd ? neg_mean2(mean ? mean + c : nullptr) : make_float2(0.f, 0.f);
        auto value = [&](uint32_t w) { return kProd ? affine2(unpack_bf16x2(w), nm, scale2) : unpack_bf16x2(w); };
#pragma unroll
        for (int t = 0; t < kTok; ++t) {
          raw[t] = col[t * pairs];
          if (kProd) {
            const float2 x = value(raw[t]);
            amax2 = make_float2(fmaxf(amax2.x, fabsf(x.x)), fmaxf(amax2.y, fabsf(x.y)));
          } else {
            m = absmax2(m, raw[t]);
          }
        }
        if (kShare == 2 && !kProd) m = __hmax2(m, __shfl_xor_sync(0xffffffffu, m, 16));
        if (!kProd) amax2 = make_float2(__low2float(m), __high2float(m));
        if (kShare == 2 && kProd) {
          amax2.x = fmaxf(amax2.x, __shfl_xor_sync(0xffffffffu, amax2.x, 16));
          amax2.y = fmaxf(amax2.y, __shfl_xor_sync(0xffffffffu, amax2.y, 16));
        }
        uint32_t byte_lo, byte_hi;
        float2 inv2;
        block_scale(amax2.x, byte_lo, inv2.x);
        block_scale(amax2.y, byte_hi, inv2.y);
        uint32_t w_lo[kTok / 4], w_hi[kTok / 4];
#pragma unroll
        for (int t = 0; t < kTok / 4; ++t) {
          const float2 a = __fmul2_rn(value(raw[4 * t]), inv2), b = __fmul2_rn(value(raw[4 * t + 1]), inv2);
          const float2 e = __fmul2_rn(value(raw[4 * t + 2]), inv2), f = __fmul2_rn(value(raw[4 * t + 3]), inv2);
          w_lo[t] = cvt_e4m3x4(a.x, b.x, e.x, f.x);
          w_hi[t] = cvt_e4m3x4(a.y, b.y, e.y, f.y);
        }
        uint8_t* dst = g_col + static_cast<size_t>(c) * N + tb * 32;
        if constexpr (kCol) {
          uint8_t* staged = s_col_codes + c * kColPitch + tb * 32 + part * kTok;
#pragma unroll
          for (int t = 0; t < kTok / 16; ++t) {
            *reinterpret_cast<uint4*>(staged + 16 * t) = make_uint4(w_lo[4 * t], w_lo[4 * t + 1], w_lo[4 * t + 2], w_lo[4 * t + 3]);
            *reinterpret_cast<uint4*>(staged + kColPitch + 16 * t) = make_uint4(w_hi[4 * t], w_hi[4 * t + 1], w_hi[4 * t + 2], w_hi[4 * t + 3]);
          }
        } else if constexpr (kShare == 1) {
          store_32b(dst, w_lo, sector);
          store_32b(dst + N, w_hi, sector);
        } else {
          // the lanes that share an item swap halves, so that each has all 32 tokens of one of the channels
          uint32_t w[8];
#pragma unroll
          for (int t = 0; t < kTok / 4; ++t) {
            const uint32_t other = __shfl_xor_sync(0xffffffffu, part ? w_lo[t] : w_hi[t], 16);
            w[t] = part ? other : w_lo[t];
            w[kTok / 4 + t] = part ? w_hi[t] : other;
          }
          store_32b(dst + part * N, w, sector);
        }
        s_col_sf[(c >> 7) * 512 + sf_tile_offset(c & 127, tb)] = static_cast<uint8_t>(byte_lo);
        s_col_sf[(c >> 7) * 512 + sf_tile_offset((c + 1) & 127, tb)] = static_cast<uint8_t>(byte_hi);
      }
    } else {
      // one (channel, block of 32 tokens) per thread and step
      for (int item = tid; item < d * 4; item += kThreads) {
        const int c = item % d, tb = item / d;
        float x[32];
        float amax = 0.f;
        const float m = mean ? mean[c] : 0.f;
#pragma unroll
        for (int t = 0; t < 32; ++t) {
          x[t] = tile[(tb * 32 + t) * d + c];
          if (kProd) x[t] = __fmul_rn(__fsub_rn(x[t], m), prod.scale);
          amax = fmaxf(amax, fabsf(x[t]));
        }
        uint32_t byte; float inv;
        block_scale(amax, byte, inv);
        uint32_t w[8];
#pragma unroll
        for (int t = 0; t < 8; ++t)
          w[t] = cvt_e4m3x4(x[4 * t] * inv, x[4 * t + 1] * inv, x[4 * t + 2] * inv, x[4 * t + 3] * inv);
        if constexpr (kCol) {
          uint4* staged = reinterpret_cast<uint4*>(s_col_codes + c * kColPitch + tb * 32);
          staged[0] = make_uint4(w[0], w[1], w[2], w[3]);
          staged[1] = make_uint4(w[4], w[5], w[6], w[7]);
        } else {
          store_32b(g_col + static_cast<size_t>(c) * N + tb * 32, w, sector);
        }
        s_col_sf[(c >> 7) * 512 + sf_tile_offset(c & 127, tb)] = static_cast<uint8_t>(byte);
      }
    }
  }
}

// kOnly: the head dim that every tensor of the launch has, for the narrow ones (0: several, or a wide one).  A tile is then
// less work between the same barriers, and four or three CTAs per SM (64 or 80 registers, at most 64 KB) cover each other's
// better than two.  64: 28.0 -> 22.7 us on four BF16 tensors of 8 x 12 heads x 1024 tokens, 24.6 -> 18.3 us on Q, dO of
// 2 x 16 and K, V of 2 x 4 heads x 4096.  32 and 96, one BF16 tensor of 2 x 16 x 4096, scaled: 13.5 -> 8.6 and 20.9 -> 16.2 us
// (five CTAs at 32, 48 registers: 9.1).  A launch that also holds wider tensors keeps two: their tiles need the registers.
template <int kOnly>
constexpr int kCtas = kOnly == 0 ? 2 : kOnly == 32 ? 4 : kOnly == 64 ? 4 : 3;   // per SM

template <typename T, bool kProd, int kOnly, bool kCol>
__global__ void __launch_bounds__(kThreads, kCtas<kOnly>) quantize_batch_kernel(const __grid_constant__ BatchParams p) {
  extern __shared__ __align__(128) uint8_t smem[];
  const int tile_bytes_max = kTokens * p.d_max * static_cast<int>(sizeof(T));
  auto ring = [&](int slot) { return reinterpret_cast<T*>(smem + slot * tile_bytes_max); };
  const int n_ring = p.ring;
  const int n_ct_max = (p.d_max / 32 + 3) / 4, n_rt_max = (p.d_max + 127) / 128;
  const int sf_bytes = (n_ct_max + n_rt_max) * 512;                  // scale bytes of a tile, staged in two alternating buffers
  uint8_t* s_sf = smem + n_ring * tile_bytes_max;
  uint8_t* s_col_codes = s_sf + 2 * sf_bytes;                        // kCol: [d][128 + 16]
  uint64_t* full = reinterpret_cast<uint64_t*>(s_col_codes + (kCol ? p.d_max * kColPitch : 0));
  int* abort_flag = reinterpret_cast<int*>(full + kMaxRing);

  const int tid = threadIdx.x;
  const int my_tiles = (p.total_tiles - static_cast<int>(blockIdx.x) + static_cast<int>(gridDim.x) - 1) /
                       static_cast<int>(gridDim.x);

  // tile index -> (tensor, slab, token tile); the copy of a tile is one contiguous range
  auto locate = [&](int tile, int& j, int& local) {
    j = 0;
#pragma unroll
    for (int i = 1; i < ATTN_QUANTIZE_MAX_JOBS; ++i)
      if (i < p.n_jobs && tile >= p.job[i].first_tile) j = i;
    local = tile - p.job[j].first_tile;
  };
  auto issue = [&](int i) {        // thread 0: request the i-th tile of this CTA into its ring slot
    int j, local;
    locate(static_cast<int>(blockIdx.x) + i * static_cast<int>(gridDim.x), j, local);
    const uint32_t bytes = static_cast<uint32_t>(kTokens * p.job[j].d * sizeof(T));
    const uint8_t* g = static_cast<const uint8_t*>(p.job[j].src) + static_cast<size_t>(local) * bytes;
    mbar_arrive_expect_tx(&full[i % n_ring], bytes);
    bulk_load_1d(ring(i % n_ring), g, bytes, &full[i % n_ring]);
  };

  if (tid == 0) {
    for (int s = 0; s < n_ring; ++s) mbar_init(&full[s], 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  griddep_begin();
  if (tid == 0)
    for (int i = 0; i < n_ring && i < my_tiles; ++i) issue(i);
  __syncthreads();

  for (int i = 0; i < my_tiles; ++i) {
    int j, local;
    locate(static_cast<int>(blockIdx.x) + i * static_cast<int>(gridDim.x), j, local);
    const BatchJob& job = p.job[j];
    const int N = job.N, d = job.d;
    const int tiles_per_slab = N / kTokens;
    const size_t slab = static_cast<size_t>(local / tiles_per_slab);
    const int tok_tile = local % tiles_per_slab;
    const size_t tok0 = static_cast<size_t>(tok_tile) * kTokens;
    const int n_ct = (d / 32 + 3) / 4, n_rt = (d + 127) / 128;
    const bool want_row = job.row_codes != nullptr, want_col = job.col_codes != nullptr;
    T* tile = ring(i % n_ring);

    uint8_t* s_row_sf = s_sf + (i & 1) * sf_bytes;
    uint8_t* s_col_sf = s_row_sf + n_ct_max * 512;
    if (d & 127)                       // the last scale tile has bytes that no block writes
      for (int w = tid; w < sf_bytes / 4; w += kThreads) reinterpret_cast<uint32_t*>(s_row_sf)[w] = 0;
    // bounded wait: a copy that never lands ends the CTA with the time-out status, not a hang
    const bool landed = mbar_wait(&full[i % n_ring], (i / n_ring) & 1, abort_flag);
    if (__syncthreads_or(!landed)) break;        // all threads take the same way out

    if constexpr (kOnly) {
      quantize_tile<T, kOnly, kProd, kCol>(tile, kOnly, job, p.prod, slab, tok0, s_row_sf, s_col_sf, s_col_codes, tid);
    } else {
      switch (d) {                      // compile-time head dims: no integer division, constant strides
                                        // (32 and 96 here too: 1 % of a step at head dim 128 that uses the producer, 338 -> 341 us)
        case 64:  quantize_tile<T, 64, kProd, kCol>(tile, d, job, p.prod, slab, tok0, s_row_sf, s_col_sf, s_col_codes, tid); break;
        case 128: quantize_tile<T, 128, kProd, kCol>(tile, d, job, p.prod, slab, tok0, s_row_sf, s_col_sf, s_col_codes, tid); break;
        case 192: quantize_tile<T, 192, kProd, kCol>(tile, d, job, p.prod, slab, tok0, s_row_sf, s_col_sf, s_col_codes, tid); break;
        case 256: quantize_tile<T, 256, kProd, kCol>(tile, d, job, p.prod, slab, tok0, s_row_sf, s_col_sf, s_col_codes, tid); break;
        default:  quantize_tile<T, 0, kProd, kCol>(tile, d, job, p.prod, slab, tok0, s_row_sf, s_col_sf, s_col_codes, tid); break;
      }
    }
    __syncthreads();
    // the source tile is consumed: refill its slot while the staged outputs leave
    if (tid == 0 && i + n_ring < my_tiles) {
      fence_proxy_async_smem();
      issue(i + n_ring);
    }
    if (!kCol && want_row) {
      uint8_t* g = job.row_scales + (slab * tiles_per_slab + tok_tile) * n_ct * 512;
      for (int w = tid; w < n_ct * 512 / 16; w += kThreads)
        reinterpret_cast<uint4*>(g)[w] = reinterpret_cast<const uint4*>(s_row_sf)[w];
    }
    if (want_col) {
      if constexpr (kCol)
        for (int w = tid; w < d * 8; w += kThreads) {
          const int c = w >> 3, chunk = w & 7;
          *reinterpret_cast<uint4*>(job.col_codes + (slab * d + c) * N + tok0 + chunk * 16) =
              *reinterpret_cast<const uint4*>(s_col_codes + c * kColPitch + chunk * 16);
        }
      for (int rt = 0; rt < n_rt; ++rt) {
        uint8_t* g = job.col_scales + ((slab * n_rt + rt) * tiles_per_slab + tok_tile) * 512;
        for (int w = tid; w < 512 / 16; w += kThreads)
          reinterpret_cast<uint4*>(g)[w] = reinterpret_cast<const uint4*>(s_col_sf + rt * 512)[w];
      }
    }
  }
  if (tid == 0 && *abort_flag) atomicExch(p.status, static_cast<int>(ATTN_ERR_TIMEOUT));
}

static size_t batch_smem_bytes(size_t elem, int d_max, int ring, bool col) {
  const int n_ct = (d_max / 32 + 3) / 4, n_rt = (d_max + 127) / 128;
  return ring * static_cast<size_t>(kTokens) * d_max * elem + 2 * (n_ct + n_rt) * 512 +
         (col ? static_cast<size_t>(d_max) * kColPitch : 0) + 64;
}

template <typename T, bool kProd, int kOnly, bool kCol>
attn_status_t launch_batch_n(BatchParams& p, cudaStream_t stream) {
  const size_t whole_sm = 227 * 1024;
  auto fits = [&](int ctas, int ring) { return ctas * (batch_smem_bytes(sizeof(T), p.d_max, ring, kCol) + 1024) <= whole_sm; };
  // as many CTAs per SM as the registers allow come first (they cover each other's stalls), the deeper ring second
  int per_sm = kCtas<kOnly>;
  while (per_sm > 1 && !fits(per_sm, 1)) --per_sm;
  p.ring = fits(per_sm, kMaxRing) ? kMaxRing : 1;
  const size_t smem = batch_smem_bytes(sizeof(T), p.d_max, p.ring, kCol);
  int sms = 0;
  const attn_status_t st = allow_smem<quantize_batch_kernel<T, kProd, kOnly, kCol>>(whole_sm, "quantize", &sms);
  if (st != ATTN_OK) return st;
  const int resident = sms * per_sm;
  const int grid = p.total_tiles < resident ? p.total_tiles : resident;
  const cudaError_t e = launch_overlapped(quantize_batch_kernel<T, kProd, kOnly, kCol>, dim3(grid), kThreads, smem, stream, 1, p);
  if (e != cudaSuccess) return fail(ATTN_ERR_CUDA, "quantize: launch: %s", cudaGetErrorString(e));
  return ATTN_OK;
}

// A launch that writes column copies only stages the codes of a tile in shared memory and copies them out in 128-byte lines:
// without the row pass to hide behind, the stores of single sectors are what it waits for.  By the sector and staged, us, 32
// heads x 4096 and 128 x 8192: BF16 6.8, 6.4 and 39.0, 37.1 at head dim 64; 14.1, 13.0 and 91.0, 84.7 at 160; 17.5, 16.8 and 122,
// 115.6 at 224; 19.7, 19.7 and 128.8, 126.3 at 256; rotated and scaled 17.7, 15.6 and 107, 101 at 96; 28.7, 27.1 and 194, 188 at 192;
// FP32 9.0, 8.4 and 76.9, 76.3 at 96.  By the sector: head dim 32 (5.0, 5.3 and 27.5, 29.0); BF16 without the producer at 96 (7.8, 7.3
// but 48.0, 52.5), 128 (9.9, 9.3 but 62.6, 65.0) and 192 (14.1, 13.8 but 100, 103.5); FP32 from 192 on, where the staged codes
// cost the second CTA of an SM or a tile of the ring (rotated and scaled 44.0, 46.4 and 270, 347 at 192).
template <typename T, bool kProd, int kOnly>
attn_status_t launch_batch_o(BatchParams& p, cudaStream_t stream) {
  if constexpr (kOnly != 32 && (kOnly != 96 || kProd || sizeof(T) == 4)) {
    bool col = sizeof(T) == 4 ? p.d_max < 192 : kProd || (p.d_max != 96 && p.d_max != 128 && p.d_max != 192);
    for (int j = 0; j < p.n_jobs; ++j) col = col && p.job[j].row_codes == nullptr;
    if (col) return launch_batch_n<T, kProd, kOnly, true>(p, stream);
  }
  return launch_batch_n<T, kProd, kOnly, false>(p, stream);
}

template <typename T, bool kProd>
attn_status_t launch_batch_t(BatchParams& p, cudaStream_t stream) {
  bool one_dim = true;
  for (int j = 0; j < p.n_jobs; ++j) one_dim = one_dim && p.job[j].d == p.d_max;
  if (one_dim && p.d_max == 32) return launch_batch_o<T, kProd, 32>(p, stream);
  if (one_dim && p.d_max == 64) return launch_batch_o<T, kProd, 64>(p, stream);
  if (one_dim && p.d_max == 96) return launch_batch_o<T, kProd, 96>(p, stream);
  return launch_batch_o<T, kProd, 0>(p, stream);
}

void fill_params(BatchParams& p, const attn_quantize_job_t* jobs, int n_jobs, int* status) {
  p.n_jobs = n_jobs;
  p.status = status;
  int tiles = 0, d_max = 0;
  for (int j = 0; j < n_jobs; ++j) {
    const attn_quantize_job_t& in = jobs[j];
    BatchJob& b = p.job[j];
    b.src = in.src;
    b.row_codes = in.out.row_codes; b.row_scales = in.out.row_scales;
    b.col_codes = in.out.col_codes; b.col_scales = in.out.col_scales;
    b.N = in.N; b.d = in.d;
    b.first_tile = tiles;
    tiles += in.B * in.H * (in.N / kTokens);
    d_max = in.d > d_max ? in.d : d_max;
  }
  p.total_tiles = tiles;
  p.d_max = d_max;
}

}  // namespace

attn_status_t launch_quantize_batch(const attn_quantize_job_t* jobs, int n_jobs, int* status, cudaStream_t stream) {
  BatchParams p = {};
  fill_params(p, jobs, n_jobs, status);
  if (jobs[0].src_dtype == ATTN_SRC_BF16) return launch_batch_t<__nv_bfloat16, false>(p, stream);
  return launch_batch_t<float, false>(p, stream);
}

attn_status_t launch_quantize_fused(const attn_quantize_job_t& job, const float* cos, const float* sin, float scale,
                                    float* mean, int* status, cudaStream_t stream) {
  if (cos == nullptr && mean == nullptr && scale == 1.f) return launch_quantize_batch(&job, 1, status, stream);
  if (mean != nullptr) {
    const attn_status_t st = launch_token_mean(job.src, job.B * job.H, job.N, job.d, cos, sin, mean, stream);
    if (st != ATTN_OK) return st;
  }
  BatchParams p = {};
  fill_params(p, &job, 1, status);
  p.prod = Producer{cos, sin, mean, scale};
  if (job.src_dtype == ATTN_SRC_BF16) return launch_batch_t<__nv_bfloat16, true>(p, stream);
  return launch_batch_t<float, true>(p, stream);
}

}  // namespace attnfp8
