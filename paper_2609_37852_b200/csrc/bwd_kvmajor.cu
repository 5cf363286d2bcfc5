// Key-major backward kernel: dK and dV (paper Appendix "Backward Correction and Gradient
// Computation", paragraph "Score-gradient quantization", merged with the GQA group reduction).
//
// One CTA, or a cluster of two, four or eight (split_of), owns 128 keys of one (batch, KV head).  It loops over the query heads of
// the group and, for each, over the query tiles from the causal diagonal to the end, 64 query rows at a time; the CTAs of
// a cluster take every second, fourth or eighth query tile and add their sums at the end.
// Per sub-tile the tensor cores recompute the TRANSPOSED products
//     S^T  = K^ Q^^T    (128 keys x 64 queries; row-blocked FP8 copies)
//     dP^T = V^ dO^^T
// so that a softmax thread owns one key (one TMEM lane) and sees 32 consecutive query rows in
// its registers: exactly one quantisation block of the operands P^T and dS^T, whose matmuls
// contract over the query index.  The thread rebuilds P = 2^(S*scale*log2e - LSE_i*log2e),
// forms dS = P (dP - D_i) in FP32, quantises both in registers, and the tensor cores accumulate
//     dV += P^^T dO^c      dK += dS^^T Q^c      (copies of dO, Q blocked along tokens)
// in tensor memory across all query tiles and all query heads of the group: the group sum is
// an FP32 sum, rounded to BF16 once at the end.
//
// Warp roles: warp 0 TMA producer; warps 1, 2, 3 issue the S^T, dP^T and dV/dK MMAs (one warp
// cannot issue tcgen05.mma fast enough for small tiles); warps 4..19 are two softmax teams that
// take alternate sub-tiles (within a team, warp % 4 selects the 32 TMEM lanes and the column
// group w takes query columns 32w..32w+31).
//
// The kernel is a template over the operand width (element bytes 1: E4M3 codes with E8M0 block
// scales, 2: BF16 without scales; 128-byte chunks per operand row) and over which gradients it
// accumulates.  The column copies are streamed one 128-byte chunk of the query dimension at a
// time (128 queries of codes, 64 of BF16); the row copies 128 queries at a time in the narrow FP8
// configuration and 64 otherwise.  When dV and dK together do not fit in tensor memory beside the
// score tiles (qk head dim above 128), the launcher runs the kernel twice: a pass that rebuilds P
// and accumulates dV, and a pass that rebuilds P and dS and accumulates dK.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "common.cuh"
#include "mma_issue.cuh"
#include "mxfp8_device.cuh"
#include "sm100_ptx.cuh"
#include "work_order.cuh"

namespace attnfp8 {

namespace {

using namespace sm100;

constexpr int kTile = 128;
constexpr int kSub = 64;
constexpr int kTeams = 2;                       // softmax teams; team t takes sub-tiles u with u % kTeams == t
constexpr int kTeamThreads = 256;               // 8 warps: 4 TMEM lane quadrants x 2 column groups
constexpr int kThreads = 128 + kTeams * kTeamThreads;
constexpr float kLog2e = 1.4426950408889634f;
constexpr int kSmemLimit = 232448;              // dynamic shared memory a CTA may ask for

enum KvMode { kBoth = 0, kDvOnly = 1, kDkOnly = 2 };

// Operand geometry, ring depths and tensor-memory map of one instantiation.
template <int kEB_, int kCq_, int kCv_, int kMode_, int kEBv_ = kEB_, int kDkTile_ = -1>
struct KvCfg {
  static constexpr int kEB = kEB_, kCq = kCq_, kCv = kCv_, kMode = kMode_;
  static constexpr int kEBv = kEBv_;                   // bytes per element of the V / dO row operands (dP^T only):
                                                       // 2 with kEB == 1 is the protected-dP ablation
  static constexpr bool kFp8 = kEB == 1;
  static constexpr bool kFp8v = kEBv == 1;
  static constexpr bool kHasDv = kMode != kDkOnly;     // accumulates dV (needs P^)
  static constexpr bool kHasDk = kMode != kDvOnly;     // accumulates dK (needs dP^T, D, dS^)
  static constexpr int kRq = kCq / kEB > 0 ? (kCq + kEB - 1) / kEB : 1;   // 128-row tiles of the Q^c operand (dqk / 128, rounded up)
  static constexpr int kRv = (kCv + kEBv - 1) / kEBv;                     // 128-row tiles of the dO^c operand
  // BF16 at head dim 256: K, V and one row stage fill shared memory, so a dK pass takes one 128-column
  // tile of dK (kDkTile = 0, 1) and the launcher runs one pass per tile
  static constexpr int kDkTile = kDkTile_;
  static constexpr int kRqAcc = kDkTile >= 0 ? 1 : kRq;                   // 128-row tiles of Q^c a pass accumulates into dK
  // Per query tile the CTA streams a 'row' set (Q and dO row copies, their scales, LSE, D: read by
  // the S^T / dP^T MMAs and the softmax) and a 'col' set (Q and dO column copies: read by the dV /
  // dK MMAs).  The row set is released early and gets the deeper ring, so that a reload never sits
  // between the end of one tile's gradient MMAs and the start of the next tile's scores.
  static constexpr int kRowTok = (kFp8 && kCq == 1 && kCv == 1) ? 128 : 64;   // queries per row stage
  static constexpr int kColTok = kTile / kEB;                                 // queries per col stage
  static constexpr int kSubPerRow = kRowTok / kSub, kSubPerCol = kColTok / kSub;
  static constexpr int kKvBytes = (kCq + (kHasDk ? kCv : 0)) * kTile * 128;
  static constexpr int kRowBytes = (kCq + (kHasDk ? kCv : 0)) * kRowTok * 128;
  // (192,128) with both gradients in one pass (see kTight below): the Q^c stage holds the 192 rows it is
  // loaded with, not two full row tiles, which leaves room for a third row stage
  static constexpr bool kTightDims = kMode == kBoth && ((kFp8 && kFp8v && kCq == 2 && kCv == 1) || (kEB == 2 && kEBv == 2 && kCq == 3 && kCv == 2));
  static constexpr int kQcRows = kTightDims ? 192 : kRqAcc * kTile;
  static constexpr int kColBytes = ((kHasDk ? kQcRows : 0) + (kHasDv ? kRv * kTile : 0)) * 128;
  // rings shrink to one stage where two do not fit (wide heads in BF16 mode): loads and MMAs of
  // successive steps then no longer overlap
  static constexpr int kColStages = kKvBytes + 2 * kRowBytes + 2 * kColBytes <= 210 * 1024 ? 2 : 1;
  static constexpr int kRowRaw = (216 * 1024 - kKvBytes - kColStages * kColBytes) / kRowBytes;
  static constexpr bool kTwoRowsFit = kKvBytes + kColStages * kColBytes + 2 * kRowBytes <= 214 * 1024;
  static constexpr int kRowCap = 3;
  static constexpr int kRowStages = kRowRaw < 2 ? (kTwoRowsFit ? 2 : 1) : (kRowRaw > kRowCap ? kRowCap : kRowRaw);
  // 64-query row stages (one sub-tile each): -LSE*log2(e) and -D of a sub-tile live in a small ring
  // of their own, written by the preparation warp, so that the operand part of a row stage is released as soon
  // as the S^T / dP^T MMAs that read it have run, not when the softmax is done with the sub-tile: the reload is
  // in flight a whole softmax step earlier.  Slot reuse is safe kRowStages + 3 sub-tiles later (the row load
  // that precedes the rewrite waits for the MMAs of sub-tile u + 3, which are issued after the team of u has
  // taken S of u + 2, i.e. finished u); an even count keeps each slot with one team.
  // (not at (192,128) in BF16 mode, one pass: a single column stage paces that kernel and the change cost 5 %)
  static constexpr bool kEarly = kRowTok == kSub && !(kEB == 2 && kTightDims);
  // arrivals that release a row stage: the commits behind the S^T and dP^T MMAs; without dP^T the preparation warp in
  // the place of the latter, once it has seen the stage (and read LSE out of it, where LSE arrives in the stage).  It has
  // to be one of them: the softmax releases S before it asks for LSE, so the S^T issuer can be three sub-tiles ahead of
  // a preparation warp that waits for LSE from memory, and a stage filled anew in the meantime would complete the phase
  // after the one that this warp has yet to see (FP8 dV pass at head dim 256: one call in about 600 waited for ever).
  static constexpr int kRowReleases = !kEarly ? 1 : 2;
  static constexpr int kLseSlots = kEarly ? ((kRowStages + 4) & ~1) : kRowStages;
  // Tensor memory.  BF16 mode has no scale factors, which leaves columns for a second S^T buffer (one per team) when
  // P^ and dS^ keep one operand buffer each; S^T and dP^T are then released one by one (kApart: the softmax takes S,
  // releases it, and takes dP after its exponentials), so that no team waits for the turnaround of a score buffer
  // (issue, completion, wake-up, load, release) the other still uses: dK / dV of the 4K layer 297 -> 276 us.  FP8 at
  // the same head dims fits as well with single scale slots, and loses (8K layer, 725 -> 770 us): its teams then are
  // busy all the time, and an exponential loop apart from the dS arithmetic leaves the other pipes idle.
  //   BF16, head dims 64 and 128:  2 x 64 + 64 + 32 + 32 + 128 + 128 = 512
  // (192,128): dV 128 + dK 192 columns beside the score tiles fill tensor memory exactly when the P^ / dS^ operands and
  // every scale-factor slot are single and the scale columns of the two gradient products are shared (one issuing
  // thread uses them one after the other; its copies and MMAs run in the order issued):
  //   FP8   64 + 64 + 16 + 16 + 128 + 192 + SF 32 = 512       BF16   64 + 64 + 32 + 32 + 128 + 192 = 512
  static constexpr bool kTight = kTightDims;
  static constexpr bool kApart = kMode == kBoth && kEB == 2 && !kTight;
  static constexpr int kSBufs = kApart ? 2 : 1;
  static constexpr int kOpBufs = kTight || kApart ? 1 : 2;   // P^ / dS^ operand buffers
  static constexpr int kSl = kTight ? 1 : 2;           // scale-factor slots per streamed stage
  static constexpr int kOpCols = 16 * kEB;             // columns of one P^ / dS^ buffer (64 queries)
  static constexpr uint32_t kColS = 0;
  static constexpr uint32_t kColdP = 64 * kSBufs;
  static constexpr uint32_t kColP = kColdP + (kHasDk ? 64 : 0);
  static constexpr uint32_t kColdS = kColP + (kHasDv ? kOpBufs * kOpCols : 0);
  static constexpr uint32_t kColdV = kColdS + (kHasDk ? kOpBufs * kOpCols : 0);
  static constexpr uint32_t kColdK = kColdV + (kHasDv ? 128 * kRv : 0);
  static constexpr uint32_t kColSFK = kColdK + (kHasDk ? (kTight ? 192 : 128 * kRqAcc) : 0);
  static constexpr uint32_t kColSFV = kColSFK + 4 * kCq;
  static constexpr uint32_t kColSFQ = kColSFV + (kHasDk && kFp8v ? 4 * kCv : 0);   // kSl slots
  static constexpr uint32_t kColSFdO = kColSFQ + 4 * kSl * kCq;                // kSl slots
  static constexpr uint32_t kColSFP = kColSFdO + (kHasDk && kFp8v ? 4 * kSl * kCv : 0);  // kOpBufs x 4
  static constexpr uint32_t kColSFdS = kTight ? kColSFP : kColSFP + (kHasDv ? 4 * kOpBufs : 0);   // kOpBufs x 4
  static constexpr uint32_t kColSFdOc = kColSFdS + (kTight ? 4 : (kHasDk ? 4 * kOpBufs : 0));     // kSl slots x row tiles
  static constexpr uint32_t kColSFQc = kTight ? kColSFdOc : kColSFdOc + (kHasDv ? 4 * kSl * kRv : 0);   // kSl slots x row tiles
  static constexpr uint32_t kColsUsed = kFp8 ? (kTight ? kColSFQc + 4 : kColSFQc + (kHasDk ? 4 * kSl * kRqAcc : 0)) : kColSFK;
  static constexpr uint32_t kTmemCols = 512;
  static_assert(kColsUsed <= 512, "tensor memory exceeded");
};

template <class C>
struct KvRowStage {
  alignas(1024) uint8_t q[C::kCq][C::kRowTok * 128];                    // Q row copy  [queries][dqk]
  alignas(1024) uint8_t dO[C::kHasDk ? C::kCv : 1][C::kHasDk ? C::kRowTok * 128 : 16];   // dO row copy [queries][dv]
  alignas(16) uint8_t sf_q[C::kCq * 512];
  alignas(16) uint8_t sf_dO[C::kCv * 512];
  alignas(16) float lse[C::kRowTok];
  alignas(16) float delta[C::kRowTok];
  alignas(16) float neg_lse2[C::kRowTok];       // -LSE * log2(e), written by the prep warp
};
template <class C>
struct KvColStage {
  alignas(1024) uint8_t qc[C::kHasDk ? C::kQcRows * 128 : 16];   // Q col copy  [dqk][queries]
  alignas(1024) uint8_t dOc[C::kHasDv ? C::kRv * kTile * 128 : 16];     // dO col copy [dv][queries]
  alignas(16) uint8_t sf_qc[C::kRqAcc * 512];
  alignas(16) uint8_t sf_dOc[C::kRv * 512];
};

template <class C>
struct KvSmem {
  alignas(1024) uint8_t k[C::kCq][kTile * 128];
  alignas(1024) uint8_t v[C::kHasDk ? C::kCv : 1][C::kHasDk ? kTile * 128 : 16];
  KvRowStage<C> rst[C::kRowStages];
  KvColStage<C> cst[C::kColStages];
  alignas(16) uint8_t sf_k[C::kCq * 512];
  alignas(16) uint8_t sf_v[C::kCv * 512];
  alignas(16) uint8_t sf_p[2][512];
  alignas(16) uint8_t sf_ds[2][512];
  uint64_t kv_full;
  uint64_t row_full[C::kRowStages], row_empty[C::kRowStages];
  uint64_t col_full[C::kColStages], col_empty[C::kColStages];
  uint64_t lse_ready[C::kLseSlots];
  alignas(16) float lse_ring[C::kEarly ? C::kLseSlots : 1][kSub];     // kEarly: -LSE * log2(e) of a sub-tile
  alignas(16) float delta_ring[C::kEarly ? C::kLseSlots : 1][kSub];   // kEarly: -D
  // Hand-offs between the issuing threads and the softmax teams, per team: a team takes every other sub-tile, and a
  // parity wait on a barrier that completes once per sub-tile would pass at once for a waiter a whole phase behind.
  // s_full stands for S, LSE and (unless kApart) dP; dp_full / dp_free for dP taken apart.
  uint64_t s_full[kTeams], s_free[kTeams];
  uint64_t dp_full[kTeams], dp_free[kTeams];
  // P^ and dS^ on their way back.  "free": the team that writes the buffer next waits on its own.  With a single
  // operand buffer P^ and dS^ are handed over separately (p_full / p_free for P^), so that the next P^ is written
  // while the dK MMAs still run.
  uint64_t p_full, p_free[2];
  uint64_t op_full[2], op_free[2];
  uint64_t done;
  uint64_t drain[3];
  uint32_t tmem_base;
  int abort_flag;
};

struct KvParams {
  const uint8_t *k_sf, *v_sf, *q_sf, *dO_sf, *qc_sf, *dOc_sf;
  const float* lse;
  const float* delta;
  __nv_bfloat16* dk;
  __nv_bfloat16* dv_out;
  int sectors;              // dk and dv_out start on 32-byte sectors
  int* status;
  int N, Nk, q0t, Hq, Hkv, dqk, dv, causal;   // N query rows, Nk keys, q0t: tile offset of the causal diagonal
  int kv_lim;               // without the causal mask: last real key of the last key tile (127: all real)
  int tail_wait;            // launched behind another key-major pass of the same call (see launch_kvmajor_t)
  int* tickets;             // the dQ kernel's ticket counter, to be cleared ahead of it; or null
  int slabs, group;         // (sequence, KV head) pairs, and how many of them run together (work_order.cuh)
  int split;                // CTAs (a cluster) that share the query tiles of one key tile: 1, 2, 4 or 8
  float scale, scale_log2;
};

__device__ __forceinline__ bool last_cta() {
  return blockIdx.x == gridDim.x - 1 && blockIdx.y == gridDim.y - 1 && blockIdx.z == gridDim.z - 1;
}

// kShared: a cluster of p.split CTAs shares the query tiles of a key tile (see split_of).
template <class C, bool kShared>
__global__ void __launch_bounds__(kThreads, 1)
kvmajor_kernel(const KvParams p, const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
               const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_dO,
               const __grid_constant__ CUtensorMap tm_qc, const __grid_constant__ CUtensorMap tm_dOc) {
  // declared with the alignment the swizzled operand tiles need, so that the compiler keeps the
  // shared state space of every access derived from it (checked below)
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  constexpr bool kFp8 = C::kFp8, kFp8v = C::kFp8v, kHasDv = C::kHasDv, kHasDk = C::kHasDk;
  constexpr int kEB = C::kEB, kCq = C::kCq, kCv = C::kCv, kRq = C::kRqAcc, kRv = C::kRv;
  constexpr int kRowStages = C::kRowStages, kColStages = C::kColStages, kRowTok = C::kRowTok;
  constexpr int kSubPerRow = C::kSubPerRow, kSubPerCol = C::kSubPerCol, kOpCols = C::kOpCols;
  constexpr bool kTight = C::kTight;
  constexpr int kOpBufs = C::kOpBufs, kSl = C::kSl;
  // 64-query row stages: LSE and D of a stage are fetched by the preparation warp with plain loads, one stage
  // ahead, instead of two more bulk copies per stage by the producer thread (which paces the kernel there)
  // (FP8 only: in BF16 mode the producer is not what paces the kernel, and the change cost 5 % there)
  constexpr bool kPrepLoads = kFp8 && C::kRowTok == kSub;
  constexpr bool kSplit = kOpBufs == 1;          // single operand buffer: P^ and dS^ are handed over separately
  constexpr bool kApart = C::kApart;
  // One CTA per key tile in BF16 mode at head dim 128 stores 16 bytes at a time: dK / dV of 2 x 16/4 heads x 4096, calls in a
  // row below the power cap, 265.3 us by the sector, 259.9 so; 32/8 x 8192 1133 and 1114.  (Head dim 64 gains as FP8 does: 8 x 12
  // x 1024 89.3 -> 86.2.  So does a cluster, which stores slices of rows: 16/4 heads x 4096 138.3 -> 137.1, 8/1 x 512 19.45 -> 19.36.)
  constexpr bool kSectors = !(C::kApart && C::kCq == 2);
  constexpr int kSBufs = C::kSBufs;
  constexpr uint32_t kColS = C::kColS, kColdP = C::kColdP, kColP = C::kColP, kColdS = C::kColdS, kColdV = C::kColdV,
                     kColdK = C::kColdK, kColSFK = C::kColSFK, kColSFV = C::kColSFV, kColSFQ = C::kColSFQ,
                     kColSFdO = C::kColSFdO, kColSFP = C::kColSFP, kColSFdS = C::kColSFdS, kColSFdOc = C::kColSFdOc,
                     kColSFQc = C::kColSFQc, kTmemCols = C::kTmemCols;
  KvSmem<C>& sm = *reinterpret_cast<KvSmem<C>*>(smem_raw);
  if (smem_u32(smem_raw) & 1023u) {               // never expected: report instead of computing garbage
    if (threadIdx.x == 0) atomicExch(p.status, static_cast<int>(ATTN_ERR_ALIGNMENT));
    return;
  }
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // The order of work_order.cuh, without its divisions, which cost the softmax loop registers: blocks are handed out
  // x-fastest, z-slowest, (sequence, KV head) pairs within a group along x, key tiles along y (the earliest keys are the
  // heaviest under the causal mask), groups along z.  The last group may be short of pairs.
  const int jt = blockIdx.y;
  const int split = kShared ? p.split : 1, part = !kShared ? 0 : static_cast<int>(blockIdx.x) % split;
  const int slab = static_cast<int>(blockIdx.z) * p.group + static_cast<int>(blockIdx.x) / split;
  if (slab >= p.slabs) {                          // (all CTAs of a cluster)
    if (p.tail_wait && tid == 0 && last_cta()) griddep_wait();
    return;
  }
  const int G = p.Hq / p.Hkv;
  const int tiles_n = p.N / kTile, tiles_nk = p.Nk / kTile;
  const int it0 = p.causal ? max(jt - p.q0t, 0) : 0;   // first query tile that sees these keys
  const int tiles_per_head = tiles_n - it0;
  // the query tiles of all heads of the group in one list; a CTA of a cluster walks every split-th of them
  const int n_list = G * tiles_per_head;
  const int n_qtiles = part < n_list ? (n_list - part + split - 1) / split : 0;
  const int n_sub = 2 * n_qtiles;
  const int nk_qk = p.dqk * kEB / 32, nk_v = p.dv * C::kEBv / 32;   // 32-byte K steps of S^T and dP^T
  // columns of dK (rows of Q^c) this pass accumulates: all of them, or one tile of 128
  const int dk_col0 = C::kDkTile >= 0 ? 128 * C::kDkTile : 0;
  const int dk_cols = C::kDkTile >= 0 ? min(128, p.dqk - dk_col0) : p.dqk;
  volatile int* abort_flag = &sm.abort_flag;

  if (tid == 0) {
    mbar_init(&sm.kv_full, 1);
    for (int s = 0; s < kRowStages; ++s) {
      // released once the softmax teams are done with the rows (kEarly: once the S^T and dP^T MMAs have read them)
      mbar_init(&sm.row_full[s], 1); mbar_init(&sm.row_empty[s], C::kRowReleases);
    }
    for (int s = 0; s < C::kLseSlots; ++s) mbar_init(&sm.lse_ready[s], 1);   // one arrival by the prep warp
    for (int s = 0; s < kColStages; ++s) { mbar_init(&sm.col_full[s], 1); mbar_init(&sm.col_empty[s], 1); }
    for (int t = 0; t < kTeams; ++t) {
      mbar_init(&sm.s_full[t], !kHasDk ? 1 : (kApart ? 2 : 3)); mbar_init(&sm.s_free[t], kTeamThreads);
      mbar_init(&sm.dp_full[t], 1); mbar_init(&sm.dp_free[t], kTeamThreads);
    }
    for (int i = 0; i < 2; ++i) { mbar_init(&sm.op_full[i], kTeamThreads); mbar_init(&sm.op_free[i], 1); mbar_init(&sm.p_free[i], 1); }
    mbar_init(&sm.p_full, kTeamThreads);
    for (int i = 0; i < 3; ++i) mbar_init(&sm.drain[i], 1);
    mbar_init(&sm.done, 1);
    sm.abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(&sm.tmem_base, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  // The query-major kernel of the same call is queued behind this grid: its CTAs take the SMs that this grid's last
  // wave leaves idle, and do not wait for this grid (nothing they do depends on its output).  So they must not start
  // before what both read is complete, and their ticket counter is cleared: the wait comes first.  (A pass behind
  // another key-major pass has nothing to wait for: that pass had waited when it let this one start.)
  if (!p.tail_wait) griddep_wait();
  if (p.tickets != nullptr && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0) {
    if (tid == 0) {
      atomicExch(p.tickets, 0);
      __threadfence();
    }
    __syncthreads();
  }
  griddep_launch_dependents();
  const uint32_t tmem = sm.tmem_base;
  bool stores = false;                                // this thread takes part in the epilogue
  // kApart: a padded key of a ragged sequence (no causal mask) has a row of dV and dK of its own and nothing else, so its
  // rows are stored as zeros, whatever its probabilities and score gradients came to (NaN behind an Inf in dO).  The other
  // configurations make the latter zero in the loop: without that branch their loops come out 1 % slower (dK / dV and dQ
  // of the 8K layer), with it the BF16 one does (dK / dV of the 4K layer at the power cap 294 us, 290 without).
  const int real_rows = kApart && !p.causal && jt == tiles_nk - 1 ? p.kv_lim + 1 : kTile;

  if (warp == 0) {
    // ------------------------------------------------------------------ producer
    if (lane == 0) {
      prefetch_tmap(&tm_k); prefetch_tmap(&tm_v); prefetch_tmap(&tm_q); prefetch_tmap(&tm_dO);
      prefetch_tmap(&tm_qc); prefetch_tmap(&tm_dOc);
      mbar_arrive_expect_tx(&sm.kv_full, kCq * (kTile * 128 + (kFp8 ? 512 : 0)) +
                                             (kHasDk ? kCv * (kTile * 128 + (kFp8v ? 512 : 0)) : 0));
      for (int c = 0; c < kCq; ++c) tma_load_2d(sm.k[c], &tm_k, &sm.kv_full, 128 * c, slab * p.Nk + jt * kTile);
      if (kFp8) bulk_load_1d(sm.sf_k, p.k_sf + (static_cast<size_t>(slab) * tiles_nk + jt) * kCq * 512, kCq * 512, &sm.kv_full);
      if (kHasDk) {
        for (int c = 0; c < kCv; ++c) tma_load_2d(sm.v[c], &tm_v, &sm.kv_full, 128 * c, slab * p.Nk + jt * kTile);
        if (kFp8v) bulk_load_1d(sm.sf_v, p.v_sf + (static_cast<size_t>(slab) * tiles_nk + jt) * kCv * 512, kCv * 512, &sm.kv_full);
      }
      int issued_row = 0, issued_col = 0;
      bool ok = true;
      for (int u = 0; u < n_sub && ok; ++u) {
        const int n = part + split * (u >> 1), half = u & 1;
        const int q_slab = slab * G + n / tiles_per_head, it = it0 + n % tiles_per_head;
        const size_t sf_tile = static_cast<size_t>(q_slab) * tiles_n + it;
        if (u % kSubPerRow == 0) {
          const int ri = u / kSubPerRow, rs = ri % kRowStages;
          const int tok0 = it * kTile + (kSubPerRow == 1 ? half * kSub : 0);     // first query of the stage
          ok = mbar_wait(&sm.row_empty[rs], ((ri / kRowStages) & 1) ^ 1, abort_flag);
          if (!ok) break;
          KvRowStage<C>& r = sm.rst[rs];
          mbar_arrive_expect_tx(&sm.row_full[rs], kCq * (kRowTok * 128 + (kFp8 ? 512 : 0)) +
                                                      (kHasDk ? kCv * (kRowTok * 128 + (kFp8v ? 512 : 0)) : 0) +
                                                      (kPrepLoads ? 0 : (kHasDk ? 2 : 1) * kRowTok * 4));
          for (int c = 0; c < kCq; ++c) tma_load_2d(r.q[c], &tm_q, &sm.row_full[rs], 128 * c, q_slab * p.N + tok0);
          if (kFp8) bulk_load_1d(r.sf_q, p.q_sf + sf_tile * kCq * 512, kCq * 512, &sm.row_full[rs]);
          if (!kPrepLoads) bulk_load_1d(r.lse, p.lse + static_cast<size_t>(q_slab) * p.N + tok0, kRowTok * 4, &sm.row_full[rs]);
          if (kHasDk) {
            for (int c = 0; c < kCv; ++c) tma_load_2d(r.dO[c], &tm_dO, &sm.row_full[rs], 128 * c, q_slab * p.N + tok0);
            if (kFp8v) bulk_load_1d(r.sf_dO, p.dO_sf + sf_tile * kCv * 512, kCv * 512, &sm.row_full[rs]);
            if (!kPrepLoads) bulk_load_1d(r.delta, p.delta + static_cast<size_t>(q_slab) * p.N + tok0, kRowTok * 4, &sm.row_full[rs]);
          }
          ++issued_row;
        }
        if (u % kSubPerCol == 0) {
          const int ci = u / kSubPerCol, cs = ci % kColStages;
          const int x0 = (it * kTile + (kSubPerCol == 1 ? half * kSub : 0)) * kEB;   // byte offset along the query dim
          ok = mbar_wait(&sm.col_empty[cs], ((ci / kColStages) & 1) ^ 1, abort_flag);
          if (!ok) break;
          KvColStage<C>& c = sm.cst[cs];
          mbar_arrive_expect_tx(&sm.col_full[cs], (kHasDk ? dk_cols * 128 + (kFp8 ? kRq * 512 : 0) : 0) +
                                                      (kHasDv ? p.dv * 128 + (kFp8 ? kRv * 512 : 0) : 0));
          if (kHasDk) {
            tma_load_2d(c.qc, &tm_qc, &sm.col_full[cs], x0, q_slab * p.dqk + dk_col0);
            if (kFp8)
              for (int r = 0; r < kRq; ++r)
                bulk_load_1d(c.sf_qc + 512 * r, p.qc_sf + ((static_cast<size_t>(q_slab) * kRq + r) * tiles_n + it) * 512, 512,
                             &sm.col_full[cs]);
          }
          if (kHasDv) {
            tma_load_2d(c.dOc, &tm_dOc, &sm.col_full[cs], x0, q_slab * p.dv);
            if (kFp8)
              for (int r = 0; r < kRv; ++r)
                bulk_load_1d(c.sf_dOc + 512 * r, p.dOc_sf + ((static_cast<size_t>(q_slab) * kRv + r) * tiles_n + it) * 512, 512,
                             &sm.col_full[cs]);
          }
          ++issued_col;
        }
      }
      if (!ok) {
        int dummy = 0;
        for (int n = max(0, issued_row - kRowStages); n < issued_row; ++n)
          mbar_wait(&sm.row_full[n % kRowStages], (n / kRowStages) & 1, &dummy);
        for (int n = max(0, issued_col - kColStages); n < issued_col; ++n)
          mbar_wait(&sm.col_full[n % kColStages], (n / kColStages) & 1, &dummy);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ S^T issuer
    // The products are spread over three issuing warps, so that none waits behind another's barriers;
    // orderings that a single issuer would give for free are carried by mbarriers instead.
    if (elect_one()) {
      const uint64_t desc_k = make_desc_sw128(smem_u32(sm.k[0]));
      bool ok = mbar_wait(&sm.kv_full, 0, abort_flag);
      // (a CTA of a cluster may have no query tile: no commit would follow its copies)
      if (ok && kFp8 && (!kShared || n_sub > 0)) {
        tc_fence_after_sync();
        sf_copy_tiles<kCq, true>(tmem + kColSFK, sm.sf_k);
      }
      // the row ring is walked with a running (stage, phase) pair: a division by a ring depth of 3 in every
      // iteration is felt in the issue rate
      int s = 0;
      uint32_t s_phase = 0;
      for (int u = 0; u < n_sub && ok; ++u) {
        const int half = u & 1, ri = u / kSubPerRow, slot = kSl == 2 ? (ri & 1) : 0, sub_r = u % kSubPerRow;
        if (u > 0 && sub_r == 0 && ++s == kRowStages) { s = 0; s_phase ^= 1u; }
        KvRowStage<C>& st = sm.rst[s];
        if (sub_r == 0) {
          ok = mbar_wait(&sm.row_full[s], s_phase, abort_flag);
          if (!ok) break;
          tc_fence_after_sync();
          if (kFp8 && kSl == 2) sf_copy_tiles<kCq, true>(tmem + kColSFQ + 4 * kCq * slot, st.sf_q);
        }
        if (u >= kSBufs) {
          // the team that had this buffer last has pulled S into registers
          const int v = u - kSBufs;
          ok = mbar_wait(&sm.s_free[v % kTeams], (v / kTeams) & 1, abort_flag);
          if (!ok) break;
          tc_fence_after_sync();
        }
        if (kFp8 && kSl == 1 && sub_r == 0) sf_copy_tiles<kCq, true>(tmem + kColSFQ, st.sf_q);
        const uint64_t desc_q = make_desc_sw128(smem_u32(st.q[0])) + sub_r * (kSub * 128 / 16);
        issue_ss<kFp8, kCq, kSub, kTile * 128 / 16, kRowTok * 128 / 16, true>(
            tmem + kColS + 64 * (u % kSBufs), desc_k, desc_q, nk_qk, tmem + kColSFK, tmem + kColSFQ + 4 * kCq * slot + 2 * half);
        mma_commit(&sm.s_full[u % kTeams]);
        if (C::kEarly) mma_commit(&sm.row_empty[s]);   // the row operands of this sub-tile have been read
      }
      if (!ok) {
        int dummy = 0;
        mma_commit(&sm.drain[0]);
        mbar_wait(&sm.drain[0], 0, &dummy);
      }
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------------ dP^T issuer + LSE preparation
    const uint64_t desc_v = make_desc_sw128(smem_u32(sm.v[0]));
    bool ok = __all_sync(0xffffffffu, mbar_wait(&sm.kv_full, 0, abort_flag));   // (one answer for the warp: elect_one needs it whole)
    if (ok && kFp8v && kHasDk && (!kShared || n_sub > 0)) {
      tc_fence_after_sync();
      if (elect_one()) sf_copy_tiles<kCv, true>(tmem + kColSFV, sm.sf_v);
    }
    int s = 0;                                        // running (stage, phase) of the row ring
    uint32_t s_phase = 0;
    // kPrepLoads: LSE and D of the next row stage (= sub-tile), in flight while this one is handled
    // (head, query tile) of the stage fetched next
    int pf_h = slab * G + (kShared ? part / tiles_per_head : 0), pf_it = it0 + (kShared ? part % tiles_per_head : 0);
    float4 pf_l = make_float4(0.f, 0.f, 0.f, 0.f), pf_d = make_float4(0.f, 0.f, 0.f, 0.f);
    auto prefetch = [&](int uu) {
      if (4 * lane < kRowTok) {
        const size_t at = static_cast<size_t>(pf_h) * p.N + pf_it * kTile + (uu & 1) * kSub + 4 * lane;
        pf_l = *reinterpret_cast<const float4*>(p.lse + at);
        if (kHasDk) pf_d = *reinterpret_cast<const float4*>(p.delta + at);
      }
      if (uu & 1) {
        if (kShared) {
          pf_it += split;
          while (pf_it >= tiles_n) { pf_it -= tiles_per_head; ++pf_h; }
        } else if (++pf_it == tiles_n) { pf_it = it0; ++pf_h; }
      }
    };
    if (kPrepLoads && n_sub > 0) prefetch(0);
    int ls = 0;                                       // kEarly: slot of the LSE / D ring (sub-tile u modulo its depth)
    for (int u = 0; u < n_sub && ok; ++u) {
      const int half = u & 1, ri = u / kSubPerRow, slot = kSl == 2 ? (ri & 1) : 0, sub_r = u % kSubPerRow;
      if (u > 0 && sub_r == 0 && ++s == kRowStages) { s = 0; s_phase ^= 1u; }
      KvRowStage<C>& st = sm.rst[s];
      if (sub_r == 0) {
        ok = __all_sync(0xffffffffu, mbar_wait(&sm.row_full[s], s_phase, abort_flag));
        if (!ok) break;
        if (kPrepLoads) {
          if (!kHasDk) mbar_arrive_warp(&sm.row_empty[s]);
          if (4 * lane < kRowTok) {
            *reinterpret_cast<float4*>(&sm.lse_ring[ls][4 * lane]) =
                make_float4(-pf_l.x * kLog2e, -pf_l.y * kLog2e, -pf_l.z * kLog2e, -pf_l.w * kLog2e);
            if (kHasDk) *reinterpret_cast<float4*>(&sm.delta_ring[ls][4 * lane]) = make_float4(-pf_d.x, -pf_d.y, -pf_d.z, -pf_d.w);
          }
          if (u + 1 < n_sub) prefetch(u + 1);
        } else
        // every lane turns four LSE values into -LSE*log2(e) for the softmax teams
        if (4 * lane < kRowTok) {
          const float4 l = *reinterpret_cast<const float4*>(&st.lse[4 * lane]);
          *reinterpret_cast<float4*>(C::kEarly ? &sm.lse_ring[ls][4 * lane] : &st.neg_lse2[4 * lane]) =
              make_float4(-l.x * kLog2e, -l.y * kLog2e, -l.z * kLog2e, -l.w * kLog2e);
          if (kHasDk) {                                 // and the row correction into its negative (in place, or into the ring)
            const float4 d = *reinterpret_cast<const float4*>(&st.delta[4 * lane]);
            *reinterpret_cast<float4*>(C::kEarly ? &sm.delta_ring[ls][4 * lane] : &st.delta[4 * lane]) = make_float4(-d.x, -d.y, -d.z, -d.w);
          }
        }
        if (C::kEarly && !kPrepLoads && !kHasDk) mbar_arrive_warp(&sm.row_empty[s]);   // LSE has been read out of the stage
        if (!kHasDk) mbar_arrive_warp(&sm.lse_ready[C::kEarly ? ls : s]);
        if (++ls == C::kLseSlots) ls = 0;
        if (kFp8v && kHasDk && kSl == 2) {
          tc_fence_after_sync();
          if (elect_one()) sf_copy_tiles<kCv, true>(tmem + kColSFdO + 4 * kCv * slot, st.sf_dO);
        }
      }
      if (kHasDk) {
        // -LSE log2(e) and -D of this sub-tile are in place.  (The phase before has completed: its team released the
        // score tile of sub-tile u - 2 before this warp went on to u - 1.)
        mbar_arrive_warp(&sm.s_full[u % kTeams]);
        if (u > 0) {
          // the team of the previous sub-tile has pulled dP into registers
          ok = __all_sync(0xffffffffu, mbar_wait(kApart ? &sm.dp_free[(u - 1) % kTeams] : &sm.s_free[(u - 1) % kTeams], ((u - 1) / kTeams) & 1, abort_flag));
          if (!ok) break;
        }
        tc_fence_after_sync();
        if (elect_one()) {
          if (kFp8v && kSl == 1 && sub_r == 0) sf_copy_tiles<kCv, true>(tmem + kColSFdO, st.sf_dO);
          const uint64_t desc_dO = make_desc_sw128(smem_u32(st.dO[0])) + sub_r * (kSub * 128 / 16);
          issue_ss<kFp8v, kCv, kSub, kTile * 128 / 16, kRowTok * 128 / 16, true>(
              tmem + kColdP, desc_v, desc_dO, nk_v, tmem + kColSFV, tmem + kColSFdO + 4 * kCv * slot + 2 * half);
          mma_commit(kApart ? &sm.dp_full[u % kTeams] : &sm.s_full[u % kTeams]);
          if (C::kEarly) mma_commit(&sm.row_empty[s]);
        }
      }
    }
    if (!ok && kHasDk) {
      int dummy = 0;
      if (elect_one()) mma_commit(&sm.drain[1]);
      mbar_wait(&sm.drain[1], 0, &dummy);
    }
  } else if (warp == 3) {
    // ------------------------------------------------------------------ dV / dK issuer
    if (elect_one()) {
      bool ok = true;
      int rs_done = 0;                                // row stage whose queries go through the softmax next
      for (int u = 0; u < n_sub && ok; ++u) {
        const int buf = kOpBufs == 2 ? (u & 1) : 0, ci = u / kSubPerCol, s = ci % kColStages, slot = kSl == 2 ? (ci & 1) : 0, sub_c = u % kSubPerCol;
        KvColStage<C>& st = sm.cst[s];
        const uint64_t desc_dOc = make_desc_sw128(smem_u32(st.dOc)), desc_qc = make_desc_sw128(smem_u32(st.qc));
        if (sub_c == 0) {
          ok = mbar_wait(&sm.col_full[s], (ci / kColStages) & 1, abort_flag);
          if (!ok) break;
          tc_fence_after_sync();
          if (kFp8 && !kTight) {
            if (kHasDv) sf_copy_tiles<kRv, true>(tmem + kColSFdOc + 4 * kRv * slot, st.sf_dOc);
            if (kHasDk) sf_copy_tiles<kRq, true>(tmem + kColSFQc + 4 * kRq * slot, st.sf_qc);
          }
        }
        // 64 queries = 2 (codes) or 4 (BF16) steps of 32 bytes; the B operands are taken 128 rows at a time
        if (kHasDv) {
          ok = kSplit ? mbar_wait(&sm.p_full, u & 1, abort_flag) : mbar_wait(&sm.op_full[buf], (u >> 1) & 1, abort_flag);
          if (!ok) break;
          tc_fence_after_sync();
          if (kFp8) sf_copy(tmem + kColSFP + 4 * buf, make_desc_sf(smem_u32(sm.sf_p[buf])));
          if (kTight && kFp8) sf_copy(tmem + kColSFdOc, make_desc_sf(smem_u32(st.sf_dOc)));
          issue_ts<kFp8, kEB, kRv, true>(tmem + kColdV, tmem + kColP + kOpCols * buf, desc_dOc, p.dv, sub_c, tmem + kColSFP + 4 * buf,
                                         tmem + kColSFdOc + 4 * kRv * slot, u > 0);
          if (kSplit) mma_commit(&sm.p_free[(u + 1) & 1]);      // P^ and its scale bytes may be rewritten (by the other team)
        }
        if (kHasDk) {
          if (kSplit || !kHasDv) {
            ok = mbar_wait(&sm.op_full[buf], (kOpBufs == 2 ? u >> 1 : u) & 1, abort_flag);
            if (!ok) break;
            tc_fence_after_sync();
          }
          if (kFp8) sf_copy(tmem + kColSFdS + 4 * buf, make_desc_sf(smem_u32(sm.sf_ds[buf])));
          if (kTight && kFp8) {
            // one pair of scale columns for both gradient products and both row tiles of Q^c, used one after the other
#pragma unroll
            for (int r = 0; r < 2; ++r) {
              sf_copy(tmem + kColSFQc, make_desc_sf(smem_u32(st.sf_qc + 512 * r)));
              issue_ts<true, 1, 1, true>(tmem + kColdK + 128 * r, tmem + kColdS, desc_qc + r * (128 * 128 / 16),
                                         r == 0 ? 128 : dk_cols - 128, sub_c, tmem + kColSFdS, tmem + kColSFQc, u > 0);
            }
          } else {
            issue_ts<kFp8, kEB, kRq, true>(tmem + kColdK, tmem + kColdS + kOpCols * buf, desc_qc, dk_cols, sub_c,
                                           tmem + kColSFdS + 4 * buf, tmem + kColSFQc + 4 * kRq * slot, u > 0);
          }
        }
        // all queries of a row stage have been through the softmax: the stage (score operands, LSE, D) is no longer read
        if (!C::kEarly && u % kSubPerRow == kSubPerRow - 1) {
          mbar_arrive(&sm.row_empty[rs_done]);
          if (++rs_done == kRowStages) rs_done = 0;
        }
        // operands and scale bytes of this buffer may be overwritten once these MMAs have run; the
        // col stage may be refilled after its last sub-tile
        mma_commit(&sm.op_free[kOpBufs == 2 ? buf : ((u + 1) & 1)]);   // indexed by the team that writes next
        if (sub_c == kSubPerCol - 1) mma_commit(&sm.col_empty[s]);
        if (u == n_sub - 1) mma_commit(&sm.done);
      }
      if (!ok) {
        int dummy = 0;
        mma_commit(&sm.drain[2]);
        mbar_wait(&sm.drain[2], 0, &dummy);
      }
    }
  } else if (warp >= 4) {
    // ------------------------------------------------------------------ softmax
    const int team = (warp - 4) >> 3;
    const int grp = ((warp - 4) >> 2) & 1;
    const int quad = warp & 3;
    const int row = quad * 32 + lane;                 // key inside the tile == TMEM lane
    const uint32_t lane_addr = static_cast<uint32_t>(quad * 32) << 16;
    bool ok = true;
    int it = it0 + (kShared ? part % tiles_per_head : 0);             // query tile of the current sub-tile (kTeams == 2: one tile per iteration)
    static_assert(kTeams == 2, "a team advances by one query tile per iteration");
    // running (stage, phase) of the row ring: the team's first sub-tile is in row stage team / kSubPerRow and
    // it advances by kTeams / kSubPerRow stages per iteration
    int s = (team / kSubPerRow) % kRowStages;
    uint32_t s_phase = ((team / kSubPerRow) / kRowStages) & 1;
    int ls = team;                                    // kEarly: running (slot, phase) of the LSE / D ring
    uint32_t ls_phase = 0;
    for (int u = team; u < n_sub; u += kTeams) {
      const int half = u & 1, buf = kOpBufs == 2 ? (u & 1) : 0;
      if (u != team) {
#pragma unroll
        for (int a = 0; a < kTeams / kSubPerRow; ++a)
          if (++s == kRowStages) { s = 0; s_phase ^= 1u; }
        if ((ls += kTeams) >= C::kLseSlots) { ls -= C::kLseSlots; ls_phase ^= 1u; }
      }
      ok = mbar_wait(&sm.s_full[team], (u / kTeams) & 1, abort_flag);
      if (!ok) break;
      tc_fence_after_sync();
      uint32_t sr[32], dpr[32];                       // S then P; dP then dS (in place)
      tmem_ld32(tmem + kColS + 64 * (u % kSBufs) + lane_addr + 32 * grp, sr);
      if (kHasDk && !kApart) tmem_ld32(tmem + kColdP + lane_addr + 32 * grp, dpr);
      tmem_wait_ld();
      tc_fence_before_sync();
      mbar_arrive(&sm.s_free[team]);
      if (!kHasDk) {                                  // (otherwise s_full stands for LSE and D as well)
        ok = C::kEarly ? mbar_wait(&sm.lse_ready[ls], ls_phase, abort_flag) : mbar_wait(&sm.lse_ready[s], s_phase, abort_flag);
        if (!ok) break;
      }
      const int col0 = half * kSub + 32 * grp;        // query row (inside the tile) of this thread's first column
      const int st0 = (u % kSubPerRow) * kSub + 32 * grp;   // the same inside the row stage
      const KvRowStage<C>& st = sm.rst[s];
      const float* s_lse = C::kEarly ? &sm.lse_ring[ls][32 * grp] : &st.neg_lse2[st0];
      const float* s_delta = C::kEarly ? &sm.delta_ring[ls][32 * grp] : &st.delta[st0];
      uint32_t words[8 * kEB];
      // P = 2^(S scale log2e - LSE log2e), two elements per instruction (fma / mul .f32x2) wherever the arithmetic
      // allows: the loop is bound by instruction issue, not by a pipe
      float amax_p = 0.f, max_s = 0.f;
      const float2 sc2 = make_float2(p.scale_log2, p.scale_log2);
      // dS = P (dP - D) of a pair of queries (dv2 holds -D)
      auto gradient = [&](int c, const float2 p2, const float2 dv2) {
        const float2 t2 = __fadd2_rn(make_float2(__uint_as_float(dpr[c]), __uint_as_float(dpr[c + 1])), dv2);
        const float2 ds2 = __fmul2_rn(p2, t2);
        dpr[c] = __float_as_uint(ds2.x);
        dpr[c + 1] = __float_as_uint(ds2.y);
        max_s = fmaxf(max_s, fmaxf(fabsf(ds2.x), fabsf(ds2.y)));
      };
      auto body = [&](auto diag_tag) {
        constexpr bool kDiag = decltype(diag_tag)::value;
#pragma unroll
        for (int c4 = 0; c4 < 32; c4 += 4) {
          const float4 l4 = lds_f4(&s_lse[c4]);
          float4 d4 = make_float4(0.f, 0.f, 0.f, 0.f);
          if (kHasDk && !kApart) d4 = lds_f4(&s_delta[c4]);
#pragma unroll
          for (int e = 0; e < 4; e += 2) {
            const int c = c4 + e;
            const float2 lv2 = e == 0 ? make_float2(l4.x, l4.y) : make_float2(l4.z, l4.w);
            float2 x2 = __ffma2_rn(make_float2(__uint_as_float(sr[c]), __uint_as_float(sr[c + 1])), sc2, lv2);
            if (kDiag) {                                      // key after the query
              if (row > col0 + c) x2.x = -INFINITY;
              if (row > col0 + c + 1) x2.y = -INFINITY;
            }
            const float2 p2 = make_float2(ex2_approx(x2.x), ex2_approx(x2.y));
            sr[c] = __float_as_uint(p2.x);
            sr[c + 1] = __float_as_uint(p2.y);
            if (kFp8) amax_p = fmaxf(amax_p, fmaxf(p2.x, p2.y));
            if (kHasDk && !kApart) gradient(c, p2, e == 0 ? make_float2(d4.x, d4.y) : make_float2(d4.z, d4.w));
          }
        }
      };
      if (p.causal && it + p.q0t == jt) body(std::true_type{}); else body(std::false_type{});
      if (!kApart && __builtin_expect(!p.causal && row > p.kv_lim && jt == p.Nk / kTile - 1, 0)) {
        // a padded key of a ragged sequence (no causal mask): its probabilities and score gradients are zero
#pragma unroll
        for (int c = 0; c < 32; ++c) { sr[c] = 0u; dpr[c] = 0u; }
        amax_p = 0.f;
        max_s = 0.f;
      }
      if (kApart) {
        ok = mbar_wait(&sm.dp_full[team], (u / kTeams) & 1, abort_flag);
        if (!ok) break;
        tc_fence_after_sync();
        tmem_ld32(tmem + kColdP + lane_addr + 32 * grp, dpr);     // in flight while P is cast
      }
      if (u >= kOpBufs && !kSplit) {
        // the MMAs of the sub-tile that last used this buffer have consumed its operands and scale bytes
        ok = mbar_wait(&sm.op_free[team], ((u - kOpBufs) >> 1) & 1, abort_flag);
        if (!ok) break;
        tc_fence_after_sync();
      }
      if (kHasDv) {
        uint32_t byte = 0;
        if (kFp8) {
          float inv;
          block_scale_finite(amax_p, byte, inv);
          const float2 inv2 = make_float2(inv, inv);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float2 a = __fmul2_rn(make_float2(__uint_as_float(sr[4 * i]), __uint_as_float(sr[4 * i + 1])), inv2);
            const float2 bq = __fmul2_rn(make_float2(__uint_as_float(sr[4 * i + 2]), __uint_as_float(sr[4 * i + 3])), inv2);
            words[i] = cvt_e4m3x4(a.x, a.y, bq.x, bq.y);
          }
        } else {
#pragma unroll
          for (int i = 0; i < 8 * kEB; ++i)
            words[i] = cvt_bf16x2(__uint_as_float(sr[(2 * i) & 31]), __uint_as_float(sr[(2 * i + 1) & 31]));
        }
        if (kSplit && u >= 1) {
          // the dV MMAs of the sub-tile before have consumed P^ and its scale bytes
          ok = mbar_wait(&sm.p_free[team], ((u - 1) >> 1) & 1, abort_flag);
          if (!ok) break;
          tc_fence_after_sync();
        }
#pragma unroll
        for (int i = 0; i < kEB; ++i) tmem_st8(tmem + kColP + kOpCols * buf + lane_addr + 8 * kEB * grp + 8 * i, words + 8 * i);
        if (kFp8) sts_u8(&sm.sf_p[buf][(row & 31) * 16 + (row >> 5) * 4 + grp], byte);
        if (kSplit) {
          tmem_wait_st();
          fence_proxy_async_smem();
          tc_fence_before_sync();
          mbar_arrive(&sm.p_full);
        }
      }
      if (kApart) {
        tmem_wait_ld();
        tc_fence_before_sync();
        mbar_arrive(&sm.dp_free[team]);
#pragma unroll
        for (int c4 = 0; c4 < 32; c4 += 4) {
          const float4 d4 = lds_f4(&s_delta[c4]);
#pragma unroll
          for (int e = 0; e < 4; e += 2) {
            const int c = c4 + e;
            gradient(c, make_float2(__uint_as_float(sr[c]), __uint_as_float(sr[c + 1])), e == 0 ? make_float2(d4.x, d4.y) : make_float2(d4.z, d4.w));
          }
        }
      }
      if (kHasDk) {
        uint32_t byte = 0;
        if (kFp8) {
          float inv;
          block_scale_finite(max_s, byte, inv);
          const float2 inv2 = make_float2(inv, inv);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float2 a = __fmul2_rn(make_float2(__uint_as_float(dpr[4 * i]), __uint_as_float(dpr[4 * i + 1])), inv2);
            const float2 bq = __fmul2_rn(make_float2(__uint_as_float(dpr[4 * i + 2]), __uint_as_float(dpr[4 * i + 3])), inv2);
            words[i] = cvt_e4m3x4(a.x, a.y, bq.x, bq.y);
          }
        } else {
#pragma unroll
          for (int i = 0; i < 8 * kEB; ++i)
            words[i] = cvt_bf16x2(__uint_as_float(dpr[(2 * i) & 31]), __uint_as_float(dpr[(2 * i + 1) & 31]));
        }
        if (kSplit && u >= 1) {
          // the dK MMAs of the sub-tile before have consumed dS^ and its scale bytes
          ok = mbar_wait(&sm.op_free[team], ((u - 1) >> 1) & 1, abort_flag);
          if (!ok) break;
          tc_fence_after_sync();
        }
#pragma unroll
        for (int i = 0; i < kEB; ++i) tmem_st8(tmem + kColdS + kOpCols * buf + lane_addr + 8 * kEB * grp + 8 * i, words + 8 * i);
        if (kFp8) sts_u8(&sm.sf_ds[buf][(row & 31) * 16 + (row >> 5) * 4 + grp], byte);
      }
      tmem_wait_st();
      fence_proxy_async_smem();
      tc_fence_before_sync();
      mbar_arrive(&sm.op_full[buf]);
      it += split;                                    // next tile of this CTA, of this head or of one that follows
      while (it >= tiles_n) it -= tiles_per_head;
    }
    // The epilogue is done by team 0 (group 0 stores dV, group 1 stores dK).
    if (team != 0) ok = false;
    if (grp == 0 ? !kHasDv : !kHasDk) ok = false;
    if (ok && n_sub > 0) ok = mbar_wait(&sm.done, 0, abort_flag);
    if (kShared) stores = ok;
    else if (ok) {
      tc_fence_after_sync();
      const size_t grow = static_cast<size_t>(slab) * p.Nk + jt * kTile + row;
      const uint32_t col = grp == 0 ? kColdV : kColdK;
      const int width = grp == 0 ? p.dv : p.dqk;
      const int first = grp == 0 ? 0 : dk_col0, count = grp == 0 ? p.dv : dk_cols;   // columns this pass holds
      const float mul = grp == 0 ? 1.f : p.scale;
      __nv_bfloat16* out_row = (grp == 0 ? p.dv_out : p.dk) + grow * width + first;
      for (int c0 = 0; c0 < count; c0 += 32) {
        uint32_t r[32];
        tmem_ld32(tmem + col + lane_addr + c0, r);
        tmem_wait_ld();
        uint32_t packed[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          __nv_bfloat162 v2 = __floats2bfloat162_rn(__uint_as_float(r[2 * c]) * mul, __uint_as_float(r[2 * c + 1]) * mul);
          packed[c] = !kApart || row < real_rows ? *reinterpret_cast<uint32_t*>(&v2) : 0u;
        }
        // (16 bytes at a time: dK / dV of 8 x 12 heads x 1024 x 64 65.5 us, now 61.5; 16 heads x 8192 at (192,128) 489, now 469)
        store_32b(out_row + c0, packed, kSectors && p.sectors != 0);
        store_32b(out_row + c0 + 16, packed + 8, kSectors && p.sectors != 0);
      }
    }
  }
  if constexpr (kShared) {
    const int ep_grp = ((warp - 4) >> 2) & 1, ep_row = (warp & 3) * 32 + lane;
    const uint32_t ep_col = tmem + (ep_grp == 0 ? kColdV : kColdK) + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    const int first = ep_grp == 0 ? 0 : dk_col0, count = ep_grp == 0 ? p.dv : dk_cols;   // columns this pass holds
    const int slice = count / split;                    // columns this CTA stores (a multiple of 16)
    // A cluster adds its partial sums column slice by column slice: each CTA sends the other CTAs their slices of its
    // accumulators (FP32, into their operand stages, no longer in use), then adds the slices it got in the order of the
    // ranks, so that the sum does not depend on timing.
    float* const inbox = reinterpret_cast<float*>(smem_raw);
    const int in_stride = ((kHasDv ? p.dv : 0) + (kHasDk ? dk_cols : 0)) / split * kTile;     // floats per sender
    const int in_grp = (ep_grp == 1 && kHasDv ? p.dv / split : 0) * kTile;
    __syncwarp();
    cluster_sync();                                   // every CTA of the cluster has finished its main loop
    if (stores && n_sub > 0) {
      tc_fence_after_sync();
      for (int to = 0; to < split; ++to) {
        if (to == part) continue;
        const uint32_t dst = cluster_map(smem_u32(inbox + (part < to ? part : part - 1) * in_stride + in_grp + ep_row), to);
        for (int c0 = 0; c0 < slice; c0 += 16) {
          uint32_t r[16];
          tmem_ld16(ep_col + to * slice + c0, r);
          tmem_wait_ld();
#pragma unroll
          for (int c = 0; c < 16; ++c) st_cluster_u32(dst + (c0 + c) * kTile * 4, r[c]);
        }
      }
    }
    __syncwarp();
    cluster_sync();
    if (stores) {
      tc_fence_after_sync();
      const size_t grow = static_cast<size_t>(slab) * p.Nk + jt * kTile + ep_row;
      const float mul = ep_grp == 0 ? 1.f : p.scale;
      __nv_bfloat16* out_row = (ep_grp == 0 ? p.dv_out : p.dk) + grow * (ep_grp == 0 ? p.dv : p.dqk) + first + part * slice;
      for (int c0 = 0; c0 < slice; c0 += 16) {
        uint32_t r[16];
        if (n_sub > 0) {
          tmem_ld16(ep_col + part * slice + c0, r);
          tmem_wait_ld();
        }
        float sum[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) sum[c] = 0.f;
        for (int from = 0; from < split && from < n_list; ++from) {
          const float* in = inbox + (from < part ? from : from - 1) * in_stride + in_grp + ep_row + c0 * kTile;
#pragma unroll
          for (int c = 0; c < 16; ++c) sum[c] += from == part ? __uint_as_float(r[c]) : lds_f32(in + c * kTile);
        }
        uint32_t packed[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const __nv_bfloat162 v2 = __floats2bfloat162_rn(sum[2 * c] * mul, sum[2 * c + 1] * mul);
          packed[c] = !kApart || ep_row < real_rows ? *reinterpret_cast<const uint32_t*>(&v2) : 0u;
        }
        store_32b(out_row + c0, packed, p.sectors != 0);
      }
    }
  }
  __syncwarp();
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, kTmemCols);
  if (tid == 0 && sm.abort_flag) atomicExch(p.status, static_cast<int>(ATTN_ERR_TIMEOUT));
  // This grid may have started while the pass ahead of it was draining.  One CTA, the last in launch
  // order, stays until that grid has completed, so that the completion of this grid implies the
  // completion of both for whatever follows in the stream.
  if (p.tail_wait && tid == 0 && last_cta()) griddep_wait();
}

// CTAs per key tile.  One CTA per key tile is the least work; but the first key tile's CTA walks G * N / 128 query tiles,
// and with few heads or short sequences it alone takes longer than the GPU takes for everything else.  Then a cluster of two,
// four or eight CTAs shares the list, at the cost of more set-ups and of an exchange of the accumulators.  The gradient call is
// estimated (us) from what calls that fit on the GPU at once were measured to take: a CTA of this kernel 6 and so much per
// query tile as the first table says, and 1 per 40 columns of accumulators that it sends where CTAs share, the last pass of
// several 2 later; an item of the dQ kernel 3 and so much per key tile as the second table says, the first of a CTA 3 later.
//   All CTAs of both kernels fit at once: the call takes as long as the longest of them.
//   This kernel's do: dQ items fill the SMs it leaves, and what they do not get done waits for its CTAs to end.
//   They do not: the sum of the work, or a dQ item behind the rounds of this kernel.  In the last two, sharing costs 3 % per
//   doubling, since a cluster waits for as many free SMs; clusters of eight leave a tenth of the SMs out.
// More CTAs only for 5 % and 0.5 us or more.  1680 random problems of up to 1.3 ms (all head dims, both modes, chunks of
// sequences) take 1.004 times what the best number for each takes, 1.003 on the 420 of them that the choice of the costs did not
// see; always one CTA 1.25, the rule before this one 1.009.  With one, two, four, eight: 8 heads on 1, 768 tokens, BF16, 93.0,
// 54.1, 33.3, 23.6 us; 2 x 4 on 1 x 2560 at 64, 113.6, 62.9, 45.6.  8 on 2 x 128 at (192,128), where the exchange takes more
// than sharing saves, 13.3, 15.0, 15.5.
// The dQ kernel counts whether it follows or not: the same sums in the same order with and without it, so that
// attn_fp8_bwd and attn_fp8_bwd_dkdv give the same bits.
int split_of(const AttnShape& s, int sms, int passes) {
  const double tiles = s.N / kTile, keys = s.Nk / kTile, G = s.Hq / s.Hkv;
  // (query tile, key tile) pairs of a head: the first key tiles are seen by all query tiles, the last ones by fewer and fewer
  const double per_head = s.causal ? tiles * (keys - tiles) + tiles * (tiles + 1) / 2 : tiles * keys;
  const double pairs = per_head * s.Hq * s.B;
  const double items = tiles * s.Hq * s.B * (s.eb == 2 && s.dqk > 192 ? 2 : 1);             // (dQ columns in two items there)
  // FP8 and BF16; qk head dim up to 64, 128, 192 and 256 (there for each pass)
  static const double kPerQuery[2][4] = {{1.35, 1.42, 1.6, 1.55}, {1.55, 1.95, 3.0, 3.5}};
  static const double kPerKey[2][4] = {{0.9, 0.9, 1.1, 1.5}, {1.0, 1.0, 1.8, 2.6}};
  const int mode = s.eb - 1, dims = (s.dqk - 1) / 64;
  const double t_pair = kPerQuery[mode][dims], t_dq = kPerKey[mode][dims], start = 3;
  const double item = 3 + t_dq * per_head / tiles, last_dq = start + 3 + t_dq * keys;       // an average item, and the longest
  const double columns = passes > 1 ? 256 : s.dqk + s.dv;
  auto estimate = [&](int split, double full) {
    const double cta = 6 + columns * (split - 1) / split / 40;
    const double longest = t_pair * std::ceil(G * tiles / split) + cta + (passes > 1 ? 2 : 0);
    const double ctas = s.B * s.Hkv * keys * split * passes, work = pairs * passes * t_pair + ctas * cta;
    const double alone = std::max(longest, last_dq), all = (work + items * item) / sms + start;
    const double room = split == 8 ? 0.9 * sms : sms;
    if (ctas + items <= room) return alone;
    if (ctas >= room) return full * std::max(std::max(longest, all), work / room + last_dq);
    if (items * item <= (room - ctas) * std::max(longest - start, 0.0)) return alone;
    return full * std::max(std::max(alone, all), work / ctas + start + item);
  };
  int best = 1;
  double least = estimate(1, 1.0), full = 1.03;
  // (slices of the columns of dK and dV are multiples of 16)
  for (int split = 2; split <= (s.dqk % 128 == 0 && s.dv % 128 == 0 ? 8 : 4); split *= 2, full += 0.03) {
    const double t = estimate(split, full);
    if (t < 0.95 * least && least - t > 0.5) { best = split; least = t; }
  }
  return best;
}

// `behind`: the launch follows another key-major pass of the same call, which writes another output
// (dV or dK, or another column tile of dK) from the same inputs.  With few KV heads a pass has fewer
// CTAs than the GPU has SMs, or a long tail behind its heaviest CTAs; programmatic stream serialisation
// lets this pass's CTAs take the SMs the pass ahead leaves idle (every key-major CTA executes
// griddepcontrol.launch_dependents once set up).
template <class C, bool kShared>
attn_status_t launch_kvmajor_s(const AttnShape& s, attn_qtensor_t q, attn_qtensor_t k, attn_qtensor_t v, attn_qtensor_t dO,
                               const float* lse, const float* delta, void* dk, void* dv, int* status,
                               cudaStream_t stream, bool behind, bool clear_tickets, int split) {
  static_assert(sizeof(KvSmem<C>) + 1024 <= kSmemLimit, "shared memory exceeded");
  // seven eighths of the accumulators (a cluster of eight) fit in the operand stages
  static_assert(((C::kHasDv ? 128 * C::kRv : 0) + (C::kHasDk ? C::kQcRows : 0)) * kTile * 7 / 2 <=
                    sizeof(KvSmem<C>::k) + sizeof(KvSmem<C>::rst) + sizeof(KvSmem<C>::cst), "inbox exceeds the operand stages");
  CUtensorMap tm_k, tm_v, tm_q, tm_dO, tm_qc, tm_dOc;
  attn_status_t st;
  const uint64_t eb = C::kEB, ebv = C::kEBv;
  const uint64_t q_rows = static_cast<uint64_t>(s.B) * s.Hq * s.N, kv_rows = static_cast<uint64_t>(s.B) * s.Hkv * s.Nk;
  if ((st = encode_tmap_u8_sw128(&tm_k, k.row_codes, s.dqk * eb, kv_rows, kTile)) != ATTN_OK) return st;
  if ((st = encode_tmap_u8_sw128(&tm_v, v.row_codes, s.dv * ebv, kv_rows, kTile)) != ATTN_OK) return st;
  if ((st = encode_tmap_u8_sw128(&tm_q, q.row_codes, s.dqk * eb, q_rows, C::kRowTok)) != ATTN_OK) return st;
  if ((st = encode_tmap_u8_sw128(&tm_dO, dO.row_codes, s.dv * ebv, q_rows, C::kRowTok)) != ATTN_OK) return st;
  const int qc_rows = C::kDkTile >= 0 ? (s.dqk - 128 * C::kDkTile < 128 ? s.dqk - 128 * C::kDkTile : 128) : s.dqk;
  if ((st = encode_tmap_u8_sw128(&tm_qc, q.col_codes, s.N * eb, static_cast<uint64_t>(s.B) * s.Hq * s.dqk, qc_rows)) != ATTN_OK) return st;
  if ((st = encode_tmap_u8_sw128(&tm_dOc, dO.col_codes, s.N * eb, static_cast<uint64_t>(s.B) * s.Hq * s.dv, s.dv)) != ATTN_OK) return st;
  KvParams p;
  p.k_sf = k.row_scales; p.v_sf = v.row_scales; p.q_sf = q.row_scales; p.dO_sf = dO.row_scales;
  p.qc_sf = q.col_scales; p.dOc_sf = dO.col_scales;
  p.lse = lse; p.delta = delta;
  p.dk = static_cast<__nv_bfloat16*>(dk); p.dv_out = static_cast<__nv_bfloat16*>(dv); p.sectors = starts_sector(dk) && starts_sector(dv); p.status = status;
  p.N = s.N; p.Nk = s.Nk; p.q0t = s.q0t; p.kv_lim = s.kv_lim; p.Hq = s.Hq; p.Hkv = s.Hkv; p.dqk = s.dqk; p.dv = s.dv; p.causal = s.causal;
  p.scale = s.scale; p.scale_log2 = s.scale * kLog2e;
  p.tail_wait = behind ? 1 : 0;
  p.tickets = clear_tickets ? ticket_counter(status) : nullptr;
  const size_t smem = sizeof(KvSmem<C>) + 1024;
  int sms = 0;
  if ((st = allow_smem<kvmajor_kernel<C, kShared>>(smem, "bwd kv-major", &sms)) != ATTN_OK) return st;
  p.split = split;
  // bytes of Q and dO per (sequence, KV head): the copies this pass reads, of the heads of its group
  const WorkOrder order = work_order(s.B * s.Hkv, 1, s.Nk / kTile,
                                     static_cast<size_t>(s.Hq / s.Hkv) * s.N * (s.dqk * eb * (C::kHasDk ? 2 : 1) +
                                                                                s.dv * ((C::kHasDk ? ebv : 0) + (C::kHasDv ? eb : 0))), s.causal, false, sms);
  p.slabs = order.heads; p.group = order.group;
  const dim3 grid = order.grid(split);
  // The first pass overlaps the kernel ahead like every other kernel only where its CTAs and those of the query-major
  // kernel fit on the GPU together (one head of 256 tokens: step 28 -> 23 us).  On larger problems its CTAs would settle
  // on whichever SMs the kernel ahead leaves first, and the kernels behind fill in worse: head dim 256, 8/2 heads, step
  // 1046 -> 1113 us; 2 x 16/4 heads of 1000 tokens 119 -> 127 us; 2 x 16/4 heads of 4096, steps in a row, 603 -> 611 us.
  const long long ctas = static_cast<long long>(s.B) * (s.Hkv * split * (s.Nk / kTile) + s.Hq * (s.N / kTile));
  const cudaError_t e = launch_kernel(kvmajor_kernel<C, kShared>, grid, kThreads, smem, stream, split, behind || ctas <= sms, p,
                                      tm_k, tm_v, tm_q, tm_dO, tm_qc, tm_dOc);
  if (e != cudaSuccess) return fail(ATTN_ERR_CUDA, "bwd kv-major: launch: %s", cudaGetErrorString(e));
  return ATTN_OK;
}

template <class C>
attn_status_t launch_kvmajor_t(const AttnShape& s, attn_qtensor_t q, attn_qtensor_t k, attn_qtensor_t v, attn_qtensor_t dO,
                               const float* lse, const float* delta, void* dk, void* dv, int* status, cudaStream_t stream,
                               int split, bool behind = false, bool clear_tickets = false) {
  if (split > 1)
    return launch_kvmajor_s<C, true>(s, q, k, v, dO, lse, delta, dk, dv, status, stream, behind, clear_tickets, split);
  return launch_kvmajor_s<C, false>(s, q, k, v, dO, lse, delta, dk, dv, status, stream, behind, clear_tickets, 1);
}

}  // namespace

attn_status_t launch_bwd_dkdv(const AttnShape& s, attn_qtensor_t q, attn_qtensor_t k, attn_qtensor_t v, attn_qtensor_t dO,
                              const float* lse, const float* delta, void* dk, void* dv, int* status,
                              cudaStream_t stream, bool clear_tickets) {
  const int cq = (s.dqk * s.eb + 127) / 128, cv = (s.dv * s.ebv + 127) / 128;
  int dev = 0, sms = 0;
  const attn_status_t found = current_device(&dev, &sms);
  if (found != ATTN_OK) return found;
  const int passes = cq < 2 * s.eb || cv < 2 * s.eb ? 1 : (s.eb == 1 ? 2 : 3);    // (256,256) takes more than one
  const int split = split_of(s, sms, passes);
  if (s.eb == 1 && s.ebv == 2) {                     // protected dP: BF16 row copies of V and dO
    if (cq == 1 && cv == 1)
      return launch_kvmajor_t<KvCfg<1, 1, 1, kBoth, 2>>(s, q, k, v, dO, lse, delta, dk, dv, status, stream, split, false, clear_tickets);
    if (cq == 1 && cv == 2)
      return launch_kvmajor_t<KvCfg<1, 1, 2, kBoth, 2>>(s, q, k, v, dO, lse, delta, dk, dv, status, stream, split, false, clear_tickets);
    return fail(ATTN_ERR_UNSUPPORTED, "bwd kv-major: protected dP is built for head dims (64,64) and (128,128)");
  }
  if (s.eb == 1 && cq == 1 && cv == 1)
    return launch_kvmajor_t<KvCfg<1, 1, 1, kBoth>>(s, q, k, v, dO, lse, delta, dk, dv, status, stream, split, false, clear_tickets);
  if (s.eb == 2 && cq == 1 && cv == 1)
    return launch_kvmajor_t<KvCfg<2, 1, 1, kBoth>>(s, q, k, v, dO, lse, delta, dk, dv, status, stream, split, false, clear_tickets);
  if (s.eb == 2 && cq == 2 && cv == 2)
    return launch_kvmajor_t<KvCfg<2, 2, 2, kBoth>>(s, q, k, v, dO, lse, delta, dk, dv, status, stream, split, false, clear_tickets);
  // qk head dim above 128: dV and dK do not fit in tensor memory together; one pass each, the
  // heavier dK pass first and the dV pass launched behind it (see launch_kvmajor_t)
  // (at (192,128) both fit when every operand buffer and scale slot is single: KvCfg::kTight)
  if (s.eb == 1 && cq == 2 && cv == 1)
    return launch_kvmajor_t<KvCfg<1, 2, 1, kBoth>>(s, q, k, v, dO, lse, delta, dk, dv, status, stream, split, false, clear_tickets);
  if (s.eb == 1 && cq == 2 && cv == 2) {
    attn_status_t st = launch_kvmajor_t<KvCfg<1, 2, 2, kDkOnly>>(s, q, k, v, dO, lse, delta, dk, dv, status, stream, split, false, clear_tickets);
    if (st != ATTN_OK) return st;
    return launch_kvmajor_t<KvCfg<1, 2, 2, kDvOnly>>(s, q, k, v, dO, lse, delta, dk, dv, status, stream, split, true);
  }
  if (s.eb == 2 && cq == 3 && cv == 2)
    return launch_kvmajor_t<KvCfg<2, 3, 2, kBoth>>(s, q, k, v, dO, lse, delta, dk, dv, status, stream, split, false, clear_tickets);
  if (s.eb == 2 && cq == 4 && cv == 4) {
    attn_status_t st = launch_kvmajor_t<KvCfg<2, 4, 4, kDkOnly, 2, 0>>(s, q, k, v, dO, lse, delta, dk, dv, status, stream, split, false, clear_tickets);
    if (st != ATTN_OK) return st;
    st = launch_kvmajor_t<KvCfg<2, 4, 4, kDkOnly, 2, 1>>(s, q, k, v, dO, lse, delta, dk, dv, status, stream, split, true);
    if (st != ATTN_OK) return st;
    return launch_kvmajor_t<KvCfg<2, 4, 4, kDvOnly>>(s, q, k, v, dO, lse, delta, dk, dv, status, stream, split, true);
  }
  return fail(ATTN_ERR_UNSUPPORTED, "bwd kv-major: no kernel for head dims (%d, %d) at %d bytes per element", s.dqk, s.dv,
              s.eb);
}

}  // namespace attnfp8
