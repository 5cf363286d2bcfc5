// The order in which the attention kernels take their work items.
//
// An item is one 128-row tile of one head (of one dQ column tile of a head).  Heaviest tiles first, over all heads and
// sequences, is the best order for the tail of a launch: with the batch slowest, the heaviest causal tiles of the second
// sequence came after the lightest of the first (2 x 16 heads x 4096 tokens: forward 118.7 us for 103.3 us of work per
// SM).  But every item reads all K and V of its KV head (or Q and dO of the group), and with more heads in flight than
// L2 holds the kernels are bound by DRAM: 8 x 12 heads, 6400 queries on 19200 keys, 470 MB of K and V, step 19.9 ms with
// the batch slowest, 23.8 ms with the tile slowest.  So the tile is the slowest index within a GROUP of (sequence, KV head)
// pairs whose operands stay in L2: 19.6 ms there; BF16 head dim 256, 4 x 12 heads x 9984, step 51.7 -> 58.6 -> 49.5 ms.
//
// A CTA with a static list takes the items c, 2n-1-c, 2n+c, ... of n CTAs, which evens out where the weight of the items
// falls steadily.  From group to group it would jump from the lightest to the heaviest tile, and CTAs on either side of the
// jump differ by a whole item: these lists run through every other group backwards (`flip`), so that the weight falls
// and rises in turn and falls in the last group (2 x 16 heads x 15488, head dim 192, forward, four pairs per group:
// 1427 -> 1382 us; batch slowest 1387, tile slowest 1485).
#pragma once
#include <cstddef>
#include <cstdint>

namespace attnfp8 {

// Division of 0 <= n < 2^31 by an invariant 0 < d < 2^31: n * ceil(2^s / d) >> s with s = 31 + ceil(log2 d) (Granlund and
// Montgomery, "Division by invariant integers using multiplication", 1994).  With the compiler's divisions instead the
// kernels that decode an item per CTA or per role took up to 9 % longer (dQ at head dim 256, 231 -> 253 us).
struct InvariantDiv {
  uint32_t m, s;
  static InvariantDiv by(long long d) {
    if (d < 1 || d > 0x7fffffffLL) return InvariantDiv{0, 0};   // more items than a launch may have: refused elsewhere
    uint32_t k = 0;
    while ((1LL << k) < d) ++k;
    return InvariantDiv{static_cast<uint32_t>(((uint64_t{1} << (31 + k)) + d - 1) / d), 31 + k};
  }
  __device__ __forceinline__ int quotient(int n) const {
    return static_cast<int>(static_cast<uint64_t>(static_cast<uint32_t>(n)) * m >> s);
  }
};

struct WorkOrder {
  int heads, group, tiles;     // heads in all (times dQ column tiles), heads of a group, tiles of a head
  int last_group;
  int flip;
  InvariantDiv per_group, per_row, per_last_row, per_slab;

  // item l of a list
  __device__ __forceinline__ void decode(int l, int& tile, int& head) const {
    const int grp = per_group.quotient(l), first = grp * group;
    l -= first * tiles;
    tile = grp < last_group ? per_row.quotient(l) : per_last_row.quotient(l);
    head = first + l - tile * min(group, heads - first);
    if (flip & (last_group - grp)) tile = tiles - 1 - tile;
  }
  // the item of a block of grid(); false: the last group is short, and the block has none
  __device__ __forceinline__ bool at_block(int& tile, int& head) const {
    tile = static_cast<int>(blockIdx.y);
    head = static_cast<int>(blockIdx.z) * group + static_cast<int>(blockIdx.x);
    return head < heads;
  }
  // the (sequence, KV head) pair of a head
  __device__ __forceinline__ int slab_of(int head) const { return per_slab.quotient(head); }

  long long items() const { return static_cast<long long>(heads) * tiles; }
  dim3 grid(int ctas_per_item = 1) const { return dim3(group * ctas_per_item, tiles, last_group + 1); }
};

// `slabs` (sequence, KV head) pairs of `per_slab` heads, `bytes` of operands per pair that its items share.
// A group takes 32 MB of them (16 and 64 MB are 0 to 2 % behind where they differ), and not less than four rounds of items
// on all SMs under the causal mask, where a group ends in a tail of light tiles and the last one is the tail of the launch
// (BF16, 2 x 16 heads x 8192: step 2871 us with four rounds, 2925 with one); without it all items weigh the same and one
// round will do (BF16 head dim 256, 8 heads x 12160: 12240 us with four, 11577 with one, 11500 with the batch slowest).  Not
// for the rounds' sake more than 80 MB, beyond which L2 (126 MB) may not hold it.
inline WorkOrder work_order(int slabs, int per_slab, int tiles, size_t bytes, bool causal, bool flip, int sms) {
  const long long fits = (32LL << 20) / bytes, most = (80LL << 20) / bytes, per = static_cast<long long>(per_slab) * tiles;
  const long long enough = ((causal ? 4 : 1) * static_cast<long long>(sms) + per - 1) / per;
  long long size = enough < most ? enough : most;
  if (size < fits) size = fits;
  if (size < 1) size = 1;
  const int groups = static_cast<int>((slabs + size - 1) / size), group = (slabs + groups - 1) / groups;
  WorkOrder o;
  o.heads = slabs * per_slab; o.group = group * per_slab; o.tiles = tiles;
  o.last_group = (slabs - 1) / group;
  o.flip = flip ? 1 : 0;
  o.per_group = InvariantDiv::by(static_cast<long long>(o.group) * tiles);
  o.per_row = InvariantDiv::by(o.group);
  o.per_last_row = InvariantDiv::by(o.heads - o.last_group * o.group);
  o.per_slab = InvariantDiv::by(per_slab);
  return o;
}

}  // namespace attnfp8
