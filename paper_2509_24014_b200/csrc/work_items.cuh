// Work items of the single-CTA attention kernels (attention.cu, attention_lone.cu): an item is one 128-row query tile of
// one (batch, head), and what its walk over the keys reads of the CSR pattern.
#pragma once

#include "internal.h"

namespace sparsed {

constexpr int kTileM = 128;   // query rows of an item: UMMA M, rows of tensor memory
constexpr int kTileN = 64;    // keys per pipeline step
constexpr int kMaxPackedBlocks = 2048;   // key blocks per row the union walk can hold (64- and 32-key blocks)
constexpr int kIdBits = 11;              // of a union entry: the block's id; above them one bit per query block keeping it
static_assert((1 << kIdBits) == kMaxPackedBlocks, "ids of union entries");
template <int kBlock>
constexpr int kMemberWords = kBlock < kTileM ? kMaxPackedBlocks / 32 : 1;   // bitmap words per query block

struct WorkItem {
  int q_tile, bh, head, batch, kv_head, q_row0, groups_here, r0;
  int list_begin, list_len;   // CSR entries of the item's query blocks; dense: key tiles of the sequence
};

// The item's row_ptr entries. Adjacent rows are adjacent in col_idx, so the item's lists are one run of entries.
__device__ __forceinline__ void read_list_bounds(const AttnParams& p, WorkItem& it) {
  it.list_begin = __ldcg(p.row_ptr + it.r0);
  it.list_len = __ldcg(p.row_ptr + it.r0 + it.groups_here) - it.list_begin;
  if (it.list_begin < 0 || it.list_len < 0 || static_cast<int64_t>(it.list_begin) + it.list_len > p.col_capacity) {
    // row_ptr points outside col_idx: not followed; the rows get zeros and the status word says why
    if (atomicCAS(&p.status->code, 0, 3) == 0) p.status->where = 2;
    it.list_begin = 0;
    it.list_len = 0;
  }
}

// with_list: read the item's row_ptr entries too
template <int kGroups, bool kDense>
__device__ __forceinline__ WorkItem describe_item(const AttnParams& p, int item, bool with_list) {
  WorkItem it;
  it.q_tile = item % p.num_q_tiles;
  it.bh = item / p.num_q_tiles;
  it.head = it.bh % p.heads_q;
  it.batch = it.bh / p.heads_q;
  it.kv_head = it.head / p.group;
  it.q_row0 = it.q_tile * kTileM;
  const int qb0 = it.q_tile * kGroups;                                   // first query block of the item
  it.groups_here = kDense ? 1 : min(kGroups, p.num_blocks - qb0);        // the last tile of a head may hold fewer
  it.r0 = it.bh * p.num_blocks + qb0;                                    // CSR row of query block qb0
  it.list_begin = 0;
  it.list_len = (p.seq_len + kTileN - 1) / kTileN;
  if (!kDense && with_list) read_list_bounds(p, it);
  return it;
}

// Packed walks (64- and 32-key blocks), one warp: one bitmap per query block of the item, then their union into `list`,
// ascending, one entry per key block; returns its length. The last tile of an odd union of 32-key blocks is filled up
// with its own last block, which no query block keeps there.
template <int kGroups, int kBlocksPerTile, int kWords>
__device__ __forceinline__ int build_list_union(const AttnParams& p, const WorkItem& it, int lane,
                                                uint32_t (&member)[kGroups][kWords], uint16_t* list) {
  const int words = (p.num_blocks + 31) >> 5;
  for (int i = lane; i < kGroups * kWords; i += 32) (&member[0][0])[i] = 0u;
  // (entries are unsigned: a list may end at 2^31 - 1, and the walk steps up to 287 beyond)
  uint32_t bound[kGroups];   // bound[g] = first CSR entry after query block g's list
#pragma unroll
  for (int g = 0; g < kGroups; ++g)
    bound[g] = static_cast<uint32_t>(__ldcg(p.row_ptr + it.r0 + min(g + 1, it.groups_here)));
  __syncwarp();
  const uint32_t list_end = static_cast<uint32_t>(it.list_begin) + static_cast<uint32_t>(it.list_len);
  for (uint32_t e0 = static_cast<uint32_t>(it.list_begin) + lane; e0 < list_end; e0 += 8 * 32) {
    int id[8];   // eight loads in flight per lane
#pragma unroll
    for (int u = 0; u < 8; ++u) id[u] = e0 + 32 * u < list_end ? __ldcg(p.col_idx + e0 + 32 * u) : -1;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      int g = 0;
#pragma unroll
      for (int j = 0; j + 1 < kGroups; ++j) g += (e0 + 32 * u >= bound[j]) ? 1 : 0;
      if (id[u] >= 0 && id[u] < p.num_blocks) atomicOr(&member[g][id[u] >> 5], 1u << (id[u] & 31));
    }
  }
  __syncwarp();
  int n = 0;
  for (int w = 0; w < words; ++w) {   // lane = bit of the word
    uint32_t mask = 0u;
#pragma unroll
    for (int g = 0; g < kGroups; ++g) mask |= ((member[g][w] >> lane) & 1u) << g;
    const uint32_t any = __ballot_sync(0xffffffffu, mask != 0u);
    if (mask != 0u)
      list[n + __popc(any & ((1u << lane) - 1u))] = static_cast<uint16_t>((w * 32 + lane) | (mask << kIdBits));
    n += __popc(any);
  }
  __syncwarp();
  if (kBlocksPerTile > 1 && (n & 1) != 0 && lane == 0) list[n] = list[n - 1] & ((1u << kIdBits) - 1u);
  return n;
}

}  // namespace sparsed
