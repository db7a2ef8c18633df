// Attention for head_dim 128, bf16 in / bf16 out, fp32 softmax, on sm_100a: dense bidirectional attention (Eq. 1 times V;
// the full-attention branch of Algorithm 1) and block-sparse attention over CSR block lists (Eq. 3 / Eq. 4 times V; the
// "Sparse Reusing" branch). Two more kernels do parts of the same work: attention_lone.cu most grids of up to one query
// tile per SM, attention_dense_pair.cu large dense ones and dense ones with row statistics (dense_choice.h).
//
// One CTA owns 128 consecutive query rows of one (batch, head) and streams 64-key tiles through a
// warp-specialised pipeline:
//   warp 4  : TMA producer  - Q once, then a K tile and a V tile per step into a ring of
//                             128B-swizzled shared memory shared by K and V
//   warp 5  : UMMA issuer   - S_j = Q K_j^T into one of two tensor-memory buffers, then
//                             O += P_j V_j with P read from tensor memory (P overwrites the
//                             first half of S_j's columns). S_{j+1} is issued before P_j V_j,
//                             so the tensor pipe works on the next logits while the softmax
//                             warps are busy with the current ones. Each batch of MMAs ends in ONE
//                             commit to the barrier of the ring slot it read: that barrier tells the
//                             softmax warps "S_j is ready" / "P_j V_j has drained" and the producer
//                             "the slot is free" (the issuing thread is the pipeline's bottleneck:
//                             a commit costs it about 150 clocks, a barrier poll about 100).
//   warps 0-3: one thread per query row - single-pass online softmax in fp32 on base-2 logits
//             against a stale running maximum (softmax_pipeline.cuh); finally O is normalised
//             and stored.
// Two CTAs fit on one SM (at most 112 KB of shared memory and 256 tensor-memory columns each).
//
// Where the keys come from:
//   * dense: every 64-key tile of the sequence in order; the last one may be ragged (any seq_len).
//     Optional output: the rows' LSE. (The dense pass that also records the row statistics of the switch
//     step runs on the kernels of attention_dense_pair.cu and, on small grids, attention_lone.cu.)
//   * 128-key blocks: the 128 query rows are one query block; its CSR list is walked as it is,
//     two tiles per block.
//   * 64- and 32-key blocks: the 128 query rows are two / four consecutive query blocks with lists
//     of their own. The CTA walks the UNION of those lists (built in shared memory by the producer warp, one
//     item ahead, from one bitmap per query block) and every warp skips, per 32-column half of a tile, the key
//     blocks its own query block did not keep: no copy out of tensor memory and no exponentials, P = 0. All 128
//     rows of every MMA belong to real queries, and neighbouring query blocks share the K/V tiles they have in
//     common.
#include "internal.h"
#include "softmax_pipeline.cuh"
#include "work_items.cuh"

namespace sparsed {
namespace {

constexpr int kHeadDim = 128;
constexpr int kSoftmaxThreads = 128;
constexpr int kThreads = 192;
constexpr int kTmemCols = 256;
constexpr int kColS = 0;      // two S buffers of 64 fp32 columns; P (bf16 pairs) reuses the first 32
constexpr int kColO = 128;    // O accumulator (fp32, 128 columns)

// Debug builds (-DSPARSED_TIMELINE) record clock64 stamps of one CTA's pipeline roles after the
// workspace status block: 3 regions of 2048 int64 (softmax thread 0, UMMA thread, TMA thread).
#ifdef SPARSED_TIMELINE
#define TL_DECL(region) long long* tl_buf = reinterpret_cast<long long*>(reinterpret_cast<uint8_t*>(p.status) + 1024) + (region) * 2048; int tl_n = 0; const bool tl_on = (blockIdx.x == 1000) && (threadIdx.x == 0 || threadIdx.x == 128 || threadIdx.x == 160);
#define TL(tag) do { if (tl_on && tl_n < 2047) { tl_buf[1 + tl_n++] = (static_cast<long long>(tag) << 48) | (clock64() & 0xFFFFFFFFFFFFll); tl_buf[0] = tl_n; } } while (0)
#else
#define TL_DECL(region)
#define TL(tag)
#endif

// Ring slots: five for 128-key blocks; four when the union walk needs room for its lists.
template <int kBlock>
struct AttnSmem {
  static constexpr bool kPacked = kBlock < kTileM;
  static constexpr int kSlots = kPacked ? 4 : 5;
  static constexpr int kGroups = kTileM / kBlock;                       // query blocks per CTA
  alignas(1024) __nv_bfloat16 q[2][kTileM * 64];           // two 64-wide halves of head_dim
  alignas(1024) __nv_bfloat16 kv[kSlots][2][kTileN * 64];  // each slot: two 64-wide halves of head_dim
  uint64_t q_full, kv_full[kSlots];
  uint64_t done[kSlots];   // the MMAs that read the slot have completed (Q K^T for a K tile, P V for a V tile)
  uint64_t p_full[2];
  uint64_t q_free;         // an output tile has been read out of the Q buffer (which staged it): the next Q may land
  uint64_t o_staged;       // every softmax warp has written its rows of the output tile into the Q buffer
  uint32_t tmem_base;
  int abort_flag;
  // Packed walks: the CTA's items, handed by the producer warp to the other roles through two buffers: the query tile
  // (-1: no more) and the key blocks in the union of its lists ...
  uint64_t item_full[2], item_free[2];
  int item[2], item_entries[2];
  alignas(16) uint32_t control[4];   // (the launch control's answer)
  uint64_t control_full;
  // ... and the union itself, ascending, one entry per key block: its id and, from bit kIdBits on, one bit per query block
  // that keeps it. One per item buffer: the next item's union is built while this one's is walked.
  alignas(16) uint16_t list[2][kPacked ? kMaxPackedBlocks + 2 : 2];
  uint32_t member[kGroups][kMemberWords<kBlock>];  // producer only: bit j of query block g = "g keeps key block j"
};

// kDense: walk every key tile of the sequence (kBlock must be 128 then; no block lists are read).
// kOverlap: begins with wait_for_previous_kernel, so that small grids may be launched overlapped. (Of the dense walk there
// are both kinds: with the wait at its start the compiler arranges the main loop differently, and long launches take
// 1.4 % longer. 128-key blocks take the same either way: 8k 229.6 against 230.5 us, 16k 551.7 against 551.0.)
template <int kBlock, bool kDense, bool kOverlap>
__global__ void __launch_bounds__(kThreads, 2)
attn_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
            const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_o, const AttnParams p) {
  static_assert(!kDense || kBlock == 128, "the dense walk uses the unpacked layout");
  using Smem = AttnSmem<kBlock>;
  constexpr bool kPacked = Smem::kPacked;
  constexpr int kSlots = Smem::kSlots;
  constexpr int kGroups = Smem::kGroups;
  constexpr int kTilesPerBlock = kBlock >= kTileN ? kBlock / kTileN : 1;   // 128-key block: two tiles
  constexpr int kBlocksPerTile = kBlock >= kTileN ? 1 : kTileN / kBlock;   // 32-key blocks: two per tile
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
  if constexpr (kOverlap) wait_for_previous_kernel();
  if ((smem_u32(smem_raw) & 1023u) != 0u) {
    // swizzled tiles need a 1024-byte aligned base; never expected, reported instead of trusted
    if (threadIdx.x == 0 && atomicCAS(&p.status->code, 0, 2) == 0) p.status->where = 1;
    return;
  }

  const int tid = threadIdx.x;
  const int warp = tid >> 5;
  const int lane = tid & 31;

  // ---- work items ----------------------------------------------------------------------
  // An item is one 128-row query tile of one (batch, head). Dense: one CTA per item, and that is all there is to it.
  // Block lists: a CTA runs through several items, and each role of the pipeline runs on into the next one on its
  // own: the producer loads the next Q, list and K/V tiles while the softmax warps are still in the previous item's
  // last tiles and epilogue, so that the start-up chain row_ptr -> col_idx -> first K tile -> first MMA of all but a
  // CTA's first item is hidden. Counters of loads, tiles and Q loads run on across items and all roles compute the same
  // values, so ring slots, S buffers and barrier phases simply continue. Which items those are:
  //   128-key blocks: blockIdx.x, blockIdx.x + gridDim.x, ...; as many CTAs as fit on the device. A selected
  //     pattern's lists are equally long, so that is balanced.
  //   64- and 32-key blocks: unions differ in length by up to 1 : 4, so the grid has one CTA per item and a CTA that
  //     runs takes over CTAs that have not been launched yet (cluster launch control), late in the item before. Block
  //     32, 8 x 32 heads x 4096 tokens, half kept: 1524 us with one item per CTA, 1450 with equal shares, 1439 this way;
  //     block 64, 32 x 65536: 8.64 ms with equal shares, 8.06 this way. (With 128-key blocks it was 1 % slower than equal
  //     shares.)
  using Item = WorkItem;
  const int n_items = p.num_items;
  auto describe = [&](int item, bool with_list) -> Item { return describe_item<kGroups, kDense>(p, item, with_list); };
  // tiles of an item in the unpacked walks (the packed walk counts its union instead)
  auto unpacked_tiles = [&](const Item& it) -> int { return kDense ? it.list_len : it.list_len * kTilesPerBlock; };

  const int first_item = blockIdx.x;
  Item cur = describe(first_item, !kPacked || warp == 4);

  // ---- set-up --------------------------------------------------------------------------
  // The producer warp owns the barriers of its own loads, so it can start them before the CTA-wide
  // set-up (tensor-memory allocation, the other barriers) has finished: the Q tile, the first block
  // ids of the list and, when the list needs no preparation, the first ring-full of K/V tiles.
  int list_ids = 0;     // unpacked walk: lane i holds the block id of list entry 32 * chunk + i
  int loads_issued = 0; // K/V loads of the first item already issued by the producer before the set-up barrier
  // rows [kv_row0, +64) (or two 32-row blocks at kv_row0 / kv_row1) of K (which = 0) or V into `slot`
  auto issue_load = [&](const Item& it, int slot, int which, int kv_row0, int kv_row1) {
    if (elect_one_sync()) {
      const CUtensorMap* tm = which == 0 ? &tm_k : &tm_v;
      if constexpr (kBlocksPerTile == 1) {
        mbar_expect_tx(&sm.kv_full[slot], kTileN * kHeadDim * 2);
        tma_load_4d(sm.kv[slot][0], tm, &sm.kv_full[slot], 0, kv_row0, it.kv_head, it.batch);
        tma_load_4d(sm.kv[slot][1], tm, &sm.kv_full[slot], 64, kv_row0, it.kv_head, it.batch);
      } else {
        // tensor-map boxes are 32 rows here; block b of the tile lands at rows 32 b
        mbar_expect_tx(&sm.kv_full[slot], kTileN * kHeadDim * 2);
        tma_load_4d(sm.kv[slot][0], tm, &sm.kv_full[slot], 0, kv_row0, it.kv_head, it.batch);
        tma_load_4d(sm.kv[slot][1], tm, &sm.kv_full[slot], 64, kv_row0, it.kv_head, it.batch);
        tma_load_4d(sm.kv[slot][0] + kBlock * 64, tm, &sm.kv_full[slot], 0, kv_row1, it.kv_head, it.batch);
        tma_load_4d(sm.kv[slot][1] + kBlock * 64, tm, &sm.kv_full[slot], 64, kv_row1, it.kv_head, it.batch);
      }
    }
    __syncwarp();
  };
  auto issue_q_load = [&](const Item& it) {
    if (elect_one_sync()) {
      mbar_expect_tx(&sm.q_full, kTileM * kHeadDim * 2);   // rows beyond the sequence arrive as zeros
      tma_load_4d(sm.q[0], &tm_q, &sm.q_full, 0, it.q_row0, it.head, it.batch);
      tma_load_4d(sm.q[1], &tm_q, &sm.q_full, 64, it.q_row0, it.head, it.batch);
    }
    __syncwarp();
  };
  // first key row of tile t in the unpacked walks
  auto unpacked_row = [&](int t) -> int {
    if constexpr (kDense) return t * kTileN;
    const int e = t / kTilesPerBlock;
    return __shfl_sync(0xffffffffu, list_ids, e & 31) * kBlock + (t % kTilesPerBlock) * kTileN;
  };
  // packed walks, producer warp: the union of the item's lists into list buffer `buf`; returns its length
  auto build_union = [&](const Item& it, int buf) -> int {
    return build_list_union<kGroups, kBlocksPerTile>(p, it, lane, sm.member, sm.list[buf]);
  };
  // the CTA's next item (-1: none), `entries` key blocks long, to the other roles
  auto publish = [&](int buf, int item, int entries) {
    __syncwarp();
    if (lane == 0) {
      sm.item[buf] = item;
      sm.item_entries[buf] = entries;
      mbar_arrive(&sm.item_full[buf]);
    }
    __syncwarp();
  };
  // ask for the item after the one at hand
  auto request_item = [&]() {
    if (elect_one_sync()) {
      mbar_expect_tx(&sm.control_full, 16);
      launch_control_request(sm.control, &sm.control_full);
    }
    __syncwarp();
  };
  // first key rows of tile t of the union in list buffer `buf`: both 32-key blocks side by side, or one 64-key block
  auto union_rows = [&](int buf, int t) -> int2 {
    constexpr uint32_t ids = (1u << kIdBits) - 1u;
    if constexpr (kBlocksPerTile == 1) {
      return make_int2(static_cast<int>(sm.list[buf][t] & ids) * kBlock, 0);
    } else {
      const uint32_t two = *reinterpret_cast<const uint32_t*>(&sm.list[buf][2 * t]);
      return make_int2(static_cast<int>(two & ids) * kBlock, static_cast<int>((two >> 16) & ids) * kBlock);
    }
  };
  int first_entries = 0;   // packed, producer: entries of the first item's union
  if (warp == 4) {
    if (lane == 0) {
      mbar_init(&sm.q_full, 1);
      for (int s = 0; s < kSlots; ++s) mbar_init(&sm.kv_full[s], 1);
      if constexpr (kPacked) {
        for (int b = 0; b < 2; ++b) {
          mbar_init(&sm.item_full[b], 1);
          mbar_init(&sm.item_free[b], 5);   // four softmax warps and the issuer
        }
        mbar_init(&sm.control_full, 1);
      }
      mbar_fence_init();
    }
    __syncwarp();
    if (elect_one_sync()) {
      tma_prefetch_desc(&tm_q);
      tma_prefetch_desc(&tm_k);
      tma_prefetch_desc(&tm_v);
      if constexpr (!kDense) tma_prefetch_desc(&tm_o);
    }
    __syncwarp();
    if constexpr (kPacked) {
      first_entries = build_union(cur, 0);
      publish(0, first_item, first_entries);
      if (first_entries > 0) issue_q_load(cur);
      const int first = min(2 * ((first_entries + kBlocksPerTile - 1) / kBlocksPerTile), kSlots);
      for (; loads_issued < first; ++loads_issued) {
        const int2 rows = union_rows(0, loads_issued >> 1);
        issue_load(cur, loads_issued, loads_issued & 1, rows.x, rows.y);
      }
    } else if (cur.list_len > 0) {
      issue_q_load(cur);
      if constexpr (!kDense) {
        if (lane < cur.list_len) list_ids = __ldcg(p.col_idx + cur.list_begin + lane);
      }
      const int first = min(2 * unpacked_tiles(cur), kSlots);   // list entries 0..2 at most: within the first chunk
      for (; loads_issued < first; ++loads_issued)
        issue_load(cur, loads_issued, loads_issued & 1, unpacked_row(loads_issued >> 1), 0);
    }
  }
  if (tid == 0) {
    for (int s = 0; s < kSlots; ++s) mbar_init(&sm.done[s], 1);
    for (int s = 0; s < 2; ++s) mbar_init(&sm.p_full[s], kSoftmaxThreads);
    mbar_init(&sm.q_free, 1);
    mbar_init(&sm.o_staged, 4);
    sm.abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 5) {
    tmem_alloc(&sm.tmem_base, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem_base;
  const uint32_t tO = tmem + kColO;
  // 64-key tiles of a union of n key blocks
  auto union_tiles = [&](int n) -> int { return kBlocksPerTile == 1 ? n : (n + kBlocksPerTile - 1) / kBlocksPerTile; };

  // Warps 4 and 5 run their loops with all 32 lanes converged and let one elected lane issue
  // the TMA / UMMA instructions: their operands then stay on the uniform datapath.
  if (warp == 4) {
    // =============================== TMA producer =======================================
    TL_DECL(2)
    bool ok = true;
    int load0 = 0;       // K/V loads issued for earlier items
    int q_tiles_done = 0;  // earlier items that had keys (each loaded a Q tile and staged an output tile)
    [[maybe_unused]] int requests = 0;   // made to the launch control
    for (int nth = 0; ok; ++nth) {       // the CTA's nth item; packed: in item buffer nth & 1
      // The Q buffer doubles as the staging tile of the previous output: the next Q may land once the softmax
      // warps have had that output read out of it (which is after the item's last MMA). The first ring-full of
      // the new item's K/V loads does not depend on its Q (their slots are freed by the previous item's MMAs),
      // so those go out first and the wait for the Q buffer comes after them. Items without keys take no part
      // in this (no Q tile, zeros stored straight from registers), so the barrier completes exactly once per Q
      // tile and this warp is never more than one phase away from it.
      bool q_pending = false;
      int n_entries = kPacked ? first_entries : cur.list_len;
      if constexpr (kPacked) {
        if (nth > 0) {
          ok = mbar_wait(&sm.control_full, (nth - 1) & 1, &sm.abort_flag, p.status, 13);
          // the softmax warps and the issuer have finished with the item that was in this buffer
          if (nth >= 2) ok = ok && mbar_wait(&sm.item_free[nth & 1], ((nth >> 1) - 1) & 1, &sm.abort_flag, p.status, 12);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          const int item = launch_control_answer(sm.control);
          __syncwarp();
          if (item < 0) {
            publish(nth & 1, -1, 0);
            break;
          }
          cur = describe(item, true);
          n_entries = build_union(cur, nth & 1);
          publish(nth & 1, item, n_entries);
          q_pending = n_entries > 0;
        }
      } else if constexpr (!kDense) {
        if (nth > 0) {
          const int item = first_item + nth * static_cast<int>(gridDim.x);
          if (item >= n_items) break;
          cur = describe(item, true);
          n_entries = cur.list_len;
          q_pending = n_entries > 0;
          list_ids = (lane < cur.list_len) ? __ldcg(p.col_idx + cur.list_begin + lane) : 0;
        }
      }
      auto settle_q = [&]() -> bool {
        bool got = true;
        if (q_tiles_done > 0) {
          got = mbar_wait(&sm.q_free, (q_tiles_done - 1) & 1, &sm.abort_flag, p.status, 11);
          got = __all_sync(0xffffffffu, got);
        }
        if (got) issue_q_load(cur);
        q_pending = false;
        return got;
      };
      const int num_tiles = kPacked ? union_tiles(n_entries) : unpacked_tiles(cur);
      const int q_at = min(2 * num_tiles, kSlots);
      // The next item is asked for two tiles before this one's last load: late enough that a CTA with a long union does
      // not hold an item that another could have started (asked for at once, 1.7 items per CTA took 12 % longer than
      // with one item per CTA), early enough for the answer to be there.
      [[maybe_unused]] const int request_at = max(2 * num_tiles - 4, nth == 0 ? loads_issued : 0);
      if constexpr (kPacked) {
        if (request_at >= 2 * num_tiles) {
          request_item();
          ++requests;
        }
      }
      // load i: K (even) or V (odd) of tile i / 2; a slot is reused every kSlots loads
      for (int i = (nth == 0 ? loads_issued : 0); ok && i < 2 * num_tiles; ++i) {
        if (q_pending && i == q_at && !settle_q()) {
          ok = false;
          break;
        }
        if constexpr (kPacked) {
          if (i == request_at) {
            request_item();
            ++requests;
          }
        }
        const int t = i >> 1;
        int kv_row0, kv_row1 = 0;
        if constexpr (!kPacked) {
          if constexpr (!kDense) {
            // block ids are fetched 32 at a time, one per lane, when the walk enters a new chunk
            const int e = t / kTilesPerBlock;
            if ((i & 1) == 0 && e > 0 && (e & 31) == 0 && t % kTilesPerBlock == 0)
              list_ids = (e + lane < n_entries) ? __ldcg(p.col_idx + cur.list_begin + e + lane) : 0;
          }
          kv_row0 = unpacked_row(t);
        } else {
          const int2 rows = union_rows(nth & 1, t);
          kv_row0 = rows.x;
          kv_row1 = rows.y;
        }
        const int g = load0 + i;
        const int slot = g % kSlots;
        TL(20 + (i & 1));
        if (g >= kSlots) {
          ok = mbar_wait(&sm.done[slot], ((g / kSlots) - 1) & 1, &sm.abort_flag, p.status, 10);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
        }
        issue_load(cur, slot, i & 1, kv_row0, kv_row1);
        TL(22);
      }
      if (ok && q_pending) ok = settle_q();
      if constexpr (kDense) break;
      load0 += 2 * num_tiles;
      if (num_tiles > 0) ++q_tiles_done;
    }
    if constexpr (kPacked) {
      // given up: the launch control's answer must not arrive after the CTA has left (bounded like every wait)
      for (uint32_t i = 0; !ok && requests > 0 && i < kSpinLimit; ++i)
        if (mbar_try_wait(&sm.control_full, (requests - 1) & 1)) break;
    }
  } else if (warp == 5) {
    // =============================== UMMA issuer ========================================
    // descriptor low words: Q is fixed; K/V slots differ only in their base address
    const uint32_t q_lo0 = umma_desc_lo(smem_u32(sm.q[0]), 16);
    const uint32_t kv_lo0 = umma_desc_lo(smem_u32(sm.kv[0][0]), 16);            // as K (K-major)
    const uint32_t v_lo0 = umma_desc_lo(smem_u32(sm.kv[0][0]), kTileN * 128);   // as V (MN-major)
    constexpr uint32_t slot_step = (2 * kTileN * 64 * 2) >> 4;                  // 16 KB per ring slot
    TL_DECL(1)
    bool ok = true;
    int load0 = 0, tile0 = 0, q_loads = 0;   // loads / tiles / Q tiles of earlier items
    for (int nth = 0; ok; ++nth) {
      int num_tiles;
      if constexpr (kPacked) {
        // (the buffer is handed back at once: the issuer needs nothing but the number of tiles)
        const int buf = nth & 1;
        ok = mbar_wait(&sm.item_full[buf], (nth >> 1) & 1, &sm.abort_flag, p.status, 23);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        const int item = sm.item[buf];
        num_tiles = union_tiles(sm.item_entries[buf]);
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.item_free[buf]);
        if (item < 0) break;
      } else {
        if (!kDense && nth > 0) {
          const int item = first_item + nth * static_cast<int>(gridDim.x);
          if (item >= n_items) break;
          cur = describe(item, true);
        }
        num_tiles = unpacked_tiles(cur);
      }
      if (!kDense && num_tiles == 0) continue;
      // S_t = Q K_t^T into S buffer (tile0 + t) & 1
      auto issue_qk = [&](int t) -> bool {
        const int g = load0 + 2 * t;
        const int slot = g % kSlots;
        TL(10);
        bool got = mbar_wait(&sm.kv_full[slot], (g / kSlots) & 1, &sm.abort_flag, p.status, 21);
        got = __all_sync(0xffffffffu, got);
        if (!got) return false;
        TL(11);
        issue_qk64(tmem + kColS + ((tile0 + t) & 1) * kTileN, q_lo0, kv_lo0 + slot * slot_step, &sm.done[slot]);
        TL(12);
        return true;
      };
      ok = mbar_wait(&sm.q_full, q_loads & 1, &sm.abort_flag, p.status, 20);
      ok = __all_sync(0xffffffffu, ok);
      ++q_loads;
      ok = ok && issue_qk(0);
      for (int t = 0; ok && t < num_tiles; ++t) {
        // The S buffer of tile t+1 last held P of the tile two before it, whose P V was issued
        // earlier by this thread, and tcgen05 operations of one thread execute in issue order.
        if (t + 1 < num_tiles && !issue_qk(t + 1)) {
          ok = false;
          break;
        }
        const int g = load0 + 2 * t + 1;
        const int slot = g % kSlots;
        const int gt = tile0 + t;
        TL(13);
        ok = mbar_wait2(&sm.p_full[gt & 1], (gt >> 1) & 1, &sm.kv_full[slot], (g / kSlots) & 1, &sm.abort_flag,
                        p.status, 22);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        TL(14);
        // the first P V of an item overwrites O: the softmax warps handed P over after they had read the
        // previous item's O out in their epilogue
        issue_pv64(tO, tmem + kColS + (gt & 1) * kTileN, v_lo0 + slot * slot_step, t > 0, &sm.done[slot]);
        TL(15);
      }
      if constexpr (kDense) break;
      load0 += 2 * num_tiles;
      tile0 += num_tiles;
    }
  } else {
    // =============================== softmax / epilogue =================================
    const uint32_t lane_base = static_cast<uint32_t>(warp * 32) << 16;
    const float scale_log2 = p.scale_log2;
    // packed walk: this warp's 32 rows belong to one query block
    const int my_group = kPacked ? (warp * 32) / kBlock : 0;
    bool ok = true;
    TL_DECL(0)
    int load0 = 0, tile0 = 0;   // loads / tiles of earlier items
    [[maybe_unused]] uint32_t out_phase = 0;   // output tiles staged so far, modulo 2
    [[maybe_unused]] Item nxt = cur;   // 128-key blocks: the next item's row_ptr entries are fetched one item ahead
    for (int nth = 0; ok; ++nth) {
      int num_tiles;
      if constexpr (kPacked) {
        ok = mbar_wait(&sm.item_full[nth & 1], (nth >> 1) & 1, &sm.abort_flag, p.status, 33);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        const int item = sm.item[nth & 1];
        if (item < 0) break;
        num_tiles = union_tiles(sm.item_entries[nth & 1]);
        cur = describe(item, false);
      } else {
        if constexpr (!kDense) {
          const int item = first_item + nth * static_cast<int>(gridDim.x);
          if (item >= n_items) break;
          cur = nxt;
          if (item + static_cast<int>(gridDim.x) < n_items) nxt = describe(item + static_cast<int>(gridDim.x), true);
        }
        num_tiles = unpacked_tiles(cur);
      }
      [[maybe_unused]] const uint16_t* list = sm.list[nth & 1];
      RowState st{-INFINITY, 0.f};
      // One 64-key tile of the softmax.
      auto tile_body = [&](int t) -> bool {
        TL(1);
        // S_t is ready when the Q K^T batch that read ring load 2t of this item has completed
        const int gk = load0 + 2 * t;
        if (!mbar_wait(&sm.done[gk % kSlots], (gk / kSlots) & 1, &sm.abort_flag, p.status, 30)) return false;
        TL(2);
        tc_fence_after();
        const int buf = (tile0 + t) & 1;   // S buffer of the tile
        const uint32_t tS = tmem + kColS + buf * kTileN + lane_base;
        uint32_t pk[32];
        if constexpr (kPacked) {
          // which 32-column halves of this tile hold key blocks that this warp's query block keeps
          bool keep0, keep1;
          if constexpr (kBlocksPerTile == 1) {
            keep0 = keep1 = ((list[t] >> (kIdBits + my_group)) & 1u) != 0u;
          } else {
            const uint32_t two = *reinterpret_cast<const uint32_t*>(list + 2 * t);
            keep0 = ((two >> (kIdBits + my_group)) & 1u) != 0u;
            keep1 = ((two >> (16 + kIdBits + my_group)) & 1u) != 0u;
          }
          if (!packed_softmax_tile<kBlocksPerTile>(tS, keep0, keep1, scale_log2, st, pk, [&](float alpha) -> bool {
                if (t == 0) return true;
                // O must be quiescent: wait until P_{t-1} V_{t-1} (which read ring load 2t-1) has drained
                const int gp = load0 + 2 * (t - 1) + 1;
                if (!mbar_wait(&sm.done[gp % kSlots], (gp / kSlots) & 1, &sm.abort_flag, p.status, 32)) return false;
                tc_fence_after();
                rescale_accumulator_row(tO + lane_base, alpha);
                if (p.slow_path_events != nullptr && lane == 0) atomicAdd(p.slow_path_events, 1ull);
                return true;
              }))
            return false;
        } else {
          uint32_t r0[32], r1[32];
          tmem_ld32(tS, r0);
          tmem_ld32(tS + 32, r1);
          tmem_wait_ld();
          TL(3);
          if constexpr (kDense) {
            const int valid_cols = p.seq_len - t * kTileN;   // ragged tail of the sequence
            if (valid_cols < kTileN) mask_columns_from(r0, r1, valid_cols);
          }
          float2 sums;
          bool exact = (st.m == -INFINITY);   // nothing accumulated yet: no reference maximum to try
          if (!__all_sync(0xffffffffu, exact)) {
            sums = softmax_group_fast(r0, r1, scale_log2, st.m, pk);
            exact = !(sums.x + sums.y <= 256.0f);   // logits outgrew the running maximum (or NaN)
          }
          if (__any_sync(0xffffffffu, exact)) {
            const float alpha = softmax_group_exact(r0, r1, scale_log2, st, pk, sums);
            if (t > 0) {
              // O must be quiescent: wait until P_{t-1} V_{t-1} (which read ring load 2t-1) has drained
              const int gp = load0 + 2 * (t - 1) + 1;
              if (!mbar_wait(&sm.done[gp % kSlots], (gp / kSlots) & 1, &sm.abort_flag, p.status, 32)) return false;
              tc_fence_after();
              rescale_accumulator_row(tO + lane_base, alpha);
              if (p.slow_path_events != nullptr && lane == 0) atomicAdd(p.slow_path_events, 1ull);
            }
          }
          st.l += sums.x + sums.y;
        }
        TL(4);
        tmem_st32(tS, pk);  // P_t over the first 32 columns of S_t
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(&sm.p_full[buf]);
        TL(5);
        return true;
      };
      for (int t = 0; ok && t < num_tiles; ++t) ok = tile_body(t);
      if constexpr (kPacked) {
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.item_free[nth & 1]);
      }
      if constexpr (kDense) {
        // ---- epilogue of the dense walk: O / l -> bf16 -> global, each row from its own thread ----------
        // (with the staged epilogue of the other walks its main loop compiled 1-2 % slower, measured, and its
        // epilogue is 0.3 % of a 64k launch)
        if (!ok) break;
        if (num_tiles > 0) {
          const int gl = load0 + 2 * (num_tiles - 1) + 1;   // the last P V read this load's slot
          ok = mbar_wait(&sm.done[gl % kSlots], (gl / kSlots) & 1, &sm.abort_flag, p.status, 31);
        }
        tc_fence_after();
        const int row = cur.q_row0 + tid;
        const bool row_valid = row < p.seq_len;
        const float inv_l = st.l > 0.f ? (1.f / st.l) : 0.f;
        __nv_bfloat16* o_row = reinterpret_cast<__nv_bfloat16*>(p.o) + cur.batch * p.o_stride_b +
                               cur.head * p.o_stride_h + static_cast<int64_t>(row) * p.o_stride_t;
        store_output_row(tO + lane_base, num_tiles > 0, inv_l, o_row, row_valid);
        if (p.lse != nullptr && row_valid)
          p.lse[static_cast<int64_t>(cur.bh) * p.seq_len + row] = (st.m + log2f(st.l)) * 0.69314718055994531f;
      } else {
        // ---- epilogue: O / l -> bf16 -> shared memory -> global (an empty list gives zeros) ----------
        if (ok && num_tiles > 0) {
          const int gl = load0 + 2 * (num_tiles - 1) + 1;   // the last P V read this load's slot
          ok = mbar_wait(&sm.done[gl % kSlots], (gl / kSlots) & 1, &sm.abort_flag, p.status, 31);
        }
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
        const float inv_l = st.l > 0.f ? (1.f / st.l) : 0.f;
        if (num_tiles == 0) {
          // no keys: zeros, straight from registers (the Q buffer may already hold a later item's tile)
          const int row = cur.q_row0 + tid;
          __nv_bfloat16* o_row = reinterpret_cast<__nv_bfloat16*>(p.o) + cur.batch * p.o_stride_b +
                                 cur.head * p.o_stride_h + static_cast<int64_t>(row) * p.o_stride_t;
          store_output_row(0u, false, 0.f, o_row, row < p.seq_len);
        } else {
          // The Q tile is dead (the item's last Q K^T completed before its last P V did): it stages the output.
          // The first warp waits for the others' rows and sends the tile off; the others run on.
          stage_output_row(tO + lane_base, true, inv_l, &sm.q[0][0], tid);
          __syncwarp();
          if (lane == 0) mbar_arrive(&sm.o_staged);
          if (warp == 0) {
            ok = mbar_wait(&sm.o_staged, out_phase, &sm.abort_flag, p.status, 34);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
          }
          out_phase ^= 1u;
          if (tid == 0) {
            // rows beyond the sequence end are clipped by the tensor map
            tma_store_4d(&tm_o, sm.q[0], 0, cur.q_row0, cur.head, cur.batch);
            tma_store_4d(&tm_o, sm.q[1], 64, cur.q_row0, cur.head, cur.batch);
            tma_store_commit();
            tma_store_wait_read();
            mbar_arrive(&sm.q_free);
          }
        }
      }
      if constexpr (kDense) break;
      tc_fence_before();   // the next item's first P V overwrites O: order these reads before its hand-over
      load0 += 2 * num_tiles;
      tile0 += num_tiles;
    }
  }

  // ---- teardown ------------------------------------------------------------------------
  tc_fence_before();
  __syncthreads();
  if (warp == 5) {
    __syncwarp();
    tmem_dealloc(tmem, kTmemCols);
  }
}

template <int kBlock, bool kDense, bool kOverlap>
cudaError_t launch(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& to,
                   const AttnParams& p, cudaStream_t stream) {
  auto kernel = attn_kernel<kBlock, kDense, kOverlap>;
  const int smem = static_cast<int>(sizeof(AttnSmem<kBlock>));
  static_assert(sizeof(AttnSmem<kBlock>) <= 113 * 1024, "two CTAs per SM");
  static SmemLimit limit;  // per template instantiation
  cudaError_t e = ensure_dynamic_smem(kernel, smem, limit);
  if (e != cudaSuccess) return e;
  long long ctas = p.num_items;
  if (ctas <= 0) return cudaSuccess;
  // 128-key blocks: at most as many CTAs as are resident at once, each with its share of the items
  if (kBlock == 128 && !kDense && p.max_ctas > 0 && ctas > p.max_ctas) ctas = p.max_ctas;
  // (128-key blocks: as many CTAs as fit may still stand for more items)
  const bool overlap = kOverlap && (kBlock < 128 || p.num_items <= p.max_ctas);
  return launch_overlapped(kernel, ctas, overlap ? p.max_ctas : 0, kThreads, smem, stream, tq, tk, tv, to, p);
}

}  // namespace

int attn_sparse_max_blocks(int block_size) { return block_size < kTileM ? kMaxPackedBlocks : 16384; }

// Tensor maps: Q and O boxes 64 x 128 rows, K and V boxes 64 x min(64, block_size) rows.
// p.num_q_tiles = ceil(seq_len / 128), p.num_blocks = seq_len / block_size.
cudaError_t launch_attn_sparse(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv,
                               const CUtensorMap& to, const AttnParams& p, int block_size, cudaStream_t stream) {
  if (block_size == 128) return launch<128, false, true>(tq, tk, tv, to, p, stream);
  if (block_size == 64) return launch<64, false, true>(tq, tk, tv, to, p, stream);
  return launch<32, false, true>(tq, tk, tv, to, p, stream);
}

// Tensor maps: Q and O boxes 64 x 128 rows, K and V boxes 64 x 64 rows. p.num_q_tiles = ceil(seq_len / 128).
cudaError_t launch_attn_dense(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv,
                              const CUtensorMap& to, const AttnParams& p, cudaStream_t stream) {
  return p.num_items <= p.max_ctas ? launch<128, true, true>(tq, tk, tv, to, p, stream)
                                   : launch<128, true, false>(tq, tk, tv, to, p, stream);
}

}  // namespace sparsed
