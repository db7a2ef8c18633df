// Attention (dense, with or without the row statistics of the switch step, and block-sparse over CSR block lists) for
// grids of no more query tiles than the device has SMs: the work of attention.cu, bit for bit, by a CTA that has an SM to
// itself.
//
// What bounds such a grid is one CTA's chain of 64-key tiles. In attention.cu that is 1290 clocks a tile: one warp issues
// both kinds of MMAs, each batch with a commit and a poll of its own, and one group of softmax warps waits for its logits,
// exponentiates, stores and hands over one tile after the other. Here
//   warps 0, 3     : TMA, a ring of K tiles and a ring of V tiles
//   warp 1         : UMMA issuer of S = Q K^T. Q is copied to tensor memory first: such an instruction takes 32 clocks
//                    instead of 48 when the 128 rows of Q need not be read from shared memory again. Four S buffers, so
//                    that it runs up to three tiles ahead
//   warp 2         : UMMA issuer of O += P V
//   warps 4-7, 8-11: two groups of softmax warps, one thread per row each; group g takes tiles g, g + 2, ...; a warp and
//                    the one of the other group with the same 32 rows pass the rows' state (reference maximum, sum) on
//                    from tile to tile through shared memory
// and a tile takes 960 clocks, 0.49 us: 2 heads x 4096 tokens 44.0 -> 35.8 us, 2 x 1024 14.8 -> 11.9. What bounds it now is
// the chain of a tile's steps, none of them alone: copies with work left out took, instead of 36.0 us (2 x 4096), 35.9 with
// K and V loaded for the first five tiles only, 34.0 without exponentials, 35.0 without either. (32 KB of K and V a tile are
// 66 GB/s; bulk copies alone get 71.2 GB/s into an SM, however many SMs take part.)
// (One issuer for both: 46.9 and 14.9 us. Q from shared memory and one loading warp: 37.7 and 13.2. The next tile's logits
// copied while a tile is finished, or each tile's columns split between two warps, 16 in all: no gain.)
// A tile is exponentiated against the reference its group knows, before the tile before it is known to have kept it; if
// it has not (rare, softmax_pipeline.cuh), the tile is done again from S, which is still in tensor memory. P is handed
// over only after that. So rows see the same maxima, and sums and products are added in the same order, as with one group.
#include "internal.h"
#include "softmax_pipeline.cuh"
#include "work_items.cuh"

namespace sparsed {
namespace {

constexpr int kHeadDim = 128;
constexpr int kLoadK = 0, kIssuerQK = 1, kIssuerPV = 2, kLoadV = 3, kSoftmax = 4;   // warps (kSoftmax: the first of 8)
constexpr int kThreads = 384;
constexpr int kSlots = 5;                   // of the K ring and of the V ring, 16 KB each
constexpr int kSBuffers = 4;
constexpr uint32_t kSlotStep = (2 * kTileN * 64 * 2) >> 4;   // a ring slot, in descriptor units
constexpr int kTmemCols = 512;
constexpr int kColO = kSBuffers * kTileN;   // O accumulator (fp32, 128 columns) behind the S buffers
constexpr int kColQ = kColO + kHeadDim;     // Q as bf16 pairs (64 columns)

// Position in a ring: slot and barrier parity of use number n, counted on by `step` uses at a time.
struct TilePos {
  int slot;
  uint32_t phase;
  __device__ __forceinline__ explicit TilePos(int n) : slot(n % kSlots), phase((n / kSlots) & 1) {}
  __device__ __forceinline__ void advance(int step) {
    slot += step;
    if (slot >= kSlots) {
      slot -= kSlots;
      phase ^= 1u;
    }
  }
};

template <int kBlock>
struct LoneSmem {
  static constexpr bool kPacked = kBlock < kTileM;
  static constexpr int kGroups = kTileM / kBlock;          // query blocks of the item
  alignas(1024) __nv_bfloat16 q[2][kTileM * 64];           // two 64-wide halves of head_dim
  alignas(1024) __nv_bfloat16 k[kSlots][2][kTileN * 64];   // each slot: two 64-wide halves of head_dim
  alignas(1024) __nv_bfloat16 v[kSlots][2][kTileN * 64];
  uint64_t q_full, q_ready;  // Q is in shared memory, in tensor memory
  uint64_t k_full[kSlots], v_full[kSlots];
  uint64_t s_full[kSlots];   // Q K^T of the slot's tile has completed: S is ready, the slot is free
  uint64_t v_done[kSlots];   // P V of the slot's tile has completed: the slot and the tile's S buffer are free
  uint64_t p_full[kSBuffers];
  uint64_t turn[2][4];       // [group][32-row quarter]: the other group has passed the rows' state on
  float2 state[kTileM];      // reference maximum and sum of each row, after the last tile done with
  float carry[kTileM];       // 128-key statistics: the sum over the group's first tile (group 0's) for group 1's
  uint32_t tmem_base;
  int abort_flag;
  int entries;               // packed walks: key blocks in the union, and the union (work_items.cuh)
  alignas(16) uint16_t list[kPacked ? kMaxPackedBlocks + 2 : 2];
  uint32_t member[kGroups][kMemberWords<kBlock>];
};

// kStatKeys: record one row statistic per 32 / 64 / 128 keys (RowStatWriter in softmax_pipeline.cuh), or none (0).
template <int kBlock, bool kDense, int kStatKeys>
__global__ void __launch_bounds__(kThreads, 1)
attn_lone_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                 const __grid_constant__ CUtensorMap tm_v, const AttnParams p) {
  static_assert(!kDense || kBlock == 128, "the dense walk uses the unpacked layout");
  using Smem = LoneSmem<kBlock>;
  constexpr bool kPacked = Smem::kPacked;
  constexpr int kGroups = Smem::kGroups;
  constexpr int kTilesPerBlock = kBlock >= kTileN ? kBlock / kTileN : 1;   // 128-key block: two tiles
  constexpr int kBlocksPerTile = kBlock >= kTileN ? 1 : kTileN / kBlock;   // 32-key blocks: two per tile
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
  const int tid = threadIdx.x;
  const int warp = tid >> 5;
  const int lane = tid & 31;
  // ---- what needs nothing of the kernel before this one (which may still run) ------------------------------------
  WorkItem it = describe_item<kGroups, kDense>(p, blockIdx.x, false);
  if (tid == kLoadK * 32) {
    mbar_init(&sm.q_full, 1);
    for (int s = 0; s < kSlots; ++s) mbar_init(&sm.k_full[s], 1);
    mbar_fence_init();
    tma_prefetch_desc(&tm_q);
    tma_prefetch_desc(&tm_k);
  } else if (tid == kLoadV * 32) {
    for (int s = 0; s < kSlots; ++s) {
      mbar_init(&sm.v_full[s], 1);
      mbar_init(&sm.s_full[s], 1);
      mbar_init(&sm.v_done[s], 1);
    }
    for (int s = 0; s < kSBuffers; ++s) mbar_init(&sm.p_full[s], 4);
    for (int s = 0; s < 8; ++s) mbar_init(&sm.turn[s >> 2][s & 3], 1);
    mbar_init(&sm.q_ready, 8);
    sm.abort_flag = 0;
    mbar_fence_init();
    tma_prefetch_desc(&tm_v);
  }
  __syncwarp();
  wait_for_previous_kernel();
  if ((smem_u32(smem_raw) & 1023u) != 0u) {
    if (threadIdx.x == 0 && atomicCAS(&p.status->code, 0, 2) == 0) p.status->where = 4;
    return;
  }

  // ---- set-up: the loading warp of K starts before the rest of the CTA is ready -------------------------------------
  int list_ids = 0;       // unpacked walk, loading warps: lane i holds the block id of list entry 32 * chunk + i
  int loads_issued = 0;
  auto fetch_ids = [&](int e, int n) {
    if constexpr (!kPacked && !kDense) list_ids = e + lane < n ? __ldcg(p.col_idx + it.list_begin + e + lane) : 0;
  };
  auto issue_load = [&](const CUtensorMap* tm, __nv_bfloat16 (&tile)[2][kTileN * 64], uint64_t* full, int2 rows) {
    if (elect_one_sync()) {
      mbar_expect_tx(full, kTileN * kHeadDim * 2);
      tma_load_4d(tile[0], tm, full, 0, rows.x, it.kv_head, it.batch);
      tma_load_4d(tile[1], tm, full, 64, rows.x, it.kv_head, it.batch);
      if constexpr (kBlocksPerTile == 2) {   // boxes of 32 rows
        tma_load_4d(tile[0] + kBlock * 64, tm, full, 0, rows.y, it.kv_head, it.batch);
        tma_load_4d(tile[1] + kBlock * 64, tm, full, 64, rows.y, it.kv_head, it.batch);
      }
    }
    __syncwarp();
  };
  // first key rows of tile t (of both its blocks with 32-key blocks)
  auto key_rows = [&](int t) -> int2 {
    if constexpr (kDense) return make_int2(t * kTileN, 0);
    constexpr uint32_t ids = (1u << kIdBits) - 1u;
    if constexpr (kPacked && kBlocksPerTile == 1) return make_int2(static_cast<int>(sm.list[t] & ids) * kBlock, 0);
    if constexpr (kPacked && kBlocksPerTile == 2) {
      const uint32_t two = *reinterpret_cast<const uint32_t*>(&sm.list[2 * t]);
      return make_int2(static_cast<int>(two & ids) * kBlock, static_cast<int>((two >> 16) & ids) * kBlock);
    }
    const int e = t / kTilesPerBlock;
    return make_int2(__shfl_sync(0xffffffffu, list_ids, e & 31) * kBlock + (t % kTilesPerBlock) * kTileN, 0);
  };
  auto tiles_of = [&](int n) -> int {   // 64-key tiles of a list (or union) of n blocks; dense: n tiles
    return kDense ? n : kBlocksPerTile == 2 ? (n + 1) / 2 : n * kTilesPerBlock;
  };
  if (!kDense && (!kPacked || warp == kLoadK)) read_list_bounds(p, it);
  if (warp == kLoadK) {
    if (elect_one_sync()) {
      mbar_expect_tx(&sm.q_full, kTileM * kHeadDim * 2);   // rows beyond the sequence arrive as zeros
      tma_load_4d(sm.q[0], &tm_q, &sm.q_full, 0, it.q_row0, it.head, it.batch);
      tma_load_4d(sm.q[1], &tm_q, &sm.q_full, 64, it.q_row0, it.head, it.batch);
    }
    __syncwarp();
    int n = it.list_len;
    if constexpr (kPacked) {
      n = build_list_union<kGroups, kBlocksPerTile>(p, it, lane, sm.member, sm.list);
      if (lane == 0) sm.entries = n;
    }
    fetch_ids(0, n);
    __syncwarp();
    for (const int first = min(tiles_of(n), 2); loads_issued < first; ++loads_issued)
      issue_load(&tm_k, sm.k[loads_issued], &sm.k_full[loads_issued], key_rows(loads_issued));
  }
  if (warp == kIssuerQK) {
    tmem_alloc(&sm.tmem_base, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem_base;
  const uint32_t tO = tmem + kColO;
  const int n_entries = kPacked ? sm.entries : it.list_len;
  const int num_tiles = tiles_of(n_entries);
  auto wait = [&](uint64_t* bar, uint32_t phase, int where) -> bool {   // the same for the whole warp
    return __all_sync(0xffffffffu, mbar_wait(bar, phase, &sm.abort_flag, p.status, where));
  };
  auto wait2 = [&](uint64_t* a, uint32_t phase_a, uint64_t* b, uint32_t phase_b, int where) -> bool {
    return __all_sync(0xffffffffu, mbar_wait2(a, phase_a, b, phase_b, &sm.abort_flag, p.status, where));
  };

  if (warp == kLoadK || warp == kLoadV) {
    // =============================== TMA: a ring of K tiles, a ring of V tiles ===========
    const bool is_k = warp == kLoadK;
    if (!is_k) fetch_ids(0, n_entries);
    TilePos pos(loads_issued);
    for (bool ok = true; loads_issued < num_tiles; ++loads_issued, pos.advance(1)) {
      const int t = loads_issued;
      if constexpr (!kPacked && !kDense) {
        // block ids are fetched 32 at a time, one per lane, when the walk enters a new chunk
        const int e = t / kTilesPerBlock;
        if (e > 0 && (e & 31) == 0 && t % kTilesPerBlock == 0) fetch_ids(e, n_entries);
      }
      const int2 rows = key_rows(t);
      if (t >= kSlots) ok = wait(is_k ? &sm.s_full[pos.slot] : &sm.v_done[pos.slot], pos.phase ^ 1u, is_k ? 70 : 71);
      if (!ok) break;
      if (is_k) {
        issue_load(&tm_k, sm.k[pos.slot], &sm.k_full[pos.slot], rows);
      } else {
        issue_load(&tm_v, sm.v[pos.slot], &sm.v_full[pos.slot], rows);
      }
    }
  } else if (warp == kIssuerQK) {
    // =============================== UMMA issuer: S = Q K^T ==============================
    const uint32_t k_lo0 = umma_desc_lo(smem_u32(sm.k[0][0]), 16);   // K-major
    TilePos pos(0), freed(0);
    bool ok = num_tiles == 0 || wait(&sm.q_ready, 0, 72);
    for (int t = 0; ok && t < num_tiles; ++t, pos.advance(1)) {
      if (t < kSBuffers) {
        ok = wait(&sm.k_full[pos.slot], pos.phase, 73);
      } else {
        // the S buffer last held P of the tile kSBuffers before, whose P V must have completed
        ok = wait2(&sm.k_full[pos.slot], pos.phase, &sm.v_done[freed.slot], freed.phase, 73);
        freed.advance(1);
      }
      if (ok) issue_qk64_ts(tmem + (t % kSBuffers) * kTileN, tmem + kColQ, k_lo0 + pos.slot * kSlotStep, &sm.s_full[pos.slot]);
    }
  } else if (warp == kIssuerPV) {
    // =============================== UMMA issuer: O += P V ===============================
    const uint32_t v_lo0 = umma_desc_lo(smem_u32(sm.v[0][0]), kTileN * 128);   // MN-major
    TilePos pos(0);
    bool ok = true;
    for (int t = 0; ok && t < num_tiles; ++t, pos.advance(1)) {
      ok = wait2(&sm.p_full[t % kSBuffers], (t / kSBuffers) & 1, &sm.v_full[pos.slot], pos.phase, 74);
      if (ok) issue_pv64(tO, tmem + (t % kSBuffers) * kTileN, v_lo0 + pos.slot * kSlotStep, t > 0, &sm.v_done[pos.slot]);
    }
  } else {
    // =============================== softmax / epilogue =================================
    const int g = (warp - kSoftmax) >> 2;
    const int quarter = warp & 3;
    const int row_in_tile = 32 * quarter + lane;
    const uint32_t lane_base = static_cast<uint32_t>(quarter * 32) << 16;
    const float scale_log2 = p.scale_log2;
    [[maybe_unused]] const int my_block = (quarter * 32) / kBlock;   // packed walks: this warp's query block of the item
    bool ok = wait(&sm.q_full, 0, 75);
    {
      // Q from shared to tensor memory, 64 columns of head_dim per group
      uint32_t r[32];
      const uint8_t* q_row = reinterpret_cast<const uint8_t*>(sm.q[g]) + row_in_tile * 128;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const uint4 x = *reinterpret_cast<const uint4*>(q_row + ((c ^ (row_in_tile & 7)) << 4));
        r[4 * c] = x.x;
        r[4 * c + 1] = x.y;
        r[4 * c + 2] = x.z;
        r[4 * c + 3] = x.w;
      }
      tmem_st32(tmem + kColQ + 32 * g + lane_base, r);
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.q_ready);
    }
    RowState st{-INFINITY, 0.f};
    // this row's first statistic
    [[maybe_unused]] float* stats = nullptr;
    [[maybe_unused]] const int stat_groups = kStatKeys > 0 ? (p.seq_len + kStatKeys - 1) / kStatKeys : 0;
    if (kStatKeys > 0 && it.q_row0 + row_in_tile < p.seq_len)
      stats = p.tile_lse + (static_cast<int64_t>(it.bh) * p.num_q_tiles + it.q_tile) * stat_groups * kTileM + row_in_tile;
    // takes over the row's state after the other group's nth tile
    auto take_state = [&](int nth) -> bool {
      if (!wait(&sm.turn[g][quarter], nth & 1, 76)) return false;
      const float2 before = sm.state[row_in_tile];
      st.m = before.x;
      st.l = before.y;
      return true;
    };
    TilePos pos(g);
    for (int t = g; ok && t < num_tiles; t += 2, pos.advance(2)) {
      if (!(ok = wait(&sm.s_full[pos.slot], pos.phase, 77))) break;
      tc_fence_after();
      const uint32_t tS = tmem + (t % kSBuffers) * kTileN + lane_base;
      bool keep0 = true, keep1 = true;   // packed walks: whether this warp's query block keeps the tile's 32-column halves
      if constexpr (kPacked && kBlocksPerTile == 1) keep0 = keep1 = ((sm.list[t] >> (kIdBits + my_block)) & 1u) != 0u;
      if constexpr (kPacked && kBlocksPerTile == 2) {
        const uint32_t two = *reinterpret_cast<const uint32_t*>(&sm.list[2 * t]);
        keep0 = ((two >> (kIdBits + my_block)) & 1u) != 0u;
        keep1 = ((two >> (16 + kIdBits + my_block)) & 1u) != 0u;
      }
      const bool kept = keep0 || keep1;
      const int valid_cols = kDense ? p.seq_len - t * kTileN : kTileN;   // ragged tail of the sequence
      uint32_t pk[32];
      float2 sums = make_float2(0.f, 0.f);
      [[maybe_unused]] float carry = 0.f;   // 128-key statistics: the tile before this one, in group 1
      bool tried = false;   // pk and sums hold the tile against st.m (where that is a number)
      auto load_logits = [&](uint32_t (&r0)[32], uint32_t (&r1)[32]) {
        tmem_ld32(tS, r0);
        tmem_ld32(tS + 32, r1);
        tmem_wait_ld();
        if (valid_cols < kTileN) mask_columns_from(r0, r1, valid_cols);
      };
      auto fast = [&]() {
        tried = !__all_sync(0xffffffffu, st.m == -INFINITY);
        if (!tried) return;
        if (kBlocksPerTile == 1 || (keep0 && keep1)) {
          uint32_t r0[32], r1[32];
          load_logits(r0, r1);
          sums = softmax_group_fast(r0, r1, scale_log2, st.m, pk);
        } else {
          uint32_t r[32], half[16];
          tmem_ld32(keep0 ? tS : tS + 32, r);
          tmem_wait_ld();
          sums = make_float2(softmax_half_fast(r, scale_log2, st.m, half), 0.f);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            pk[j] = keep0 ? half[j] : 0u;
            pk[16 + j] = keep0 ? 0u : half[j];
          }
        }
      };
      if (kept) fast();
      if (t > 0) {
        const float m = st.m;
        if (!(ok = take_state((t - 1) >> 1))) break;   // after tile t - 1
        if (kStatKeys == 128 && g == 1) carry = sm.carry[row_in_tile];
        if (kept && __any_sync(0xffffffffu, m != st.m)) fast();
      }
      if (kept) {
        const bool exact = !tried || !(sums.x + sums.y <= 256.0f);   // no reference yet, logits that outgrew it, or NaN
        if (__any_sync(0xffffffffu, exact)) {
          uint32_t r0[32], r1[32];
          load_logits(r0, r1);
          if (!keep0) {
#pragma unroll
            for (int j = 0; j < 32; ++j) r0[j] = 0xff800000u;   // -inf
          }
          if (!keep1) {
#pragma unroll
            for (int j = 0; j < 32; ++j) r1[j] = 0xff800000u;
          }
          const float alpha = softmax_group_exact(r0, r1, scale_log2, st, pk, sums);
          if constexpr (kStatKeys == 128) carry *= alpha;
          if (t > 0) {
            // O must be quiescent: wait until P_{t-1} V_{t-1} has drained
            const TilePos last(t - 1);
            if (!(ok = wait(&sm.v_done[last.slot], last.phase, 78))) break;
            tc_fence_after();
            rescale_accumulator_row(tO + lane_base, alpha);
            if (p.slow_path_events != nullptr && lane == 0) atomicAdd(p.slow_path_events, 1ull);
          }
        }
        st.l += sums.x + sums.y;
      } else {
#pragma unroll
        for (int j = 0; j < 32; ++j) pk[j] = 0u;
      }
      sm.state[row_in_tile] = make_float2(st.m, st.l);
      if (kStatKeys == 128 && g == 0) sm.carry[row_in_tile] = sums.x + sums.y;
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.turn[g ^ 1][quarter]);
      tmem_st32(tS, pk);  // P_t over the first 32 columns of S_t
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.p_full[t % kSBuffers]);
      if (kStatKeys > 0 && stats != nullptr) {
        if constexpr (kStatKeys == 64) __stcs(stats + t * kTileM, st.m + fast_log2(sums.x + sums.y));
        if constexpr (kStatKeys == 32) {
          __stcs(stats + 2 * t * kTileM, st.m + fast_log2(sums.x));
          if (2 * t + 1 < stat_groups) __stcs(stats + (2 * t + 1) * kTileM, st.m + fast_log2(sums.y));
        }
        // (the sequence is a whole number of 128-key groups here: each ends with a tile of group 1)
        if (kStatKeys == 128 && g == 1) __stcs(stats + (t >> 1) * kTileM, st.m + fast_log2(carry + (sums.x + sums.y)));
      }
    }
    // ---- epilogue: O / l -> bf16 -> shared memory -> global, 64 columns of head_dim per group ----------------------
    const int row = it.q_row0 + row_in_tile;
    __nv_bfloat16* o = reinterpret_cast<__nv_bfloat16*>(p.o) + it.batch * p.o_stride_b + it.head * p.o_stride_h;
    if (num_tiles == 0) {
      // no keys: zeros, straight from registers
      if (g == 0) store_output_row(0u, false, 0.f, o + static_cast<int64_t>(row) * p.o_stride_t, row < p.seq_len);
    } else {
      // Every thread goes through the barrier below even after a wait has run out (it then stages zeros), so that none is
      // left waiting there; what is done after it is decided by the shared flag.
      if (ok && (num_tiles & 1) == g) ok = take_state((num_tiles - 1) >> 1);   // the other group did the last tile
      const TilePos last(num_tiles - 1);
      ok = ok && wait(&sm.v_done[last.slot], last.phase, 79);
      tc_fence_after();
      const float inv_l = st.l > 0.f ? (1.f / st.l) : 0.f;
      // the Q tile in shared memory is dead: it stages the output, group g's 64 columns in half g
      stage_output_half(tO + lane_base + 64 * g, ok, inv_l, sm.q[g], row_in_tile);
      named_barrier_sync(1 + g, 128);
      if (*reinterpret_cast<volatile int*>(&sm.abort_flag) == 0) {
        // Eight threads to a row's 128 bytes. (A TMA store's thread would wait 1300 clocks for the tile to be read.)
        const int chunk = lane & 7;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int r = 16 * i + 4 * quarter + (lane >> 3);
          const uint4 x = *reinterpret_cast<const uint4*>(reinterpret_cast<const uint8_t*>(sm.q[g]) + r * 128 +
                                                          ((chunk ^ (r & 7)) << 4));
          if (it.q_row0 + r < p.seq_len)
            *reinterpret_cast<uint4*>(o + static_cast<int64_t>(it.q_row0 + r) * p.o_stride_t + 64 * g + 8 * chunk) = x;
        }
        if (g == 0 && p.lse != nullptr && row < p.seq_len)
          p.lse[static_cast<int64_t>(it.bh) * p.seq_len + row] = (st.m + log2f(st.l)) * 0.69314718055994531f;
      }
    }
  }

  // ---- teardown ------------------------------------------------------------------------
  tc_fence_before();
  __syncthreads();
  if ((warp == kLoadK || warp == kLoadV) && sm.abort_flag != 0) {
    // given up: the loads in flight must have landed before the CTA leaves (bounded like every wait)
    auto drain = [&](uint64_t* bar, uint32_t phase) {
      for (uint32_t n = 0; n < kSpinLimit && !mbar_try_wait(bar, phase); ++n) {
      }
    };
    for (int t = max(loads_issued - kSlots, 0); t < loads_issued; ++t)
      drain((warp == kLoadK ? sm.k_full : sm.v_full) + t % kSlots, (t / kSlots) & 1);
    drain(&sm.q_full, 0);
  }
  if (warp == kIssuerQK) {
    __syncwarp();
    tmem_dealloc(tmem, kTmemCols);
  }
}

template <int kBlock, bool kDense, int kStatKeys>
cudaError_t launch(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const AttnParams& p,
                   cudaStream_t stream) {
  auto kernel = attn_lone_kernel<kBlock, kDense, kStatKeys>;
  const int smem = static_cast<int>(sizeof(LoneSmem<kBlock>));
  static_assert(sizeof(LoneSmem<kBlock>) > 114 * 1024 && sizeof(LoneSmem<kBlock>) <= 227 * 1024, "one CTA per SM");
  static SmemLimit limit;  // per template instantiation
  cudaError_t e = ensure_dynamic_smem(kernel, smem, limit);
  if (e != cudaSuccess) return e;
  if (p.num_items <= 0) return cudaSuccess;
  return launch_overlapped(kernel, p.num_items, p.max_ctas / 2, kThreads, smem, stream, tq, tk, tv, p);
}

}  // namespace

// Tensor maps of both as in attention.cu.
cudaError_t launch_attn_sparse_lone(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv,
                                    const AttnParams& p, int block_size, cudaStream_t stream) {
  if (block_size == 128) return launch<128, false, 0>(tq, tk, tv, p, stream);
  if (block_size == 64) return launch<64, false, 0>(tq, tk, tv, p, stream);
  return launch<32, false, 0>(tq, tk, tv, p, stream);
}

cudaError_t launch_attn_dense_lone(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv,
                                   const AttnParams& p, cudaStream_t stream) {
  if (p.tile_lse == nullptr) return launch<128, true, 0>(tq, tk, tv, p, stream);
  if (p.stat_keys == 128) return launch<128, true, 128>(tq, tk, tv, p, stream);
  if (p.stat_keys == 64) return launch<128, true, 64>(tq, tk, tv, p, stream);
  return launch<128, true, 32>(tq, tk, tv, p, stream);
}

}  // namespace sparsed
