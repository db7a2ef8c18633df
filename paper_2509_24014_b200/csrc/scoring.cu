// Block-pooled attention scores A' = avgpool(softmax(Q K^T / sqrt(d)), block_size) from Q and K alone
// ("Isolated Selection"; the avgpool line of Algorithm 1), streamed one 128-row query tile at a time so that
// the l x l matrix is never stored.
//
// What bounds it: one exponential per logit. The SM's exponential unit does 16 a clock, so a 128 x 64 tile of
// logits takes 512 clocks there against 384 on the tensor pipe (eight M128 N64 K16 MMAs at 48 clocks). Every logit
// is therefore exponentiated ONCE where that is possible:
//
//   * kOnePass  the row sums of every key block are kept, relative to a per-row reference that is fixed with the
//               first tile, until the row's denominator is known; then they are divided by it and summed over the
//               rows of each query block. One fp32 per row and key block, in the tensor-memory columns that the
//               two logit buffers leave free: 128 of a CTA's 256, so up to 128 key blocks per row.
//   * kOnePassWide  the same with one CTA per SM and all of its tensor memory: up to 384 key blocks per row. Half
//               as many softmax warps keep the exponential unit less busy, but there is one pass instead of two.
//   * kOnePassMost  ... and 128 more sums in 64 KB of shared memory: up to 512 (4 % slower for telling them apart).
//   * kPooled   the caller (or a kRowStats pass) has the rows' log-sum-exp: p = exp(s - LSE) is the probability
//               itself, and the block sums are folded into A' whenever 128 of them have come together.
//   * kRowStats log-sum-exp of every row: the first of the two passes that rows with more than 512 key blocks
//               take.
//
// Pipeline per CTA (320 threads, two CTAs per SM but for kOnePassWide / Most): warp 8 streams 64-key K tiles by TMA
// into a ring of four, warp 9 issues S = Q K^T (one commit per tile: "S ready" for the softmax warps, "slot free" for
// the producer), warps 0-3 and 4-7 are two groups with one thread per query row each. The groups take turns at 128
// keys (two tiles), so that a key block belongs to one of them; each has one S buffer and its own reference and
// denominator of every row, which meet at the end. A thread copies its row of S into registers, hands the buffer back
// at once, exponentiates and sums. Four such warps per scheduler cover each other's waits: with two (one group per
// CTA, two S buffers) the first case below took 2.53 ms, with the next tile's copy pipelined into the current one's
// exponentials as well 2.70 ms. Sums run in a fixed order, so results are bitwise reproducible. When the keys of its
// block-row(s) fit in shared memory the CTA ranks them itself (warp_select_row) and writes the CSR lists.
//
// Measured on B200, from Q and K alone (two passes over the logits before, with two CTAs of four softmax warps):
//   28 heads x 16384 tokens, block 128   6.21 -> 2.43 ms (kOnePass. At 1850 MHz 739 clocks a tile and SM, of which the
//                                        exponential unit needs 512: it bounds the launch together with what its warps
//                                        wait for. Half of the exponentials left out 523 clocks, all of them 498, but the
//                                        clock then falls to 1.6 GHz under the power limit: 1.99 and 1.92 ms. Fold and
//                                        ranking are 1.4 %. No step at whole waves: 203-206 us a wave, 14 to 36 heads)
//   32 heads x 8192 tokens, block 128    1.79 -> 0.72 ms (kOnePass)
//   28 heads x 16384 tokens, block 64    6.24 -> 3.00 ms (kOnePassWide; in two passes 5.0)
//   8 heads x 65536 tokens, block 128    27.4 -> 12.8 ms (kOnePassMost; in two passes 22.3)
//   8 heads x 65536 tokens, block 64     27.6 -> 21.9 ms (kRowStats, kPooled)
// and with the caller's LSE (kPooled, one pass before as well):
//   28 heads x 16384 tokens, block 128   2.48 -> 2.38 ms
//   8 heads x 65536 tokens, block 128    11.2 -> 10.9 ms
//   32 heads x 4096 tokens, block 32     0.193 -> 0.196 ms
#include "internal.h"
#include "softmax_pipeline.cuh"
#include "topk_device.cuh"

namespace sparsed {
namespace {

constexpr int kHeadDim = 128;
constexpr int kTileM = 128;     // query rows per CTA
constexpr int kTileN = 64;      // keys per pipeline step
constexpr int kThreads = 320;
constexpr int kSlots = 4;       // 16 KB ring slots, one K tile each
constexpr int kColStat = 128;   // columns 0-127: one S buffer per group; from 128 on: one block sum per column and row
constexpr int kMaxKeys = 2048;  // ranking keys held in shared memory: (block-rows per tile) x (key blocks per row)

enum ScoreMode { kOnePass, kOnePassWide, kOnePassMost, kPooled, kRowStats };
__host__ __device__ constexpr bool one_per_sm(int mode) { return mode == kOnePassWide || mode == kOnePassMost; }
__host__ __device__ constexpr int tmem_cols(int mode) { return one_per_sm(mode) ? 512 : 256; }
// block sums held per row: in tensor memory, in shared memory, in all
__host__ __device__ constexpr int tmem_sums(int mode) { return tmem_cols(mode) - kColStat; }
__host__ __device__ constexpr int smem_sums(int mode) { return mode == kOnePassMost ? 128 : 0; }
__host__ __device__ constexpr int block_sums(int mode) { return tmem_sums(mode) + smem_sums(mode); }

// Of 16 pairs of exponentials, how many are taken off the exponential unit (exp2_by_polynomial, 16 instructions a pair).
// Only where one CTA per SM leaves issue slots: 28 x 16384 block 64 3292 -> 2996 us with two, 3078 with three, 2982 with
// four; 8 x 65536 block 128 14040 -> 13266, 12800, 13108. As chosen, 32 x 24576 block 64 8190 -> 7445, 28 x 8704 block 64
// 950 -> 869, 16 x 8192 block 32 498 -> 459, 8 x 49152 block 128 7966 -> 7268, 2 x 16384 block 32 (512 key blocks) 282 ->
// 257. With two CTAs per SM there is nothing to gain (28 x 16384 block 128 2458, 2460, 2443, 2493; 2 x 1024 13.9, 13.9,
// 14.8, 14.6): fewer clocks there run at a lower clock, see above.
__host__ __device__ constexpr int poly_pairs(int mode) { return mode == kOnePassMost ? 3 : mode == kOnePassWide ? 2 : 0; }

// A row's reference is the maximum of both groups' first 64-key tiles, and stays until the sum of a later tile outgrows
// this: only fp32 sums are taken here (no bf16 probabilities), so 2^60 is as safe as 1. Sums may thus stand up to 2^66
// above their reference, which is why they are brought to another one in two steps (PowerOfTwo). Both groups start from
// the same reference because a sum's rounding depends on it: equal key blocks then have bitwise equal scores whichever
// group sums them, and rank by index as they should. (A group that has outgrown it goes on with one of its own.)
constexpr float kOutgrown = 1152921504606846976.f;   // 2^60

// 2^e as a product of two factors, each well inside the fp32 range: a sum of 2^60 brought down by 2^-150 is 2^-90, while
// 2^-150 by itself is zero. far is 1 or 2^-64, so that nothing is rounded by applying it.
struct PowerOfTwo {
  float far, near;
};
__device__ __forceinline__ PowerOfTwo power_of_two(float e) {
  const bool low = e < -32.f;   // (2^-32 divided by the largest denominator, 2^76, is still a normal number)
  return {low ? 0x1p-64f : 1.f, fast_exp2(low ? e + 64.f : e)};
}

template <int kMode>
struct ScoreSmem {
  alignas(1024) __nv_bfloat16 q[2][kTileM * 64];           // two 64-wide halves of head_dim
  alignas(1024) __nv_bfloat16 k[kSlots][2][kTileN * 64];   // each slot: two 64-wide halves of head_dim
  uint32_t keys[kMaxKeys];          // ordered keys of this CTA's block-row(s)
  float quarter[4][block_sums(kMode)];   // block sums over each 32-row quarter of the tile
  union {
    int hist[4][256];               // one histogram per ranking warp
    float first_max[2][kTileM];     // before that: the maximum of each row over each group's first tile
  };
  uint64_t q_full, k_full[kSlots];
  uint64_t done[kSlots];            // the MMAs that read the slot have completed: S of that tile is ready
  uint64_t s_free[2];               // every warp of the group has copied its rows of the S buffer into registers
  float more[smem_sums(kMode) > 0 ? smem_sums(kMode) : 1][kTileM];   // block sums beyond those in tensor memory
  float2 ml[2][kTileM];             // each group's (reference, denominator) of each row
  uint32_t tmem_base;
  int abort_flag;
};

// One 32-bit cell per lane, at the warp's lanes of column `taddr`.
__device__ __forceinline__ void tmem_st1(uint32_t taddr, float v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(taddr), "r"(__float_as_uint(v)) : "memory");
}

// v[j] of lane i = element (i, j): returns sum over i of element (i, lane), added pairwise in a fixed tree.
__device__ __forceinline__ float warp_column_sums(float (&v)[32], int lane) {
#pragma unroll
  for (int half = 16; half > 0; half >>= 1) {
    const bool upper = (lane & half) != 0;
#pragma unroll
    for (int j = 0; j < half; ++j) {
      const float keep = upper ? v[j + half] : v[j];
      const float give = upper ? v[j] : v[j + half];
      v[j] = keep + __shfl_xor_sync(0xffffffffu, give, half);
    }
  }
  return v[0];
}

__device__ __forceinline__ float2 twice(float c) { return make_float2(c, c); }

// 2^x without the exponential unit: x = n + f with n whole and |f| <= 1/2, 2^f by the polynomial of degree 6 with the least
// largest relative error there (1.9e-9, found by Lawson's reweighted least squares; 7.9e-8 with its fp32 roundings, where
// ex2.approx has 2^-22), times 2^n put together from its bits. The clamps keep n in [-127, 128], whose bits are those of 0
// and infinity, and hand NaN on.
__device__ __forceinline__ float2 exp2_by_polynomial(float2 x) {
  auto clamp = [](float v) -> float {
    float y;
    asm("max.NaN.f32 %0, %1, 0fC2FE0000;" : "=f"(y) : "f"(v));   // -127
    asm("min.NaN.f32 %0, %1, 0f43000000;" : "=f"(y) : "f"(y));   // 128
    return y;
  };
  x = make_float2(clamp(x.x), clamp(x.y));
  const float2 t = __fadd2_rn(x, twice(12582912.f));   // 1.5 * 2^23 + n: n in the low bits
  const float2 f = __fadd2_rn(x, __ffma2_rn(t, twice(-1.f), twice(12582912.f)));
  float2 y = twice(0x1.41d332d89fe66p-13f);
  y = __ffma2_rn(y, f, twice(0x1.5f456a8954f25p-10f));
  y = __ffma2_rn(y, f, twice(0x1.3b2dbbc1d72d0p-7f));
  y = __ffma2_rn(y, f, twice(0x1.c6aed4b954772p-5f));
  y = __ffma2_rn(y, f, twice(0x1.ebfbdadcaf7c8p-3f));
  y = __ffma2_rn(y, f, twice(0x1.62e430c7e91fcp-1f));
  y = __ffma2_rn(y, f, twice(1.f));
  return __fmul2_rn(y, make_float2(__uint_as_float(__float_as_uint(t.x) * 8388608u + 0x3f800000u),
                                   __uint_as_float(__float_as_uint(t.y) * 8388608u + 0x3f800000u)));
}

// Sum of 2^(scale * s - m) over 32 columns, kPairs of its 16 pairs of exponentials by the polynomial. (The same columns of
// every 32 keys, so that equal key blocks have equal sums.)
template <int kPairs>
__device__ __forceinline__ float exp_sum(const uint32_t (&r)[32], float scale_log2, float m) {
  const float2 sc = make_float2(scale_log2, scale_log2);
  const float2 nm = make_float2(-m, -m);
  float2 a0 = make_float2(0.f, 0.f), a1 = make_float2(0.f, 0.f);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float2 x0 = __ffma2_rn(make_float2(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1])), sc, nm);
    const float2 x1 = __ffma2_rn(make_float2(__uint_as_float(r[4 * j + 2]), __uint_as_float(r[4 * j + 3])), sc, nm);
    const bool polynomial = (kPairs == 2 && j % 4 == 1) || (kPairs == 3 && (j == 1 || j == 4 || j == 6));   // spread evenly
    a0 = __fadd2_rn(a0, make_float2(fast_exp2(x0.x), fast_exp2(x0.y)));
    a1 = __fadd2_rn(a1, polynomial ? exp2_by_polynomial(x1) : make_float2(fast_exp2(x1.x), fast_exp2(x1.y)));
  }
  const float2 a = __fadd2_rn(a0, a1);
  return a.x + a.y;
}

template <int kMode>
__global__ void __launch_bounds__(kThreads, one_per_sm(kMode) ? 1 : 2)
score_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k, const ScoreParams p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  ScoreSmem<kMode>& sm = *reinterpret_cast<ScoreSmem<kMode>*>(smem_raw);
  constexpr int kTmemCols = tmem_cols(kMode);
  constexpr int kChunk = block_sums(kMode);
  constexpr bool kKeepsSums = kMode == kOnePass || one_per_sm(kMode);
  wait_for_previous_kernel();
  if ((smem_u32(smem_raw) & 1023u) != 0u) {
    if (threadIdx.x == 0 && atomicCAS(&p.status->code, 0, 2) == 0) p.status->where = 2;
    return;
  }
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  const int num_q_tiles = (p.seq_len + kTileM - 1) / kTileM;
  const int num_tiles = (p.seq_len + kTileN - 1) / kTileN;
  const int q_tile = blockIdx.x % num_q_tiles;
  const int bh = blockIdx.x / num_q_tiles;
  const int head = bh % p.heads_q;
  const int batch = bh / p.heads_q;
  const int kv_head = head / p.group;
  const int q_row0 = q_tile * kTileM;

  // Group g takes tiles 4i + 2g and 4i + 2g + 1. Its j-th tile is key tile tile_of(g, j); counted over both groups it is
  // number index_of(g, j) in the order in which tiles are loaded and multiplied: the groups alternate as long as both
  // have tiles left (group 0 has up to two more).
  const int tiles1 = (num_tiles >> 2) * 2 + max((num_tiles & 3) - 2, 0);
  const int tiles0 = num_tiles - tiles1;
  auto tile_of = [&](int g, int j) -> int { return (j >> 1) * 4 + 2 * g + (j & 1); };
  auto index_of = [&](int g, int j) -> int { return j < tiles1 ? 2 * j + g : tiles1 + j; };
  auto group_of = [&](int i) -> int { return i < 2 * tiles1 ? (i & 1) : 0; };
  auto step_of = [&](int i) -> int { return i < 2 * tiles1 ? (i >> 1) : i - tiles1; };   // j of number i

  // ---- set-up (the producer warp owns the barriers of its loads and starts them right away) -------
  if (warp == 8) {
    if (lane == 0) {
      mbar_init(&sm.q_full, 1);
      for (int s = 0; s < kSlots; ++s) mbar_init(&sm.k_full[s], 1);
      mbar_fence_init();
    }
    __syncwarp();
  }
  auto issue_k_load = [&](int i) {
    const int slot = i % kSlots;
    const int key0 = tile_of(group_of(i), step_of(i)) * kTileN;
    mbar_expect_tx(&sm.k_full[slot], kTileN * kHeadDim * 2);   // keys beyond the sequence arrive as zeros
    tma_load_4d(sm.k[slot][0], &tm_k, &sm.k_full[slot], 0, key0, kv_head, batch);
    tma_load_4d(sm.k[slot][1], &tm_k, &sm.k_full[slot], 64, key0, kv_head, batch);
  };
  if (warp == 8 && elect_one_sync()) {
    tma_prefetch_desc(&tm_q);
    tma_prefetch_desc(&tm_k);
    mbar_expect_tx(&sm.q_full, kTileM * kHeadDim * 2);
    tma_load_4d(sm.q[0], &tm_q, &sm.q_full, 0, q_row0, head, batch);
    tma_load_4d(sm.q[1], &tm_q, &sm.q_full, 64, q_row0, head, batch);
    for (int i = 0; i < min(num_tiles, kSlots); ++i) issue_k_load(i);
  }
  if (tid == 0) {
    for (int s = 0; s < kSlots; ++s) mbar_init(&sm.done[s], 1);
    for (int s = 0; s < 2; ++s) mbar_init(&sm.s_free[s], 4);
    sm.abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 9) {
    tmem_alloc(&sm.tmem_base, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem_base;

  if (warp == 8) {
    // =============================== TMA producer =======================================
    bool ok = true;
    for (int i = kSlots; ok && i < num_tiles; ++i) {
      ok = mbar_wait(&sm.done[i % kSlots], (i / kSlots - 1) & 1, &sm.abort_flag, p.status, 40);
      ok = __all_sync(0xffffffffu, ok);
      if (ok && elect_one_sync()) issue_k_load(i);
      __syncwarp();
    }
  } else if (warp == 9) {
    // =============================== UMMA issuer ========================================
    const uint32_t q_lo0 = umma_desc_lo(smem_u32(sm.q[0]), 16);
    const uint32_t k_lo0 = umma_desc_lo(smem_u32(sm.k[0][0]), 16);
    constexpr uint32_t slot_step = (2 * kTileN * 64 * 2) >> 4;   // 16 KB per ring slot
    bool ok = mbar_wait(&sm.q_full, 0, &sm.abort_flag, p.status, 50);
    ok = __all_sync(0xffffffffu, ok);
    for (int i = 0; ok && i < num_tiles; ++i) {
      const int slot = i % kSlots;
      const int g = group_of(i), j = step_of(i);
      ok = j == 0 ? mbar_wait(&sm.k_full[slot], (i / kSlots) & 1, &sm.abort_flag, p.status, 51)
                  : mbar_wait2(&sm.k_full[slot], (i / kSlots) & 1, &sm.s_free[g], (j - 1) & 1, &sm.abort_flag, p.status, 52);
      ok = __all_sync(0xffffffffu, ok);
      if (ok) issue_qk64(tmem + g * kTileN, q_lo0, k_lo0 + slot * slot_step, &sm.done[slot]);
    }
  } else {
    // =============================== exponentials, block sums, ranking ===================
    const int g = warp >> 2;              // group
    const int wq = warp & 3;              // 32-row quarter of the tile
    const int rit = tid & (kTileM - 1);   // row in tile
    const uint32_t lane_base = static_cast<uint32_t>(wq * 32) << 16;
    const uint32_t t_stat = tmem + kColStat + lane_base;
    const float scale_log2 = p.scale_log2;
    const int row = q_row0 + rit;
    const bool row_valid = row < p.seq_len;
    const int bs = p.block_size;
    const int bs_shift = 31 - __clz(bs);   // (a division per tile took 3-12 % of the kernel's time)
    const int nb = kMode == kRowStats ? 0 : p.seq_len / bs;
    const int rows_here = kTileM / bs;                       // block-rows of A' in this tile: 1, 2 or 4
    const bool rank_here = kMode != kRowStats && p.row_ptr != nullptr;
    const float inv_area = 1.f / (static_cast<float>(bs) * static_cast<float>(bs));
    float m = -INFINITY;   // reference of this row in this group (base-2 logits)
    float l = 0.f;         // sum of 2^(s - m)
    float carry = 0.f;     // 128-key blocks: sum over the block's first 64 keys
    if constexpr (kMode == kPooled) {
      // natural-log LSE -> base-2 reference: 2^(s - m) is the probability
      m = row_valid ? p.lse[static_cast<int64_t>(bh) * p.seq_len + row] * 1.44269504088896341f : INFINITY;
    }

    // this row's sum over key block jb0 + col
    auto put_sum = [&](int col, float v) {
      if (smem_sums(kMode) == 0 || col < tmem_sums(kMode)) {
        tmem_st1(t_stat + col, v);
      } else {
        sm.more[col - tmem_sums(kMode)][rit] = v;
      }
    };
    // Block sums held in tensor memory (columns of key blocks [jb0, jb0 + n)) times the row's weight (both factors) in the
    // group that summed them, then summed over the rows of each query block: A' to memory and / or to the ranking keys. All
    // eight warps, in step.
    auto fold = [&](int jb0, int n, PowerOfTwo w0, PowerOfTwo w1) {
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      tc_fence_before();
      named_barrier_sync(1, 2 * kTileM);
      tc_fence_after();
      for (int c = 32 * g; c < n; c += 64) {
        uint32_t r[32];
        float v[32];
        if (smem_sums(kMode) == 0 || c < tmem_sums(kMode)) {
          tmem_ld32(t_stat + c, r);
          tmem_wait_ld();
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(sm.more[c + j - tmem_sums(kMode)][rit]);
        }
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const bool second = (((c + j) * bs) & 128) != 0;
          v[j] = __uint_as_float(r[j]) * (second ? w1.far : w0.far) * (second ? w1.near : w0.near);
        }
        sm.quarter[wq][c + lane] = warp_column_sums(v, lane);   // columns at and beyond n are not used below
      }
      tc_fence_before();
      named_barrier_sync(1, 2 * kTileM);
      tc_fence_after();
      for (int c = tid; c < n; c += 2 * kTileM) {
        const float q0 = sm.quarter[0][c], q1 = sm.quarter[1][c], q2 = sm.quarter[2][c], q3 = sm.quarter[3][c];
        float score[4] = {q0, q1, q2, q3};
        if (bs == 128) score[0] = (q0 + q1) + (q2 + q3);
        if (bs == 64) {
          score[0] = q0 + q1;
          score[1] = q2 + q3;
        }
        const int jb = jb0 + c;
#pragma unroll
        for (int rh = 0; rh < 4; ++rh) {
          const int ib = q_tile * rows_here + rh;
          if (rh < rows_here && ib < nb) {
            const float a = score[rh] * inv_area;
            if (p.scores != nullptr) p.scores[(static_cast<int64_t>(bh) * nb + ib) * nb + jb] = a;
            if (rank_here) sm.keys[rh * nb + jb] = ordered_key(a);
          }
        }
      }
    };

    bool ok = true;
    int jb0 = 0;   // key block of column 0
    const int my_tiles = g == 0 ? tiles0 : tiles1;
    if constexpr (kKeepsSums) {
      // the common reference: the maximum over the first tile of either group (which the loop below copies once more)
      float mx = -INFINITY;
      if (my_tiles > 0) {
        ok = mbar_wait(&sm.done[index_of(g, 0)], 0, &sm.abort_flag, p.status, 61);
        ok = __all_sync(0xffffffffu, ok);
        tc_fence_after();
        uint32_t r0[32], r1[32];
        tmem_ld32(tmem + g * kTileN + lane_base, r0);
        tmem_ld32(tmem + g * kTileN + lane_base + 32, r1);
        tmem_wait_ld();
        const int valid_cols = p.seq_len - tile_of(g, 0) * kTileN;
        if (valid_cols < kTileN) mask_columns_from(r0, r1, valid_cols);
#pragma unroll
        for (int c = 0; c < 32; ++c) mx = fmaxf(mx, fmaxf(__uint_as_float(r0[c]), __uint_as_float(r1[c])));
      }
      sm.first_max[g][rit] = mx;
      named_barrier_sync(1, 2 * kTileM);
      m = fmaxf(mx, sm.first_max[g ^ 1][rit]) * scale_log2;
    }
    for (int j = 0; j < my_tiles; ++j) {
      const int i = index_of(g, j);
      const int t = tile_of(g, j);
      // (after a wait has run out the remaining tiles are walked without waiting, so that all eight warps still meet in
      // the same barriers; what they hold is not ranked)
      ok = ok && mbar_wait(&sm.done[i % kSlots], (i / kSlots) & 1, &sm.abort_flag, p.status, 60);
      ok = __all_sync(0xffffffffu, ok);
      tc_fence_after();
      uint32_t r0[32], r1[32];
      const uint32_t tS = tmem + g * kTileN + lane_base;
      tmem_ld32(tS, r0);
      tmem_ld32(tS + 32, r1);
      tmem_wait_ld();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.s_free[g]);
      const int valid_cols = p.seq_len - t * kTileN;   // ragged tail of the sequence
      if (valid_cols < kTileN) mask_columns_from(r0, r1, valid_cols);
      float s0 = exp_sum<poly_pairs(kMode)>(r0, scale_log2, m);
      float s1 = exp_sum<poly_pairs(kMode)>(r1, scale_log2, m);
      if constexpr (kMode != kPooled) {
        const bool outgrown = !(s0 + s1 <= kOutgrown);   // no reference yet (m = -inf), far larger logits, or NaN
        if (__any_sync(0xffffffffu, outgrown)) {
          // take the tile's own maximum as the reference and bring everything summed so far to it
          float mx = -INFINITY;
#pragma unroll
          for (int c = 0; c < 32; ++c) mx = fmaxf(mx, fmaxf(__uint_as_float(r0[c]), __uint_as_float(r1[c])));
          const float m_new = outgrown ? fmaxf(m, mx * scale_log2) : m;
          const PowerOfTwo alpha = power_of_two(m_new > m ? m - m_new : 0.f);
          m = m_new;
          l *= alpha.far * alpha.near;
          // a row whose logits so far are all -inf: 2^(-inf - 0) = 0, not NaN
          const float ref = m == -INFINITY ? 0.f : m;
          s0 = exp_sum<poly_pairs(kMode)>(r0, scale_log2, ref);
          s1 = exp_sum<poly_pairs(kMode)>(r1, scale_log2, ref);
          if constexpr (kKeepsSums) {
            carry = carry * alpha.far * alpha.near;
            // (columns of the other group are left alone; its threads rescale theirs)
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            const int per_span = 128 / bs;
            for (int s = g; s <= (t >> 1); s += 2)
              for (int c = s * per_span; c < (s + 1) * per_span; ++c) {
                if (smem_sums(kMode) == 0 || c < tmem_sums(kMode)) {
                  uint32_t r;
                  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(t_stat + c) : "memory");
                  tmem_wait_ld();
                  tmem_st1(t_stat + c, __uint_as_float(r) * alpha.far * alpha.near);
                } else {
                  float& sum = sm.more[c - tmem_sums(kMode)][rit];
                  sum = sum * alpha.far * alpha.near;
                }
              }
            // the loop also writes the columns that this tile is about to fill, unread: those stores come first. (Leaving
            // those columns out instead takes 1 % longer: 32 x 4096, block 32, 206.4 against 210.2 us.)
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
          }
        }
        l += s0 + s1;
      }
      if constexpr (kMode != kRowStats) {
        const int col = ((t * kTileN) >> bs_shift) - jb0;   // first block of the tile
        if (bs == 128) {
          if ((t & 1) == 0) {
            carry = s0 + s1;
          } else {
            put_sum(col, carry + (s0 + s1));
          }
        } else if (bs == 64) {
          put_sum(col, s0 + s1);
        } else {
          put_sum(col, s0);
          put_sum(col + 1, s1);   // (beyond the last block if their number is odd: not folded)
        }
        if constexpr (kMode == kPooled) {
          // 128 blocks are bs spans of 128 keys: bs / 2 spans, bs tiles of each group
          if (((j + 1) & (bs - 1)) == 0) {
            fold(jb0, min(kChunk, nb - jb0), {1.f, 1.f}, {1.f, 1.f});
            jb0 += kChunk;
          }
        }
      }
    }
    if (*reinterpret_cast<volatile int*>(&sm.abort_flag) != 0) ok = false;
    // the two groups' references and denominators of a row meet
    PowerOfTwo w0 = {1.f, 1.f}, w1 = {1.f, 1.f};
    if constexpr (kMode != kPooled) {
      sm.ml[g][rit] = make_float2(m, l);
      named_barrier_sync(1, 2 * kTileM);
      const float2 a = sm.ml[0][rit], b = sm.ml[1][rit];
      const float top = fmaxf(a.x, b.x);
      const PowerOfTwo f0 = power_of_two(a.x - top), f1 = power_of_two(b.x - top);
      const float denom = a.y * f0.far * f0.near + b.y * f1.far * f1.near;
      if constexpr (kMode == kRowStats) {
        if (ok && g == 0 && row_valid)
          p.lse_out[static_cast<int64_t>(bh) * p.seq_len + row] = (top + log2f(denom)) * 0.69314718055994531f;
      }
      w0 = {f0.far, row_valid ? f0.near / denom : 0.f};
      w1 = {f1.far, row_valid ? f1.near / denom : 0.f};
    }
    if constexpr (kMode != kRowStats) {
      if (nb > jb0) fold(jb0, min(kChunk, nb - jb0), w0, w1);
      named_barrier_sync(1, 2 * kTileM);   // the ranking keys are complete
      if (ok && rank_here && warp < rows_here) {
        // one warp per block-row: isolated top-k (Eq. 5 / Eq. 6) and the CSR list
        const int ib = q_tile * rows_here + warp;
        if (ib < nb) {
          const int k_total = p.k_pre + p.k_gen;
          const int64_t r = static_cast<int64_t>(bh) * nb + ib;
          warp_select_row(sm.keys + warp * nb, nb, p.pb, p.k_pre, p.k_gen, sm.hist[warp], p.col_idx + r * k_total, lane);
          if (lane == 0) {
            p.row_ptr[r] = static_cast<int32_t>(r * k_total);
            if (r == static_cast<int64_t>(gridDim.x / num_q_tiles) * nb - 1)
              p.row_ptr[r + 1] = static_cast<int32_t>((r + 1) * k_total);
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 9) {
    __syncwarp();
    tmem_dealloc(tmem, kTmemCols);
  }
}

template <int kMode>
cudaError_t launch(const CUtensorMap& tq, const CUtensorMap& tk, const ScoreParams& p, int batch, cudaStream_t stream) {
  auto kernel = score_kernel<kMode>;
  static_assert(sizeof(ScoreSmem<kMode>) <= (kMode == kOnePassMost ? 227 : kMode == kOnePassWide ? 120 : 113) * 1024,
                "two CTAs per SM, or one");
  // (one per SM: more than half of its shared memory, so that two CTAs never compete for its tensor memory)
  const int smem = kMode == kOnePassWide ? 120 * 1024 : static_cast<int>(sizeof(ScoreSmem<kMode>));
  static SmemLimit limit;  // per template instantiation
  cudaError_t e = ensure_dynamic_smem(kernel, smem, limit);
  if (e != cudaSuccess) return e;
  const int num_q_tiles = (p.seq_len + kTileM - 1) / kTileM;
  const long long ctas = static_cast<long long>(batch) * p.heads_q * num_q_tiles;
  if (ctas <= 0) return cudaSuccess;
  return launch_overlapped(kernel, ctas, one_per_sm(kMode) ? p.max_ctas / 2 : p.max_ctas, kThreads, smem, stream, tq, tk, p);
}

}  // namespace

bool score_ranks_in_kernel(int nb, int block_size) { return nb * (kTileM / block_size) <= kMaxKeys; }
bool score_in_one_pass(int nb) { return nb <= block_sums(kOnePassMost); }

cudaError_t launch_row_stats(const CUtensorMap& tq, const CUtensorMap& tk, const ScoreParams& p, int batch,
                             cudaStream_t stream) {
  return launch<kRowStats>(tq, tk, p, batch, stream);
}

cudaError_t launch_pooled_scores(const CUtensorMap& tq, const CUtensorMap& tk, const ScoreParams& p, int batch,
                                 cudaStream_t stream) {
  if (p.lse != nullptr) return launch<kPooled>(tq, tk, p, batch, stream);
  const int nb = p.seq_len / p.block_size;
  if (nb <= block_sums(kOnePass)) return launch<kOnePass>(tq, tk, p, batch, stream);
  if (nb <= block_sums(kOnePassWide)) return launch<kOnePassWide>(tq, tk, p, batch, stream);
  return launch<kOnePassMost>(tq, tk, p, batch, stream);
}

}  // namespace sparsed
