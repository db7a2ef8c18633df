// Pattern selection from the row statistics of the switch step's full-attention pass
// ("Isolated Selection": A' = avgpool(A, block_size), then Eq. 5 / Eq. 6), without a second
// Q K^T pass.
//
// The dense attention kernel can record, for every query row i and every group g of block_size
// keys, v[g][i] = log2 sum_{j in g} 2^(s_ij), the group's share of the row's softmax denominator.
// With the row's final log-sum-exp, 2^(v[g][i] - LSE_i) is exactly the probability mass row i
// puts on key block g, so A'[ib][jb] is the sum of that mass over the rows of query block ib,
// divided by block_size^2.
//
// One CTA owns one 128-row query tile of one (batch, head), i.e. one, two or four query blocks. Its statistics are one
// contiguous run (layout [bh][128-row query tile][key block][row]), read by four warps that go their own ways: a warp takes
// eight key blocks at a time, lane l of it rows 4l .. 4l + 3 of each in one 16-byte load, and asks for the next eight as
// soon as it has taken the exponentials of these. A lane's four rows are added up, then the eight lanes of a 32-row
// quarter by a butterfly that leaves each lane with one key block of the eight (seven shuffles for all; a fixed tree, the
// same for every key block: bitwise reproducible). The quarters are then combined into the CTA's block-row(s) of A',
// which are optionally written out, and one warp per block-row ranks it (warp_select_row) and writes the CSR list.
// HBM-bound: 4 * 128 * ceil(L/128) * (L / block_size) bytes read per (batch, head).
//
// Seven CTAs per SM are the most whose registers do not spill. 32 heads, block 128: 65536 tokens 776 -> 643 us (4.3 GB: 6.7
// TB/s), 16384 (28 heads) 60 -> 52, 8192 27.7 -> 22; block 32, 4096 tokens 28 -> 23 - before, the exponentials went through
// shared memory, 32 key blocks at a time with two barriers each, to be added up by one lane per key block, six CTAs per SM.
// (With two batches of loads in flight, five CTAs: 8 heads x 65536 196 us against 187; six or eight CTAs 193, 189. What is
// left at 8192 is one CTA's own chain, 6 us from its first load to its ranked row.)
#include "internal.h"
#include "topk_device.cuh"

namespace sparsed {
namespace {

constexpr int kRows = 128;
constexpr int kCtasPerSm = 7;
constexpr int kBatch = 8;           // key blocks a warp takes at a time: 16-byte loads each thread has in flight
constexpr int kMaxBlocks = 2048;    // key blocks per row: seq_len <= 2048 * block_size

// Floats between the quarters' sums of one key block: four quarters of eight key blocks then lie in 32 different banks.
__host__ __device__ constexpr int quarter_pitch(int nb) { return (nb + 31) / 32 * 32 + 8; }

// Shared memory (dynamic, sized for the actual sequence): the per-block mass of each 32-row quarter of the query tile, the
// ordered keys of this CTA's block-row(s), one top-k histogram per block-row.
struct PoolSmem {
  float* quarter_sum;               // [32-row quarter][key block]
  uint32_t* keys;                   // [block-row of this CTA][key block]
  int* hist;                        // [block-row][256]
};

__host__ __device__ inline size_t pool_smem_bytes(int nb, int rows_here) {
  return sizeof(float) * 4 * quarter_pitch(nb) + sizeof(uint32_t) * rows_here * nb + sizeof(int) * 256 * rows_here;
}

__global__ void __launch_bounds__(kRows, kCtasPerSm) pool_select_kernel(const PoolParams p) {
  extern __shared__ __align__(16) uint8_t pool_smem_raw[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int L = p.seq_len;
  const int bs = p.block_size;
  const int nb = L / bs;                    // key blocks per row = statistics per row
  const int rows_here = kRows / bs;         // block-rows of A' this CTA produces: 1, 2 or 4
  const int pitch = quarter_pitch(nb);
  PoolSmem sm;
  {
    float* f = reinterpret_cast<float*>(pool_smem_raw);
    sm.quarter_sum = f;
    f += 4 * pitch;
    sm.keys = reinterpret_cast<uint32_t*>(f);
    sm.hist = reinterpret_cast<int*>(sm.keys + rows_here * nb);
  }
  const int num_q_tiles = (L + kRows - 1) / kRows;
  const int q_tile = blockIdx.x % num_q_tiles;
  const int bh = blockIdx.x / num_q_tiles;
  // Lane l owns rows 4l..4l+3 of the query tile. seq_len is a multiple of 32 here, so a group of four rows is valid or
  // invalid as a whole and 16-byte aligned.
  const int row4 = q_tile * kRows + lane * 4;
  const bool rows_valid = row4 < L;
  float4 lse2 = make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
  if (rows_valid) {
    const float4 t = *reinterpret_cast<const float4*>(p.lse + static_cast<int64_t>(bh) * L + row4);
    const float c = 1.44269504088896341f;
    lse2 = make_float4(t.x * c, t.y * c, t.z * c, t.w * c);
  }
  // statistics layout [bh][query tile][key block][128 rows]: this CTA's share is one contiguous run
  const float* src = p.tile_lse + (static_cast<int64_t>(bh) * num_q_tiles + q_tile) * nb * kRows + lane * 4;

  auto load = [&](float4 (&v)[kBatch], int jb0) {
#pragma unroll
    for (int u = 0; u < kBatch; ++u)
      v[u] = (rows_valid && jb0 + u < nb) ? __ldcs(reinterpret_cast<const float4*>(src + static_cast<int64_t>(jb0 + u) * kRows))
                                          : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
  };
  constexpr int kStep = 4 * kBatch;   // of the four warps together
  float4 v[kBatch];
  load(v, warp * kBatch);
  for (int jb0 = warp * kBatch; jb0 < nb; jb0 += kStep) {
    // this lane's four rows' mass on the key blocks [jb0, jb0 + 8)
    float m[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u)
      m[u] = (fast_exp2(v[u].x - lse2.x) + fast_exp2(v[u].y - lse2.y)) +
             (fast_exp2(v[u].z - lse2.z) + fast_exp2(v[u].w - lse2.w));
    load(v, jb0 + kStep);
    // ... the quarter's: eight lanes', key block jb0 + (lane & 7) left in each
#pragma unroll
    for (int half = kBatch / 2; half > 0; half >>= 1) {
      const bool upper = (lane & half) != 0;
#pragma unroll
      for (int u = 0; u < half; ++u) {
        const float keep = upper ? m[u + half] : m[u];
        const float give = upper ? m[u] : m[u + half];
        m[u] = keep + __shfl_xor_sync(0xffffffffu, give, half);
      }
    }
    const int jb = jb0 + (lane & 7);
    if (jb < nb) sm.quarter_sum[(lane >> 3) * pitch + jb] = m[0];
  }
  __syncthreads();

  const float inv_area = 1.f / (static_cast<float>(bs) * static_cast<float>(bs));
  for (int jb = tid; jb < nb; jb += kRows) {
    const float q0 = sm.quarter_sum[jb], q1 = sm.quarter_sum[pitch + jb], q2 = sm.quarter_sum[2 * pitch + jb],
                q3 = sm.quarter_sum[3 * pitch + jb];
    float score[4];
    if (bs == 128) {
      score[0] = ((q0 + q1) + (q2 + q3)) * inv_area;
    } else if (bs == 64) {
      score[0] = (q0 + q1) * inv_area;
      score[1] = (q2 + q3) * inv_area;
    } else {
      score[0] = q0 * inv_area;
      score[1] = q1 * inv_area;
      score[2] = q2 * inv_area;
      score[3] = q3 * inv_area;
    }
#pragma unroll
    for (int rh = 0; rh < 4; ++rh) {
      const int ib = q_tile * rows_here + rh;
      if (rh < rows_here && ib < nb) {
        sm.keys[rh * nb + jb] = ordered_key(score[rh]);
        if (p.scores != nullptr) p.scores[(static_cast<int64_t>(bh) * nb + ib) * nb + jb] = score[rh];
      }
    }
  }
  __syncthreads();
  // one warp per block-row: isolated top-k (Eq. 5 / Eq. 6) and the CSR list
  if (warp < rows_here) {
    const int ib = q_tile * rows_here + warp;
    if (ib < nb) {
      const int k_total = p.k_pre + p.k_gen;
      const int64_t r = static_cast<int64_t>(bh) * nb + ib;
      warp_select_row(sm.keys + warp * nb, nb, p.pb, p.k_pre, p.k_gen, sm.hist + warp * 256, p.col_idx + r * k_total, lane);
      if (lane == 0) {
        p.row_ptr[r] = static_cast<int32_t>(r * k_total);
        if (r == static_cast<int64_t>(p.bh) * nb - 1) p.row_ptr[r + 1] = static_cast<int32_t>((r + 1) * k_total);
      }
    }
  }
}

}  // namespace

int pool_select_max_blocks() { return kMaxBlocks; }

cudaError_t launch_pool_select(const PoolParams& p, cudaStream_t stream) {
  const int nb = p.seq_len / p.block_size;
  if (nb > kMaxBlocks) return cudaErrorInvalidValue;
  const int smem = static_cast<int>(pool_smem_bytes(nb, kRows / p.block_size));
  static SmemLimit limit;
  cudaError_t e = ensure_dynamic_smem(pool_select_kernel, smem, limit);
  if (e != cudaSuccess) return e;
  const int num_q_tiles = (p.seq_len + kRows - 1) / kRows;
  const long long ctas = static_cast<long long>(p.bh) * num_q_tiles;
  if (ctas <= 0) return cudaSuccess;
  pool_select_kernel<<<static_cast<unsigned>(ctas), kRows, smem, stream>>>(p);
  return cudaGetLastError();
}

}  // namespace sparsed
