// The rules by which an attention call goes to one of the kernels that can do it. Host arithmetic only.
#pragma once

namespace sparsed {

// Whether the last wave of `clusters` clusters over `pairs` SM pairs runs as clusters of one stream each. Such a
// cluster takes 0.65-0.8 of the time of one with two. So a last wave that would leave half of the SM pairs idle or
// more is launched that way: 16 x 3072 (1.3 waves) 95.0 -> 84.4 us (statistics recorded). So is a grid of less than half
// a wave, but only those of fewer than 256 keys come here (choose_dense_kernel). From two full waves on it gained nothing
// (32 x 4096, 3.46 waves): there the launch is at the power limit, and an emptier last wave raises the clock (1755 MHz
// against 1687 at 37 x 4096, 4.0 waves), which leaves 5 % of its cost (979 against 1029 TFLOP/s).
inline bool dense_pair_splits(long long clusters, long long pairs) {
  const long long last = pairs > 0 ? clusters % pairs : 0;
  return last != 0 && 2 * last <= pairs && clusters < 2 * pairs;
}

// Time of `units` equal pieces of work on `slots`, in full waves. The last wave counts as 0.65 if it is at most half
// full and its half-empty SMs run faster (two CTAs per SM, or split clusters), else as 0.5 and half its share (the
// SMs that are busy have the power of the others).
inline double dense_waves(long long units, long long slots, bool half_wave) {
  const long long last = units % slots;
  const double whole = static_cast<double>(units / slots);
  if (last == 0) return whole;
  const double share = static_cast<double>(last) / static_cast<double>(slots);
  return whole + (half_wave && 2 * last <= slots ? 0.65 : 0.5 + 0.5 * share);
}

// Whether the kernel whose MMAs span CTA pairs (attention_dense_pair.cu) takes a plain pass over bh heads of all batch
// entries that lone_ctas_pay has not taken; the single-CTA kernel (attention.cu) takes the others. Both give the same bits. max_ctas: CTAs of the latter
// that fit on the device at once, two per SM.
//
// Per query row the pair kernel takes 3-7 % less under sustained load, which is bound by power (it fetches each K/V
// tile once for 512 rows instead of once for 128): 32 heads x 8192 956 -> 928 us, 8 x 32 x 4096 1990 -> 1915, 32 x
// 16384 3720 -> 3495. Launches too short to reach the power limit, or with rests between them, gain nothing from
// that, and the longer set-up and tear-down of a cluster costs them 2-8 % (20 launches after a rest: 8 heads x 4096
// 60.0 against 64.3 us, 20 heads 172 against 179). So the pair kernel runs where it was no slower either way:
//   * where the last wave runs as clusters of one stream each: its SMs would be half empty in both kernels (6 x 8192 217 ->
//     198 us, 3 x 16384 417 -> 374; where that is the only wave there is at most one query tile per SM, and lone_ctas_pay
//     has taken the call);
//   * from 2^29 logits on (32 heads x 4096, 8 x 8192), which take 200 us. With fewer, 12 heads x 6144 lose 1 % after
//     a rest, and 5 heads x 4096 9 % even under sustained load: 40 clusters leave 68 SMs empty, 160 CTAs
//     none.
// A wave of either is the same number of rows, but the last one may be emptier: 8 heads x 14000 are 3.03 waves of
// clusters (740 us) and 2.97 of single CTAs (690). So the waves are counted as well.
inline bool dense_pair_pays(long long bh, int seq_len, int max_ctas) {
  if (seq_len < 4096 || max_ctas < 4) return false;
  const long long tiles = (static_cast<long long>(seq_len) + 127) / 128;
  const long long clusters = bh * ((tiles + 3) / 4), pairs = max_ctas / 4;
  const bool split = dense_pair_splits(clusters, pairs);
  const double logits = static_cast<double>(bh) * seq_len * seq_len;
  if (!split && logits < static_cast<double>(1 << 29)) return false;
  return 0.965 * dense_waves(clusters, pairs, split) < dense_waves(bh * tiles, max_ctas, true);
}

// Whether attention on `items` query tiles over `keys` keys to a row goes to the kernel whose CTAs have an SM each
// (attention_lone.cu), before the choice above is asked. It gives the same bits as the others. Up to one item per SM it
// was the fastest (us, 20 calls in a row): dense from four tiles of 64 keys on, against the single-CTA kernel 2 heads x
// 256 6.95 -> 6.36, 2 x 320 7.61 -> 6.68, 2 x 1024 14.8 -> 11.9, 8 x 2304 (144 items) 29.1 -> 23.4, and against split
// clusters 2 x 4096 44.0 -> 35.8, 2 x 9400 102 -> 77.5; switch steps 2 x 256 12.1 -> 10.7, 2 x 1024 18.9 -> 15.8, 8 x 2304
// 43.1 -> 28.5, 2 x 8192 88.8 -> 78.4. With fewer keys its longer set-up shows: 2 x 100 5.1 -> 5.9. Beyond one item per SM
// its items come one after the other, set-up and all: 32 x 1900 58 -> 77.
//
// That is for a call alone. Calls side by side on several streams lose by it once all their items together are more than
// the SMs, where two CTAs of the other kernels share one. A plain call's rule cannot see its neighbours; the line lies
// where a pair of equal calls loses about as much as a call alone gains. Dense, alone | a pair (time over that of the
// single-CTA kernel): 100 items x 256 keys 0.96 | 1.05, x 768 0.87 | 0.97; 128 x 512 0.90 | 1.14, 148 x 256 0.95 | 1.36,
// x 512 0.87 | 1.30; 128 x 1024 0.84 | 1.09, 144 x 1024 0.82 | 1.17, x 2048 0.75 | 1.11, 128 x 4096 0.87 | 1.01. So beyond
// two thirds of the SMs it takes 1024 keys. (Three calls of 64 items: x 1024 keys 0.87; four: 1.10.) Switch steps gain
// either way, their other kernel takes two SMs to a cluster: 144 x 1024 0.85 | 0.82.
inline bool lone_ctas_pay(bool with_stats, long long items, long long keys, int max_ctas) {
  const long long sms = max_ctas / 2;
  return items <= sms && keys >= (with_stats || 3 * items <= 2 * sms ? 256 : 1024);
}

enum class DenseKernel { kSingle, kPair, kLone };

// Dense attention over bh heads of all batch entries. The single-CTA kernel records no row statistics.
inline DenseKernel choose_dense_kernel(bool with_stats, long long bh, int seq_len, int max_ctas) {
  const long long items = bh * ((static_cast<long long>(seq_len) + 127) / 128);
  if (lone_ctas_pay(with_stats, items, seq_len, max_ctas)) return DenseKernel::kLone;
  return with_stats || dense_pair_pays(bh, seq_len, max_ctas) ? DenseKernel::kPair : DenseKernel::kSingle;
}

// lone_ctas_pay for block-sparse attention. Alone, the lists may be of any length: 2 heads x 1024 block 128, one block a row
// 5.85 -> 5.56, six 12.3 -> 10.5; 16 x 512 block 32 (walked as the union of four rows' lists) one 7.72 -> 7.15, ten 11.9
// -> 10.4; 2 x 4096 block 32, twelve 21.8 -> 16.3; no blocks at all, 8 x 1024 block 32, 4.2 -> 3.7; one whole row among
// rows of one block, 2 x 8192 block 64, 91 -> 71. Side by side (alone | a pair): block 128, 72 items x 128 keys 0.98 | 0.98,
// 80 x 256 0.95 | 1.09, x 512 0.93 | 1.05, 128 x 1024 0.86 | 1.18, x 2048 0.82 | 1.13, 148 x 2048 0.81 | 1.25, x 3072 0.79 |
// 1.17; block 64 and 32, whose unions are longer than the lists, 100 x 128 0.90 | 1.10, 128 x 256 0.88 | 1.18 and 0.84 |
// 1.09, 144 x 512 0.82 | 1.14 and 0.83 | 1.12. keys: on average in the `rows` lists, as far as `nnz` (all entries) says;
// 0 if it does not.
inline bool sparse_lone_ctas_pay(long long items, long long nnz, long long rows, int num_blocks, int block_size,
                                 int max_ctas) {
  const long long sms = max_ctas / 2;
  if (items > sms || rows < 1) return false;
  if (nnz < 0) nnz = 0;
  if (nnz > rows * num_blocks) nnz = rows * num_blocks;   // (room rather than entries)
  const long long keys = nnz * block_size / rows;
  const bool packed = block_size < 128;
  if (2 * items <= sms) return true;
  return keys >= (3 * items <= 2 * sms ? (packed ? 0 : 512) : (packed ? 512 : 2048));
}

}  // namespace sparsed
