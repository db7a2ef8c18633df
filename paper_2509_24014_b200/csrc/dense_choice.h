// The rule by which plain dense attention goes to one of its two kernels. Host arithmetic only.
#pragma once

namespace sparsed {

// Whether the last wave of `clusters` clusters over `pairs` SM pairs runs as clusters of one stream each. Such a
// cluster takes 0.65-0.8 of the time of one with two. So a last wave that would leave half of the SM pairs idle or
// more is launched that way: 16 x 3072 (1.3 waves) 95.0 -> 84.4 us (statistics recorded); so is a grid of less than half
// a wave, of which only the shortest sequences still come here (lone_ctas_pay below). From two full waves on the launch runs into the power
// limit, which an emptier last wave only relieves (32 x 4096, 3.46 waves: no gain).
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
// entries; the single-CTA kernel (attention.cu) takes the others. Both give the same bits. max_ctas: CTAs of the latter
// that fit on the device at once, two per SM.
//
// Per query row the pair kernel takes 3-7 % less under sustained load, which is bound by power (it fetches each K/V
// tile once for 512 rows instead of once for 128): 32 heads x 8192 956 -> 928 us, 8 x 32 x 4096 1990 -> 1915, 32 x
// 16384 3720 -> 3495. Launches too short to reach the power limit, or with rests between them, gain nothing from
// that, and the longer set-up and tear-down of a cluster costs them 2-8 % (20 launches after a rest: 8 heads x 4096
// 60.0 against 64.3 us, 20 heads 172 against 179). So the pair kernel runs where it was no slower either way:
//   * where the last wave, or the only one, runs as clusters of one stream each: its SMs would be half empty in both
//     kernels (6 x 8192 217 -> 198 us, 3 x 16384 417 -> 374; an only wave that is split is up to one query tile per SM, and
//     goes to a third kernel first, see below);
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
inline bool lone_ctas_pay(long long items, long long keys, int max_ctas) {
  return items <= max_ctas / 2 && keys >= 256;
}

// The same for block-sparse attention, where the lists may be of any length: 2 heads x 1024 block 128, one block a row
// 5.85 -> 5.56, six 12.3 -> 10.5; 16 x 512 block 32 (walked as the union of four rows' lists) one 7.72 -> 7.15, ten 11.9
// -> 10.4; 2 x 4096 block 32, twelve 21.8 -> 16.3; no blocks at all, 8 x 1024 block 32, 4.2 -> 3.7; one whole row among
// rows of one block, 2 x 8192 block 64, 91 -> 71.
inline bool sparse_lone_ctas_pay(long long items, int max_ctas) { return items <= max_ctas / 2; }

}  // namespace sparsed
