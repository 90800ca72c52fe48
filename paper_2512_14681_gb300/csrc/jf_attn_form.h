// Launch form of the split-KV attention (host side; no CUDA types, so that the rule compiles and is
// tested on the host alone).
//
// A unit (chain, KV head, tile of up to 128 query rows) has 8 key lanes, spread over 8, 4, 2 or 1 CTAs (one
// cluster; one CTA per SM). max_clusters[i] clusters of 2^i CTAs are resident at once (152, 76, 36, 15
// on a GB300). Wide clusters shorten a unit, narrow ones fit more units at once and fold less through
// memory. Every form computes the same lane states and folds them in the same order, so the choice
// affects time only.
#pragma once

namespace jf {

// Units of a forward of M rows spread evenly over `chains` chains (exact for equal chains, e.g.
// B sequences with one n-row window each), capped by the launch's upper bound.
inline int attn_units_estimate(int M, int chains, int units_bound, int Hkv, int G, int q_rows_per_tile) {
  const int cb = chains > 0 ? chains : 1;
  const long long rows_per_chain = (M + cb - 1) / cb;
  const long long tiles = (rows_per_chain * G + q_rows_per_tile - 1) / q_rows_per_tile;
  const long long est = (long long)Hkv * cb * tiles;
  return est < units_bound ? (int)est : units_bound;
}

// Waves of `units` units with `at_once` of them resident at a time (none known: one).
inline int attn_waves(int units, int at_once) {
  const int n = at_once > 0 ? at_once : 1;
  return (units + n - 1) / n;
}

// CTAs per unit: the widest clusters that need no more waves than the next narrower ones. Past one wave
// of single CTAs, pairs when their waves (half as long, plus about an eighth of a single CTA's for the
// prologue and the fold) are the shorter. One 7B layer (4 KV heads, 7 query heads each), us with
// 8 / 4 / 2 / 1 CTAs per unit: 8 units at P = 4096 116 / 122 / 134 / 146; 16 units 131 / 128 / 140 / 150;
// 36 units at 2048 168 / 149 / 158 / 158; 56 units at 4096 220 / 205 / 198 / 204; 112 units 373 / 343 /
// 331 / 309.
inline int attn_ctas_per_unit(int units, const int (&max_clusters)[4]) {
  for (int i = 3; i > 0; --i)
    if (attn_waves(units, max_clusters[i]) <= attn_waves(units, max_clusters[i - 1])) return 1 << i;
  return attn_waves(units, max_clusters[1]) * 5 < attn_waves(units, max_clusters[0]) * 9 ? 2 : 1;
}

}  // namespace jf
