// How the keys of a slice are cut for the f32 attention: host code, apart so that it compiles without CUDA.
#pragma once

namespace scalekv {
namespace f32 {

constexpr int kMaxSplit = 8;                                // CTAs that may share a slice's keys (portable cluster size)

// CTAs that share a slice's keys.  ctas: CTAs of an unsplit launch.  In steps of a key tile: a CTA that has its SM to itself takes 1 per
// tile, two that share one 1.35 each.  (The CTAs of a recorded window, one per key tile and slice, are not counted: they hold an SM for about a tile's
// time, and with them counted as others the split at mid sizes would be smaller.  Not measured.)
// Combining costs 1.5; 0.8 for slices of two tiles, which gain by a split wherever two CTAs for one find an SM each (64 queries behind 57
// entries, 4 / 16 / 32 / 64 / 73 slices, us per launch, one CTA -> two: 10.4 / 10.6 / 10.6 / 10.6 / 10.8 -> 8.7 / 9.0 / 9.0 / 9.7 / 9.9) and at
// 1.5 had none.  0.8 would cut longer slices into more pieces as well, where nobody has measured it (3 tiles and 50 CTAs, 8 and 300, 14 and 740).
inline int key_split(int ctas, int tiles, int n_sm) {
  const float join = tiles == 2 ? 0.8f : 1.5f;
  auto cost = [&](int c) {
    const int n = ctas * c, per = (tiles + c - 1) / c, waves = (n + 2 * n_sm - 1) / (2 * n_sm);
    return (n <= n_sm ? 1.f : 1.35f) * (float)(waves * (per + 3)) + (c > 1 ? join : 0.f);
  };
  int split = 1;
  for (int c = 2; c <= kMaxSplit && c <= tiles; ++c)
    if (cost(c) < cost(split)) split = c;
  return split;
}

}  // namespace f32
}  // namespace scalekv
