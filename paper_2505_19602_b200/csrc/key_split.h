// How the keys of a slice are cut for the f32 attention: host code, apart so that it compiles without CUDA.
#pragma once

namespace scalekv {
namespace f32 {

constexpr int kMaxSplit = 8;                                // CTAs that may share a slice's keys (portable cluster size)

// CTAs that share a slice's keys.  ctas: CTAs of an unsplit launch.  fit: clusters of c CTAs that the device runs at once (0: none).  In steps of a
// key tile: a CTA that has its SM to itself takes 1 per tile, two that share one 1.35 each.
// A cluster has to fit one GPC: of 296 places on 148 SMs clusters of 2 .. 8 use 148, 93, 71, 56, 45, 37, 33 times c.  With waves of 296 CTAs instead, a launch
// whose clusters just did not fit ran a second wave for the last few (us, 296 places / those that fit; key tiles x CTAs: 13 x 96, three for one 50.3 /
// two 38.7; 28 x 41, seven 51.0 / six 36.8; 35 x 46, six 63.5 / five 44.5; 20 x 192, three 102 / one 87.5; 14 x 190, three 85 / one 70).
// Combining costs 0.8 where the unsplit launch is no more than a wave (one CTA / as here: 2 x 64 10.6 / 9.7, 3 x 64 17.9 / 16.9, 5 x 90 26.4 /
// 23.4, 9 x 148 43.6 / 39.4, 12 x 149 58.9 / 55.8, 34 x 198 139 / 133).  CTAs of longer launches follow on one another, not in waves, and a split loses
// what the model takes the last wave for: 1.5 (8 x 360 81.2, at 0.8 83.8; 11 x 396 94.7, 103.7; 14 x 740 208, 214).
inline int key_split(int ctas, int tiles, int n_sm, const int *fit) {
  const float join = ctas <= 2 * n_sm ? 0.8f : 1.5f;
  auto cost = [&](int c) {
    const int n = ctas * c, per = (tiles + c - 1) / c, at_once = c > 1 ? fit[c] : 2 * n_sm, waves = (ctas + at_once - 1) / at_once;
    return (n <= n_sm ? 1.f : 1.35f) * (float)(waves * (per + 3)) + (c > 1 ? join : 0.f);
  };
  int split = 1;
  for (int c = 2; c <= kMaxSplit && c <= tiles; ++c)
    if (fit[c] > 0 && cost(c) < cost(split)) split = c;
  return split;
}

}  // namespace f32
}  // namespace scalekv
