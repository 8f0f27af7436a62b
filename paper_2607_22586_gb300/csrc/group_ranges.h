// Group ranges of the CUDA-core mass pass (plain C++).
//
// Each CTA of the pass takes a key tile and a range of the proxy groups. The
// groups lie in ranges of gper, the last one shorter where they do not divide;
// the anchor (group G) is a last range of its own (own), or part of the last one.
#ifndef MMSHIFT_GROUP_RANGES_H_
#define MMSHIFT_GROUP_RANGES_H_

#include <algorithm>
#include <cmath>

#ifdef __CUDACC__
#define MMSHIFT_HD __host__ __device__
#else
#define MMSHIFT_HD
#endif

namespace mmshift {

struct GroupRanges {
  int gper, ngr;   // groups per range, ranges
  bool own;
};

// Groups [g0, g1) of range i; g1 = G + 1 takes the anchor too.
MMSHIFT_HD inline void range_groups(const GroupRanges& r, int G, int i, int& g0, int& g1) {
  g0 = i * r.gper < G ? i * r.gper : G;
  g1 = i == r.ngr - 1 ? G + 1 : (g0 + r.gper < G ? g0 + r.gper : G);
}

// An SM takes n CTAs two at a time and a last odd one alone at about 0.6 of the
// rate, each for its tiles of `tile` rows and about half a tile more for its keys;
// the anchor goes with the last range (about 0.3 of a tile for its sums) or alone,
// beside an odd CTA if there is one. Of all range lengths the one with the least
// time by that. Ranges for about three rounds of two CTAs, the anchor counted as a
// group, left last rounds nearly empty and tiles partly filled: 4001 keys, 8 groups
// of 112 rows, 263 us a call in ranges of two groups, 242 of four; 346 keys over
// eight KV heads 126 -> 97; 42 calls of 200 to 4000 keys 3 % less on average.
// G groups of RG rows, anchor_rows anchor rows, keyu key tiles over the KV heads
// and layers, nsm SMs.
inline GroupRanges choose_ranges(int G, int RG, int anchor_rows, int tile, long long keyu, int nsm) {
  const int G1 = std::max(G, 1);
  GroupRanges r{G1, 1, false};
  double best = -1;
  for (int n = 1; n <= G1; ++n) {
    const int len = (G1 + n - 1) / n;              // groups per range
    if ((G1 + len - 1) / len != n) continue;       // the same length as a smaller n
    const double ctas = (double)((keyu * n + nsm - 1) / nsm), odd = ctas - 2 * std::floor(ctas / 2);
    for (int alone = 0; alone <= (G ? 1 : 0); ++alone) {
      const int last = (G - (n - 1) * len) * RG + (alone ? 0 : anchor_rows);
      const double each = std::max((std::min(len, G) * RG + tile - 1) / tile + 0.5,
                                   (last + tile - 1) / tile + (alone ? 0.5 : 0.8));
      const double time = ctas * each + std::max(0.67 * odd * each, alone ? 1.5 * keyu / nsm : 0.0);
      if (best < 0 || time < best) {
        best = time;
        r.gper = len;
        r.own = alone != 0;
        r.ngr = n + alone;
      }
    }
  }
  return r;
}

}  // namespace mmshift

#endif  // MMSHIFT_GROUP_RANGES_H_
