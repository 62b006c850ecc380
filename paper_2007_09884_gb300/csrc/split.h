// split.h -- how a search's simplices are split into work units (host only, no
// CUDA: the tests compile it alone).
#pragma once

#include <algorithm>

namespace opmm {

// A search launch shape: simplices per block (in NG groups) and trial points
// per simplex.
struct SplitShape {
  int G, NG, nt;
};

// One Nelder-Mead step of a search unit against its 32-candidate chunks, in
// thousands of SM cycles (2 x 32 packed, 150 samples at 1 kHz; one simplex
// 22.6, 8 33.7, 16 39.8, 32 53.1, 48 79.2, 64 simplices 101): a chunk's and a
// decision's latency first, the SM's throughput from about 24 chunks on.  The
// other shapes and windows are not modelled apart: the split compares unit
// sizes of one shape on one window, where only the ratios count (4 x 16 63.7
// and 104 at 32 and 64 simplices, 500 Hz x 300 samples 88.9 and 173.5).
inline double unit_step(int chunks) { return std::max(21.0 + 1.5 * chunks, 5.0 + 2.18 * chunks); }

inline double unit_step(const SplitShape& s, int m) {   // of m simplices in NG even groups
  int chunks = 0;
  for (int h = 0; h < s.NG; ++h) chunks += (s.nt * ((m * (h + 1)) / s.NG - (m * h) / s.NG) + 31) / 32;
  return unit_step(chunks);
}

// Units per saccade: the number of units that n saccades' S simplices are
// split into evenly, at most G simplices each, or 0 for full units of G and a
// last one with the rest.  The split with the least turns of the blocks times
// the step of one unit: a batch with many units per block keeps its units as
// large as they come (a simplex costs 1.6 k cycles a step in a unit of 64 and
// 2.5 k in one of 16), a few saccades are spread over every SM (one saccade
// of 186 simplices: 93 units of two instead of 6 of 32).  A simplex evolves
// the same in any unit, so the results do not depend on the split.
//
// Among the unit counts of one unit size m the smallest, ceil(S / m), has the
// fewest turns, so only those are tried: at most G of them however many
// simplices there are (every count from S / G to S took 0.1 ms at 65,536
// candidates and 6.6 ms at 2^20, more than such a search of one saccade).
inline int split_units(int n, int S, const SplitShape& shape, int blocks) {
  const int least = (S + shape.G - 1) / shape.G;
  double best = 1e300;
  int pick = least;
  for (int m = (S + least - 1) / least; m >= 1; --m) {
    const int ng = (S + m - 1) / m;
    if ((S + ng - 1) / ng != m) continue;   // no count has this unit size
    const double turns = std::max(1.0, (double)(((long long)n * ng + blocks - 1) / blocks));
    const double t = turns * unit_step(shape, m);
    if (t < best * 0.999) {
      best = t;
      pick = ng;
    }
  }
  // with many units per saccade an even split only rounds every group up to
  // whole chunks, and full units lose only in their last one
  return pick == least && (S % shape.G == 0 || least > 8) ? 0 : pick;
}

}  // namespace opmm
