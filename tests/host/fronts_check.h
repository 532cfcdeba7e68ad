// Reference lists of a level's faces and edges for the checks of build_fronts (host)
// and of the device row lists: build_skel's fronts, found by separator mask and low cell.
#pragma once

#include <cstdio>
#include <map>
#include <utility>
#include <vector>

#include "symbolic.h"

inline int fails = 0;
#define CHECK(c, ...)                      \
  do {                                     \
    if (!(c)) {                            \
      if (fails < 20) {                    \
        std::printf("FAIL %s: ", #c);      \
        std::printf(__VA_ARGS__);          \
        std::printf("\n");                 \
      }                                    \
      ++fails;                             \
    }                                      \
  } while (0)

// the DOFs still there after the level's cells are eliminated
inline std::vector<uint8_t> after_cells(const hif::CellPlan& cp, int64_t N) {
  std::vector<uint8_t> alive(N, 0);
  for (int32_t g : cp.active) alive[g] = 1;
  for (int c = 0; c < cp.ncell; ++c)
    for (int64_t t = cp.off[c]; t < cp.off[c] + cp.p[c]; ++t) alive[cp.dofs[t]] = 0;
  return alive;
}

// separator mask of an active DOF
inline int sep_of(const hif::CellPlan& cp, int32_t g) { return (int)(cp.packed[cp.slot[g]] >> 48); }

// drop some of the DOFs that lie on one separator plane (a face's) or on two (an edge's)
inline void drop_some(const hif::CellPlan& cp, int planes, int every, std::vector<uint8_t>& alive) {
  int t = 0;
  for (int32_t g : cp.active) {
    const int m = sep_of(cp, g);
    if (((m & 1) + (m >> 1 & 1) + (m >> 2 & 1)) == planes && alive[g] && t++ % every == 0) alive[g] = 0;
  }
}

inline std::map<std::pair<int, int>, int> index_fronts(const hif::CellPlan& cp, const hif::SkelPlan& ref) {
  std::map<std::pair<int, int>, int> at;
  for (int f = 0; f < ref.nfront; ++f)
    at[{sep_of(cp, ref.rowDof[ref.rowOff[f]]), ref.cells[(size_t)f * ref.ncellPer]}] = f;
  return at;
}
