// build_fronts (the plan of a factorization) against build_skel, front by front: the
// same separator masks, cells and DOFs in the same order.  Arguments: n m [p].
#include <cstdlib>

#include "fronts_check.h"

using namespace hif;

int main(int argc, char** argv) {
  const int n = std::atoi(argv[1]), m = std::atoi(argv[2]);
  Symbolic sym(n, m, argc > 3);
  const int64_t N = (int64_t)n * n * n;
  long long fronts = 0;
  for (int level = 0; level < sym.levels(); ++level) {
    CellPlan cp;
    sym.build_cells(level, cp);
    std::vector<uint8_t> alive = after_cells(cp, N);
    for (int kind = 1; kind <= 2; ++kind) {
      SkelPlan ref, sp;
      sym.build_skel(cp, kind, alive, ref);
      sym.build_fronts(cp, kind, alive, sp);
      const auto at = index_fronts(cp, ref);
      CHECK(sp.nfront == ref.nfront && (int)at.size() == ref.nfront && sp.ncellPer == ref.ncellPer,
            "level %d kind %d: %d fronts, %d expected", level, kind, sp.nfront, ref.nfront);
      for (int f = 0; f < sp.nfront; ++f) {
        const auto it = at.find({sp.sep[f], sp.cells[(size_t)f * sp.ncellPer]});
        if (it == at.end()) {
          CHECK(false, "no such front");
          continue;
        }
        const int r = it->second;
        CHECK(sp.nF[f] == ref.nF[r] && sp.memOff[f + 1] - sp.memOff[f] == ref.nF[r], "front size");
        for (int i = 0; i < sp.ncellPer; ++i)
          CHECK(sp.cells[(size_t)f * sp.ncellPer + i] == ref.cells[(size_t)r * sp.ncellPer + i], "cells");
        for (int i = 0; i < std::min(sp.nF[f], ref.nF[r]); ++i)
          CHECK(sp.mem[sp.memOff[f] + i] == ref.rowDof[ref.rowOff[r] + i], "DOF %d of a front", i);
      }
      fronts += sp.nfront;
    }
    // the faces lose every third DOF, the edges every fifth
    drop_some(cp, 1, 3, alive);
    drop_some(cp, 2, 5, alive);
    std::vector<int32_t> next;
    for (int32_t g : cp.active)
      if (alive[g]) next.push_back(g);
    sym.set_active(next);
  }
  std::printf("%lld fronts\n%s\n", fronts, fails ? "FAILED" : "OK");
  return fails ? 1 : 0;
}
