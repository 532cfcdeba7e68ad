// Row lists of faces and edges as the factorization makes them on the GPU
// (build_fronts, cell_positions, skel_rows) against the host's build_skel and
// filter_rows: the same counts and, row by row, the same positions in the front's
// cells; for the three block sizes and with and without rows dropped before.
// Arguments: n m [p].
#include <cstdlib>

#include "common.cuh"
#include "fronts_check.h"
#include "front.cuh"

using namespace hif;

template <typename U, typename V>
static U* upload(const V& v) {
  U* p = nullptr;
  HIF_CUDA_TRY(cudaMalloc(&p, sizeof(U) * (v.size() + 1)));
  HIF_CUDA_TRY(cudaMemcpy(p, v.data(), sizeof(U) * v.size(), cudaMemcpyHostToDevice));
  return p;
}

int main(int argc, char** argv) try {
  const int n = std::atoi(argv[1]), m = std::atoi(argv[2]);
  const bool periodic = argc > 3;
  Symbolic sym(n, m, periodic);
  const int64_t N = (int64_t)n * n * n;
  long long rows = 0;
  for (int level = 0; level < sym.levels(); ++level) {
    CellPlan cp;
    sym.build_cells(level, cp);
    std::vector<CellDesc> cells(cp.ncell);
    for (int c = 0; c < cp.ncell; ++c)
      cells[c] = CellDesc{0, cp.off[c], (int)(cp.off[c + 1] - cp.off[c]), cp.p[c]};
    CellDesc* cells_d = upload<CellDesc>(cells);
    int32_t* lists_d = upload<int32_t>(cp.dofs);
    int32_t* posb_d = upload<int32_t>(std::vector<int32_t>(8 * N, -77));
    const LevelGeom geo{n, cp.s, cp.C, periodic ? 1 : 0};
    cell_positions(geo, cells_d, cp.ncell, lists_d, posb_d, 0);
    const std::vector<uint8_t> alive = after_cells(cp, N);
    std::vector<uint8_t> later = alive;
    drop_some(cp, 1, 3, later);
    uint8_t* later_d = upload<uint8_t>(later);
    for (int kind = 1; kind <= 2; ++kind) {
      SkelPlan sp;
      sym.build_fronts(cp, kind, alive, sp);
      const int nf = sp.nfront, ncp = sp.ncellPer;
      if (nf == 0) continue;
      std::vector<RowFront> rf(nf);
      for (int f = 0; f < nf; ++f) {
        rf[f] = RowFront{{0, 0, 0, 0}, sp.sep[f], sp.nF[f]};
        for (int i = 0; i < ncp; ++i) rf[f].cell[i] = sp.cells[(size_t)f * ncp + i];
      }
      RowFront* rf_d = upload<RowFront>(rf);
      // the edges' rows are filtered after the faces have dropped DOFs
      for (int filter = 0; filter < kind; ++filter) {
        SkelPlan ref;
        sym.build_skel(cp, kind, alive, ref);
        if (filter) sym.filter_rows(ref, later);
        const auto at = index_fronts(cp, ref);
        for (int mean : {100, 500, 5000}) {   // 32, 128 and 256 threads
          std::vector<int> nR(nf, -1);
          int* nR_d = upload<int>(nR);
          skel_rows(geo, rf_d, nf, ncp, cells_d, lists_d, posb_d, filter ? later_d : nullptr, mean, nR_d,
                    nullptr, nullptr, 0);
          HIF_CUDA_TRY(cudaMemcpy(nR.data(), nR_d, sizeof(int) * nf, cudaMemcpyDeviceToHost));
          std::vector<int64_t> off(nf + 1, 0);
          bool same = true;
          for (int f = 0; f < nf; ++f) {
            const auto it = at.find({sp.sep[f], rf[f].cell[0]});
            CHECK(it != at.end() && nR[f] == ref.nR[it->second], "rows of front %d: %d", f, nR[f]);
            same = same && it != at.end() && nR[f] == ref.nR[it->second];
            off[f + 1] = off[f] + sp.nF[f] + nR[f];
          }
          if (!same) {   // the positions are only written where they are known to fit
            cudaFree(nR_d);
            continue;
          }
          std::vector<int32_t> pos(off[nf] * ncp, -77);
          int32_t* pos_d = upload<int32_t>(pos);
          int64_t* off_d = upload<int64_t>(off);
          skel_rows(geo, rf_d, nf, ncp, cells_d, lists_d, posb_d, filter ? later_d : nullptr, mean, nullptr,
                    off_d, pos_d, 0);
          HIF_CUDA_TRY(cudaMemcpy(pos.data(), pos_d, sizeof(int32_t) * pos.size(), cudaMemcpyDeviceToHost));
          for (int f = 0; f < nf; ++f) {
            const int r = at.find({sp.sep[f], rf[f].cell[0]})->second;
            const int64_t cnt = (off[f + 1] - off[f]) * ncp;
            for (int64_t e = 0; e < cnt; ++e)
              CHECK(pos[off[f] * ncp + e] == ref.rowPos[ref.rowOff[r] * ncp + e],
                    "level %d kind %d front %d row %lld cell %lld", level, kind, f, (long long)(e / ncp),
                    (long long)(e % ncp));
          }
          rows += off[nf];
          for (void* p : {(void*)nR_d, (void*)pos_d, (void*)off_d}) cudaFree(p);
        }
      }
      cudaFree(rf_d);
    }
    for (void* p : {(void*)cells_d, (void*)lists_d, (void*)posb_d, (void*)later_d}) cudaFree(p);
    std::vector<uint8_t> left = later;
    drop_some(cp, 2, 5, left);
    std::vector<int32_t> next;
    for (int32_t g : cp.active)
      if (left[g]) next.push_back(g);
    sym.set_active(next);
  }
  std::printf("%lld rows\n%s\n", rows, fails ? "FAILED" : "OK");
  return fails ? 1 : 0;
} catch (const Error& e) {
  std::printf("%s\n", e.msg.c_str());
  return 2;
}
