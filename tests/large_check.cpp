// Host check of the layouts for windows whose shortened graph does not fit a
// CTA's shared memory (make_slice_layout's kGraphGlobal), built with g++ by
// tests/test_large_windows_host.py.
//
// usage: large_check l m a0x a0y .. b2x b2y rounds W shorten limit
// The kernels have a layout within `limit` bytes of shared memory wherever the
// plain CSC and CSR arrays (make_layout) with the path state in global memory
// had one; path mode has one with the learned weights' edge ids in global memory
// wherever it had one with the plain arrays.  In the region of global memory the entries, the pre-BP scratch and
// the slots of the largest and of smaller shortened graphs are disjoint where
// they live together.  Prints "ok", with the number of layouts that needed it.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <string>

#include "../paper_2403_18901_gb300/csrc/qdec_internal.h"
#include "../paper_2403_18901_gb300/csrc/gdg_kernel.cuh"

namespace qd {
std::string last;
void set_error(const std::string& m) { last = m; }
}  // namespace qd

#define REQ(c)                                              \
  do {                                                      \
    if (!(c)) return std::printf("line %d: %s\n", __LINE__, #c), 1; \
  } while (0)

int main(int argc, char** argv) {
  int x[18];
  if (argc != 19) return 2;
  for (int i = 0; i < 18; ++i) x[i] = std::atoi(argv[i + 1]);
  qd_bb_code code{x[0], x[1], {x[2], x[4], x[6]}, {x[3], x[5], x[7]}, {x[8], x[10], x[12]}, {x[9], x[11], x[13]}};
  const int W = x[15];
  const bool shorten = x[16] != 0;
  const unsigned limit = (unsigned)x[17];
  qd::DemHost d;
  if (!qd::build_dem_host(code, qd_noise{0.003, x[14]}, d)) return std::printf("dem: %s\n", qd::last.c_str()), 1;
  int used = 0;
  for (int k = 0; k < qd::n_windows(d, W, 1); ++k) {
    qd::WindowHost h;
    if (!qd::build_window(d, W, 1, k, shorten, h) || !qd::build_slices(h))
      return std::printf("window %d: %s\n", k, qd::last.c_str()), 1;
    const qd::SliceDims D{h.row_quads, h.col_cells, h.srow_quads, h.scol_cells};
    for (int nb : {1, 16, 47})
      for (int m = 0; m < 4; ++m) {
        const bool ranker = m & 1, lw = m & 2;
        if (qd::make_layout(h.n_rows, h.n_cols, h.n_edges, h.n_short, h.short_edges_max, nb, 8, false, ranker, lw).U > limit)
          continue;
        auto lay = [&](bool gg) {
          return qd::make_slice_layout(D, h.n_rows, h.n_cols, h.n_short, nb, 0, ranker, lw, true, gg ? qd::kGraphGlobal : qd::kGraphShared);
        };
        if (lw) {  // path mode's, with the edge ids in global memory
          const qd::Layout L = qd::make_slice_layout(D, h.n_rows, h.n_cols, h.n_short, nb, limit, ranker, lw, false,
                                                     qd::kIdsGlobal);
          const qd::Layout O = qd::make_layout(h.n_rows, h.n_cols, h.n_edges, h.n_short, h.short_edges_max, nb, 1, true,
                                               ranker, lw);
          REQ(O.total - O.g_bytes > limit || L.total <= limit);
          const qd::SlotPlan S = qd::slot_plan(L, D.srow_quads, D.scol_cells, L.rw, L.sw, L.total, false, 1);
          REQ(S.ref == 0 && S.cef >= 256u * D.srow_quads && S.ids >= S.cef + 64u * D.scol_cells && S.ids == L.ids);
          REQ(S.cent >= S.rent + 512u * D.srow_quads && S.U >= S.cent + 128u * D.scol_cells && S.U == L.U);
          REQ(S.U + S.b_size <= L.total && L.V + L.p_end <= L.total && S.nslots == 1 && L.ids % 16u == 0);
        }
        if (lay(false).U <= limit) continue;
        ++used;
        const qd::Layout L = lay(true);
        REQ(L.gg == qd::kGraphGlobal && L.U <= limit && L.U % 16u == 0 && L.total % 16u == 0 && L.U >= L.s_vperm + 2u * h.n_short);
        const unsigned end = L.total - L.U, nsp = qd::up32(h.n_short), nrp = qd::up32(h.n_rows), ncp = qd::up32(h.n_cols);
        for (int part = 0; part < 3; ++part) {  // the largest graph, a half, the smallest
          const int nq = part == 0 ? D.srow_quads : (part == 1 ? D.srow_quads / 2 : 1);
          const int cells = part == 0 ? D.scol_cells : (part == 1 ? D.scol_cells / 2 : 1);
          const qd::SlotPlan S = qd::slot_plan(L, nq, cells, L.rw, L.sw, end, true, 8);
          REQ(S.rent == 0 && S.cent >= 512u * nq && S.ref >= S.cent + 128u * cells);
          REQ(S.cef >= S.ref + (lw ? 256u * nq : 0u) && S.U >= S.cef + (lw ? 64u * cells : 0u));
          // entries are written while the selection, the sort and the scratch are read
          REQ(S.U <= L.p_post && S.U <= L.p_sort && S.U <= L.p_scr);
          REQ(S.nslots == 8 && S.U + 8u * S.b_size <= end && S.b_size <= L.b_size && S.U % 16u == 0);
        }
        REQ(L.p_key >= L.p_post + 4u * (ncp + 1) && L.p_cns >= L.p_key + 4u * ncp && L.p_par >= L.p_cns + 16u * (nrp + 1));
        REQ(L.p_sort >= L.p_par + 8u * L.rw && L.p_sort + 8u * (unsigned)L.sortn <= end);
        REQ(L.p_scr >= L.p_par + 8u * L.rw && L.p_scr + 4u * (nsp + 2u * nrp) <= end);
        REQ(!L.pre_stage);
      }
  }
  std::printf("ok %d\n", used);
  return 0;
}
