// Host check of the sliced window graphs (build_slices) and of the decode
// kernels' shared-memory layout (make_slice_layout), built with g++ by
// tests/test_slices_host.py.
//
// usage: slice_check l m a0x a0y .. b2x b2y rounds W F merge shorten trials
// For every window: each edge is stored once per side and the two sides agree
// on its position; every other place is a dummy; a column's checks ascend in
// window row.
// For random shortened graphs (and the one of the highest degrees) the slices
// stay within the bounds.  Layout regions are 16-byte aligned and disjoint
// where they live together.  Prints "ok" or the first violation.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <string>

#include "../paper_2403_18901_gb300/csrc/qdec_internal.h"
#include "../paper_2403_18901_gb300/csrc/gdg_kernel.cuh"

namespace qd {
std::string last;
void set_error(const std::string& m) { last = m; }
}  // namespace qd

namespace {
#define REQ(c, ...)                \
  do {                             \
    if (!(c)) {                    \
      std::printf(__VA_ARGS__);    \
      std::printf(" [%s]\n", #c);  \
      return false;                \
    }                              \
  } while (0)

bool check_graph(const qd::WindowHost& h) {
  const int nr = h.n_rows, nc = h.n_cols, nrs = (nr + 31) / 32, ncs = (nc + 31) / 32;
  REQ((int)h.s_roff.size() == nrs + 1 && (int)h.s_coff.size() == ncs + 1, "offsets");
  const unsigned low = qd::kWideSlice - 1;
  for (int q = 0; q < ncs; ++q) {
    const int w = (int)(h.s_coff[q + 1] & low) - (int)(h.s_coff[q] & low);
    for (int x = 0; x < 4; ++x) REQ((w >= 4 - x) == (q < h.cls[x]), "slice %d of width %d: class %d", q, w, x);
  }
  size_t real = 0, dummies = 0;
  std::vector<int> seen(h.n_edges, 0);
  for (int l = 0; l < nc; ++l) {
    const int c = h.s_col[l], d = h.col_ptr[c + 1] - h.col_ptr[c], c0 = h.s_coff[l >> 5] & low;
    const int w = (int)(h.s_coff[(l >> 5) + 1] & low) - c0;
    REQ(d <= w, "column %d wider than its slice", l);
    REQ(h.s_llr[l] == h.llr[c], "prior of column %d", l);
    for (int u = 0; u < w; ++u) {
      const uint32_t e = h.s_cent[(size_t)(c0 + u) * 32 + (l & 31)];
      if (u >= d) {
        REQ(e == (uint32_t)(32 * nrs) << 16, "column %d: place %d is no dummy", l, u);
        continue;
      }
      const int r = (int)(e >> 16), pos = (int)(e & 0xFFFF), fe = h.s_cef[(size_t)(c0 + u) * 32 + (l & 31)];
      REQ(r < nr && pos < qd::kMaxRowDeg, "column %d entry %d", l, u);
      REQ(fe == h.col_ptr[c] + u && h.col_rows[fe] == h.s_row[r], "column %d entry %d: edge", l, u);
      seen[fe]++;
      const size_t ri = ((size_t)(h.s_roff[r >> 5] + (pos >> 2)) * 32 + (r & 31)) * 4 + (pos & 3);
      REQ((pos >> 2) < h.s_roff[(r >> 5) + 1] - h.s_roff[r >> 5], "check %d position %d", r, pos);
      REQ(h.s_rent[ri] == l && h.s_ref[ri] == fe, "check %d position %d: other side", r, pos);
    }
  }
  for (int e = 0; e < h.n_edges; ++e) REQ(seen[e] == 1, "edge %d stored %d times", e, seen[e]);
  for (size_t i = 0; i < h.s_rent.size(); ++i) (h.s_rent[i] < nc ? real : dummies)++;
  for (int x : h.s_rent)
    REQ(x < nc || x == 32 * ncs, "check entry is neither a column nor the dummy");
  REQ((int)real == h.n_edges && real + dummies == (size_t)128 * h.row_quads, "check entries");
  return true;
}

struct Region {
  const char* name;
  unsigned off, bytes;
};
bool disjoint(std::vector<Region> rs, unsigned lo, unsigned hi, const char* part) {
  std::sort(rs.begin(), rs.end(), [](const Region& a, const Region& b) { return a.off < b.off; });
  unsigned end = lo;
  for (const Region& r : rs) {
    REQ(r.off % 16u == 0, "%s.%s at %u", part, r.name, r.off);
    if (!r.bytes) continue;
    REQ(r.off >= end, "%s.%s at %u overlaps (ends %u)", part, r.name, r.off, end);
    end = r.off + r.bytes;
    REQ(end <= hi, "%s.%s ends at %u past %u", part, r.name, end, hi);
  }
  return true;
}

// the slices a shortened graph of these window columns takes
bool check_short(const qd::WindowHost& h, const std::vector<int>& cols) {
  std::vector<int> cd, rd(h.n_rows, 0);
  for (int c : cols) {
    cd.push_back(h.col_ptr[c + 1] - h.col_ptr[c]);
    for (int e = h.col_ptr[c]; e < h.col_ptr[c + 1]; ++e) rd[h.col_rows[e]]++;
  }
  std::sort(cd.rbegin(), cd.rend());
  std::sort(rd.rbegin(), rd.rend());
  int cells = 0, quads = 0;
  for (size_t i = 0; i < cd.size(); i += 32) cells += cd[i];
  for (size_t i = 0; i < rd.size(); i += 32) quads += (rd[i] + 3) / 4;
  REQ(cells <= h.scol_cells, "column slices %d > %d", cells, h.scol_cells);
  REQ(quads <= h.srow_quads, "check slices %d > %d", quads, h.srow_quads);
  int rwz = 0, n3 = 0;
  while (32 * rwz < h.n_rows && rd[32 * rwz] > 0) ++rwz;
  while (32 * n3 < (int)cd.size() && cd[32 * n3] >= 3) ++n3;
  for (int m = 0; m < 24; ++m) {  // the shot's own layout
    const qd::SliceDims D{h.row_quads, h.col_cells, h.srow_quads, h.scol_cells};
    const unsigned budget = m & 8 ? 76000u : 232000u;
    const bool ranker = m & 1, lw = m & 2, glob = m & 4;
    qd::Layout L = qd::make_slice_layout(D, h.n_rows, h.n_cols, h.n_short, 22, budget, ranker, lw, glob);
    if (!glob && m >= 16 && L.total < budget) L.total = budget;
    const unsigned end = glob ? L.total - L.U : L.total;
    const qd::SlotPlan S = qd::slot_plan(L, quads, cells, rwz, n3, end, glob, 8);
    const unsigned nsp = qd::up32(h.n_short), rw = L.rw;
    const std::vector<Region> ent = {{"rent", S.rent, 512u * quads}, {"cent", S.cent, 128u * cells},
                                     {"ref", S.ref, lw ? 256u * quads : 0u}, {"cef", S.cef, lw ? 64u * cells : 0u}};
    if (!disjoint(ent, L.s_dyn, S.U, "entries")) return false;
    REQ(S.U <= L.U && S.b_size <= L.b_size, "plan larger than its bound");
    const std::vector<Region> slot = {{"post", 0, 4u * (nsp + 1)}, {"acc", S.b_acc, 128u * n3},
                                      {"hfl", S.b_hfl, 32u * n3}, {"status", S.b_status, nsp},
                                      {"cns", S.b_cns, 16u * (32u * rwz + 1)}, {"deg", S.b_deg, 32u * rw},
                                      {"sp", S.b_sp, 4u * rw}, {"unsat", S.b_unsat, 4u * rw},
                                      {"hq", S.b_hq, ranker ? 128u * n3 : 0u}};
    if (!disjoint(slot, 0, S.b_size, "slot")) return false;
    REQ(S.b_size % 16u == 0 && S.nslots >= 1 && S.nslots <= 8, "%d slots", S.nslots);
    REQ((glob ? 0u : S.U) + S.b_size * (unsigned)S.nslots <= end, "slots past the end");
    REQ(!glob || S.nslots == 8, "%d slots in global memory", S.nslots);
  }
  return true;
}

bool check_layout(const qd::WindowHost& h, int nb, unsigned budget, bool ranker, bool lw, bool glob) {
  const qd::SliceDims D{h.row_quads, h.col_cells, h.srow_quads, h.scol_cells};
  const int nr = h.n_rows, nc = h.n_cols, ns = h.n_short;
  const qd::Layout L = qd::make_slice_layout(D, nr, nc, ns, nb, budget, ranker, lw, glob);
  const unsigned nrp = qd::up32(nr), ncp = qd::up32(nc), nsp = qd::up32(ns), rw = L.rw;
  REQ(L.total % 16u == 0 && L.U % 16u == 0 && L.V % 16u == 0 && L.b_size % 16u == 0, "alignment");
  const std::vector<Region> keep = {{"sbits", L.sbits, 4u * rw}, {"cbits", L.cbits, 4u * L.cw},
                                    {"res_status", L.res_status, 4u * nb}, {"res_pm", L.res_pm, 8u * nb},
                                    {"res_ebits", L.res_ebits, 4u * L.sw * nb}, {"red", L.red, 512u},
                                    {"misc", L.misc, 64u}, {"plan", L.plan, (unsigned)sizeof(qd::SlotPlan)}};
  if (!disjoint(keep, 0, L.V, "persistent")) return false;
  std::vector<Region> sg = {{"sel", L.sel, 2u * ns}, {"roff", L.s_roff, 2u * (rw + 1)},
                            {"coff", L.s_coff, 2u * (L.sw + 1u)}, {"cls", L.s_cls, 16u}, {"llr", L.s_llr, 4u * nsp},
                            {"vdeg", L.s_vdeg, nsp}, {"cperm", L.s_cperm, 2u * nr}, {"vperm", L.s_vperm, 2u * ns}};
  if (!disjoint(sg, L.V, L.s_dyn, "shortened graph")) return false;
  sg.push_back({"entries", L.s_dyn, L.U - L.s_dyn});
  const unsigned base = glob ? 0u : L.V, hi = glob ? L.total - L.U : L.total;
  std::vector<Region> pre = {{"post", L.p_post + base, 4u * (ncp + 1)}, {"key", L.p_key + base, 4u * ncp},
                             {"cns", L.p_cns + base, 16u * (nrp + 1)}, {"par", L.p_par + base, 8u * rw}};
  if (L.pre_stage & qd::kStageRent) pre.push_back({"q_rent", L.q_rent + base, 256u * D.row_quads});
  if (L.pre_stage & qd::kStageCent) pre.push_back({"q_cent", L.q_cent + base, 128u * D.col_cells});
  if (L.pre_stage & qd::kStageLlr) pre.push_back({"q_llr", L.q_sllr + base, 4u * ncp});
  if (L.pre_stage & qd::kStageOff) {
    pre.push_back({"q_roff", L.q_roff + base, 2u * (rw + 1)});
    pre.push_back({"q_coff", L.q_coff + base, 2u * (L.cw + 1u)});
  }
  REQ(!glob || !L.pre_stage, "staging for a union in global memory");
  REQ(budget < 230000u || glob || L.total > 200000u || L.pre_stage == 15u, "a roomy budget stages everything");
  if (!disjoint(pre, base, hi, "pre-BP")) return false;
  // the sort: filled from the keys; then read while the shortened graph is written
  const unsigned need = 8u * (unsigned)L.sortn, scr = 4u * (nsp + 2u * nrp);
  REQ(L.sortn >= ns && !(L.sortn & (L.sortn - 1)), "sort size");
  if (!disjoint({{"key", L.p_key + base, 4u * ncp}, {"sort", L.p_sort + base, need}}, base, hi, "ranking")) return false;
  if (!disjoint({{"scratch", L.p_scr + base, scr}}, base, hi, "scratch")) return false;
  if (!glob) {
    std::vector<Region> a(sg.begin(), sg.end() - 1);
    a.push_back({"sort", L.p_sort + base, need});
    if (!disjoint(a, L.V, hi, "selection")) return false;
    sg.push_back({"scratch", L.p_scr + base, scr});
    if (!disjoint(sg, L.V, hi, "shortening")) return false;
  }
  REQ((glob ? 0u : L.U) + L.b_size * (glob ? 8u : 1u) <= hi, "slots past the end");
  return true;
}
}  // namespace

int main(int argc, char** argv) {
  if (argc != 21) return 2;
  int x[20];
  for (int i = 0; i < 20; ++i) x[i] = std::atoi(argv[i + 1]);
  qd_bb_code code{x[0], x[1], {x[2], x[4], x[6]}, {x[3], x[5], x[7]}, {x[8], x[10], x[12]}, {x[9], x[11], x[13]}};
  const int rounds = x[14], W = x[15], F = x[16], merge = x[17], shorten = x[18], trials = x[19];
  qd::DemHost d;
  const bool ok = rounds > 0 ? qd::build_dem_host(code, qd_noise{0.003, rounds}, d)
                             : qd::build_dem_code_capacity(code, 0.04, 0.001, d);
  if (!ok) return std::printf("dem: %s\n", qd::last.c_str()), 1;
  std::mt19937 rng(5);
  for (int k = 0; k < qd::n_windows(d, W, F); ++k) {
    qd::WindowHost h;
    if (!qd::build_window(d, W, F, k, shorten != 0, h, merge) || !qd::build_slices(h))
      return std::printf("window %d: %s\n", k, qd::last.c_str()), 1;
    if (h.n_cols == 0) continue;
    if (!check_graph(h)) return 1;
    qd::WindowHost same = h, next;  // a window with the same matrix and other priors takes its slices
    for (float& l : same.llr) l *= 1.5f;
    same.s_rent.clear();
    same.s_col.clear();
    if (!qd::build_slices(same, &h) || !check_graph(same)) return 1;
    if (same.s_rent != h.s_rent) return std::printf("window %d: slices not taken\n", k), 1;
    if (qd::build_window(d, W, F, k ? k - 1 : 0, shorten != 0, next, merge) && next.n_cols) {
      qd::build_slices(next, &h);  // whatever its matrix
      if (!check_graph(next)) return 1;
    }
    std::vector<int> cols(h.n_cols);
    for (int c = 0; c < h.n_cols; ++c) cols[c] = h.s_col[c];  // the highest degrees first
    for (int t = 0; t < trials; ++t) {
      if (!check_short(h, std::vector<int>(cols.begin(), cols.begin() + h.n_short))) return 1;
      std::shuffle(cols.begin(), cols.end(), rng);
      if (t & 1)  // the columns of few checks, so that those checks are as heavy as they get
        std::stable_sort(cols.begin(), cols.end(),
                         [&](int a, int b) { return h.col_rows[h.col_ptr[a]] < h.col_rows[h.col_ptr[b]]; });
    }
    for (int nb : {1, 22, 47})
      for (unsigned budget : {0u, 76000u, 115000u, 232000u})
        for (int m = 0; m < 8; ++m)
          if (!check_layout(h, nb, budget, m & 1, m & 2, m & 4)) return 1;
  }
  std::printf("ok\n");
  return 0;
}
