// qdec_api.cu -- the C ABI of libqdec (see include/qdec.h).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <memory>
#include <mutex>
#include <string>
#include <vector>

#include "gdg_kernel.cuh"
#include "qdec_internal.h"

namespace qd {
static thread_local std::string g_err;
void set_error(const std::string& m) { g_err = m; }
}  // namespace qd

using qd::set_error;

#define QD_CK(call)                                                                   \
  do {                                                                                \
    cudaError_t e_ = (call);                                                          \
    if (e_ != cudaSuccess) {                                                          \
      set_error(std::string(#call) + ": " + cudaGetErrorString(e_));                  \
      return QD_ECUDA;                                                                \
    }                                                                                 \
  } while (0)

#define QD_CK_ST(call)             \
  do {                             \
    const qd_status s_ = (call);   \
    if (s_ != QD_OK) return s_;    \
  } while (0)

#define QD_REQ(cond, msg)    \
  do {                       \
    if (!(cond)) {           \
      set_error(msg);        \
      return QD_EINVAL;      \
    }                        \
  } while (0)

struct qd_dem {
  qd::DemHost h;
  // device copies, uploaded on first device use (so that the host-side
  // queries work on a machine without a GPU)
  mutable int* d_cptr = nullptr;
  mutable int* d_cdet = nullptr;
  mutable uint32_t* d_cobs = nullptr;
  mutable uint32_t* d_thr = nullptr;
};

namespace {

// Launch shapes of the decode kernel: shot mode (persistent CTAs of up to
// kShotWarps warps, one warp per decision path, as many as fit in shared
// memory) and path mode (one CTA of kPathThreads threads per (shot, path)).
constexpr int kShotWarps = 8;
// CTAs per SM at most: three take 80 registers a thread.  5000 shots of
// [[144,12,12]] run 4 % faster so than with two and 128 registers (the paper
// preset 5 %); with learned weights or a ranker 3 and 6 % slower.
constexpr int kShotCtas = 3;
// Warps of a CTA that has its SM for itself: 150 shots of [[144,12,12]] with the
// paper preset's 22 paths, all windows, 12.7 ms with 8, 11.2 with 12, 11.6 with 16;
// [[288,12,18]] 34.4, 32.4 and 34.1 ms (configured, 16 paths); the configured preset
// of [[144,12,12]] 18.9, 18.8 and 19.5.
constexpr int kWideWarps = 12;
// Path mode's CTAs: 512 threads, one per SM; 256, two; 128, four (the same 128
// registers a thread), see path_shape.
constexpr int kPathShapes = 3;
constexpr int kPathThreads = 512;
constexpr long long kPathModeMaxShots = 64;
constexpr int kCounters = 8;

// Shot mode on up to `ctas` CTAs per SM, and its snapshot plan (qd::ForkDev):
// queue order [nb], then the node chain [nb][dmx]; fork_nodes = 0: none.
struct ShotShape {
  qd::Layout L{};
  int warps = kShotWarps;
  int ctas = 2;         // CTAs per SM planned
  int grid_per_sm = 1;  // and resident
  int wave = 1;         // path slots of a typical shot
  const int16_t* d_fork = nullptr;  // in one of WinGpu::d_fork
  int fork_nodes = 0;
  bool fork_on = false;
};

struct PathShape {
  qd::Layout L{};
  bool fits = false;
  int pcl = 1;  // CTAs per cluster sharing a shot's pre-BP
};

struct WinGpu {
  qd::WindowHost h;
  qd::WinDev dv{};
  ShotShape sh[kShotCtas];  // shot mode, by CTAs per SM
  int best = 0;             // the one for large batches
  int16_t* d_fork[4] = {};  // the shapes' snapshot plans, by layout_form
  PathShape pa[kPathShapes];  // path mode, kPathThreads >> i threads
  char* d_graph = nullptr;
  int* d_ccptr = nullptr;  // committed columns: CSR of their global detector ids
  int* d_ccdet = nullptr;
  uint32_t* d_ccobs = nullptr;
  uint32_t* d_wthr = nullptr;  // window-local sampling thresholds (on first use)
  // union region in global memory (windows too large for shared memory, or
  // launch mode 3): layout, CTAs per SM, and whether the shared-memory
  // layouts fit at all
  qd::Layout Lg{};
  int grid_g = 1;
  bool fits = true;
  // message reuse: this window's column -> the previous window's column of
  // the same DEM column (-1: none); nullptr for the first window
  int16_t* d_prev = nullptr;
  float* d_wts = nullptr;  // learned weights in the pre-BP's order, room for wts_rows iterations
  int wts_rows = 0;
};

template <class T>
cudaError_t upload(T** dst, const std::vector<T>& v) {
  size_t n = std::max<size_t>(v.size(), 1);
  cudaError_t e = cudaMalloc((void**)dst, n * sizeof(T));
  if (e != cudaSuccess) return e;
  if (!v.empty()) e = cudaMemcpy(*dst, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
  return e;
}

// Arrays in one allocation: every array starts on a 16-byte boundary and is
// padded to a multiple of 16 bytes, as the kernels' bulk (TMA) copies into
// shared memory require.
struct Blob {
  std::vector<char> bytes;
  template <class T>
  size_t put(const std::vector<T>& v) {
    const size_t o = bytes.size(), n = v.size() * sizeof(T);
    bytes.resize((o + n + 15) & ~(size_t)15);
    if (n) memcpy(bytes.data() + o, v.data(), n);
    return o;
  }
  cudaError_t upload(char** dst) const {
    const cudaError_t e = cudaMalloc((void**)dst, std::max<size_t>(bytes.size(), 16));
    return e != cudaSuccess ? e : cudaMemcpy(*dst, bytes.data(), bytes.size(), cudaMemcpyHostToDevice);
  }
};

qd_status ensure_device(const qd_dem* d) {
  if (d->d_thr) return QD_OK;
  QD_CK(upload(&d->d_cptr, d->h.col_ptr));
  QD_CK(upload(&d->d_cdet, d->h.col_dets));
  QD_CK(upload(&d->d_cobs, d->h.col_obs));
  std::vector<uint32_t> thr(d->h.col_thr);  // in fours, the last ones padded with columns that never fire
  thr.resize((thr.size() + 3) & ~(size_t)3, 0u);
  QD_CK(upload(&d->d_thr, thr));
  return QD_OK;
}

}  // namespace

struct qd_decoder {
  const qd_dem* dem = nullptr;
  qd_gdg_params P{};
  qd::KParams kp{};
  long long max_shots = 0;
  std::vector<WinGpu> wins;
  int corr_words = 0, dmx = 0, ns_max = 0, sm_count = 0, sw_max = 0;
  int launch_mode = 0;  // 0 automatic, 1 shot mode, 2 path mode, 3 shot mode with the union region in global memory
  char* d_uscratch = nullptr;  // global union regions (one per resident CTA)
  size_t uscratch_bytes = 0;
  char* d_path_res = nullptr;
  int* d_arrive = nullptr;
  size_t trace_bytes = 0, smem_max = 0;
  int smem_optin = 0, smem_sm = 0, smem_reserved = 0;  // dynamic per CTA at most, per SM, taken by each CTA
  bool hist_on = false;  // layouts hold the quantised history (ranker or dump)
  bool lw_on = false;    // layouts keep the shortened edges' full-window ids (learned weights)
  void* d_ranker = nullptr;  // grid-rounded parameters (644 floats), then the 256 B fragments
  int* d_work = nullptr;
  long long* d_counters = nullptr;  // kCounters entries (qd_decoder_counters_ex)
  uint32_t* d_corr = nullptr;
  // shot mode's snapshots of shared path prefixes: one pool per resident CTA
  char* d_snap = nullptr;
  size_t snap_cta_bytes = 0;
  int snap_ctas = 0;
  bool fork_on = true;
  bool sched_on = true;  // preemption at step boundaries (with fork_on)
  // message reuse between windows (qd_gdg_params.reuse_msgs): per shot the
  // values a window keeps for the next [max_shots][keep_ld], and every
  // candidate path's values [slots][nb][ns_max]
  float* d_keep = nullptr;
  int keep_ld = 0;
  float* d_kpath = nullptr;
  size_t kpath_slots = 0;
  uint32_t *d_det = nullptr, *d_obs = nullptr, *d_pred = nullptr, *d_fail = nullptr, *d_resid = nullptr;
  long long* d_nfail = nullptr;
  // buffers that larger ones have replaced: a CUDA graph captured before may
  // still write to them, so they stay until the decoder goes
  std::vector<void*> retired;
};

namespace {
// A larger buffer in the place of *p, which is kept (qd_decoder::retired).
template <class T>
qd_status replace_buffer(qd_decoder* dec, T** p, size_t bytes) {
  T* q = nullptr;
  QD_CK(cudaMalloc((void**)&q, bytes));
  if (*p) dec->retired.push_back(*p);
  *p = q;
  return QD_OK;
}

// What the decoder's layouts are made for: learned weights, quantised history.
int layout_form(bool lw, bool hist) { return (lw ? 1 : 0) | (hist ? 2 : 0); }

// Path mode's CTAs per shot: the paths, rounded up to whole clusters.
int path_ctas(const qd_decoder* dec, const PathShape& p) { return (dec->kp.nb + p.pcl - 1) / p.pcl * p.pcl; }

// Global union regions for the windows that need them (all windows when
// `all`): one region per resident CTA, allocated once, never on a decode call.
qd_status ensure_uscratch(qd_decoder* dec, bool all) {
  size_t need = 0;
  for (const WinGpu& g : dec->wins)
    if (all || !g.fits)
      need = std::max(need, (size_t)dec->sm_count * g.grid_g * (size_t)(g.Lg.total - g.Lg.U));
  for (const WinGpu& g : dec->wins)  // path mode's edge ids
    if (g.pa[0].fits && g.pa[0].L.gg == qd::kIdsGlobal)
      need = std::max(need, (size_t)std::min(dec->max_shots, kPathModeMaxShots) * path_ctas(dec, g.pa[0]) *
                                (size_t)g.pa[0].L.ids);
  if (need <= dec->uscratch_bytes) return QD_OK;
  QD_CK_ST(replace_buffer(dec, &dec->d_uscratch, need));
  dec->uscratch_bytes = need;
  return QD_OK;
}

// Shot mode's plan for sharing path prefixes (qd::ForkDev).  The decision of
// path p at depth d is summarised as (contrary value at d, main-branch
// thresholds of Alg. 3 at d (when Alg. 3 is on), message restart after d);
// two paths with equal summaries at depths 1..D-1 hold the same state after
// the BP of step D.  The queue order runs `wave` paths at once first, each
// sharing as little as possible with those before it, then takes the paths
// that share the deepest prefix with a path before them; node = the deepest
// state such a later path shares with an earlier one.
struct ForkPlan {
  std::vector<int16_t> order, chain, fnode, fdep;
  int n_nodes = 0;
  bool on = false;  // more paths than warps: a plan (preemption, and snapshots when n_nodes > 0)
};

ForkPlan fork_plan(const qd::KParams& P, int dmx, int wave) {
  const int nb = P.nb;
  auto dmax = [&](int p) { return qd::path_dmax(P, p, qd::path_split(P, p)); };
  auto sig = [&](int p, int d) {
    const int split = qd::path_split(P, p);
    const int contrary = split ? (d == split ? 1 : 0) : (d <= P.k ? (p >> (P.k - d)) & 1 : 0);
    const int mainr = P.low_err ? 0 : ((p == 0 || (split && d <= split)) ? 1 : 0);
    const int re = qd::path_reinit(P, p, split) == d ? 1 : 0;
    return contrary | (mainr << 1) | (re << 2);
  };
  // deepest D with equal summaries below it that both paths reach
  auto shared = [&](int p, int q) {
    const int m = std::min(dmax(p), dmax(q));
    int D = 1;
    while (D < m && sig(p, D) == sig(q, D)) ++D;
    return D;
  };
  ForkPlan F;
  std::vector<int> order;
  std::vector<char> used(nb, 0);
  std::vector<int> share(nb, 0);  // deepest prefix shared with a path before it in the order
  for (int pos = 0; pos < nb; ++pos) {
    int best = -1, bkey = 0, bs = 0;
    for (int q = 0; q < nb; ++q) {
      if (used[q]) continue;
      int s = 0;
      for (int p : order) s = std::max(s, shared(p, q));
      const int key = pos < wave ? -s : s;
      if (best < 0 || key > bkey || (key == bkey && dmax(q) > dmax(best))) {
        best = q;
        bkey = key;
        bs = s;
      }
    }
    used[best] = 1;
    share[best] = pos < wave ? 0 : bs;
    order.push_back(best);
  }
  // nodes: (depth, summaries below it) of every later path's shared prefix
  std::vector<std::vector<int>> keys;
  auto key_of = [&](int p, int D) {
    std::vector<int> k{D};
    for (int d = 1; d < D; ++d) k.push_back(sig(p, d));
    return k;
  };
  for (int q = 0; q < nb; ++q)
    if (share[q] >= 1) {
      const std::vector<int> k = key_of(q, share[q]);
      if (std::find(keys.begin(), keys.end(), k) == keys.end()) keys.push_back(k);
    }
  if (nb <= wave || nb > qd::kMaxForkNodes || (int)keys.size() > qd::kMaxForkNodes) return F;
  F.on = true;
  F.n_nodes = (int)keys.size();
  F.order.assign(order.begin(), order.end());
  F.chain.assign((size_t)nb * dmx, (int16_t)-1);
  F.fnode.assign(nb, (int16_t)-1);
  F.fdep.assign(nb, (int16_t)0);
  for (int p = 0; p < nb; ++p) {
    for (int D = 1; D <= dmax(p) && D <= dmx; ++D) {
      const auto it = std::find(keys.begin(), keys.end(), key_of(p, D));
      if (it != keys.end()) F.chain[(size_t)p * dmx + D - 1] = (int16_t)(it - keys.begin());
    }
    if (share[p] >= 1) {
      F.fnode[p] = F.chain[(size_t)p * dmx + share[p] - 1];
      F.fdep[p] = (int16_t)share[p];
    }
  }
  return F;
}

qd::SliceDims slice_dims(const qd::WindowHost& h) {
  return qd::SliceDims{h.row_quads, h.col_cells, h.srow_quads, h.scol_cells};
}

// Dynamic shared memory of one of n CTAs per SM.
unsigned smem_budget(const qd_decoder* dec, int n) {
  return (unsigned)std::max(0, std::min(dec->smem_optin, dec->smem_sm / n - dec->smem_reserved)) & ~15u;
}

// Path slots of a typical shot within L.total: shortened graphs hold fewer and
// thinner columns than the window's mean (the ranking keeps likely faults;
// measured 671 to 750 edges for the 432 columns of [[144,12,12]] (3,1)
// windows, half the mean), their check slices are about half full, two thirds
// of them non-empty, and half of the columns have degree three or more.
int typical_slots(const qd::Layout& L, const qd::WindowHost& h, int most) {
  const double edges = 0.67 * h.n_edges / std::max(1, h.n_cols) * h.n_short;
  const int nq = std::min(h.srow_quads, (int)(2.0 * edges / 128) + 1);
  const int cells = std::min(h.scol_cells, (int)(1.4 * edges / 32) + 1);
  const qd::SlotPlan S =
      qd::slot_plan(L, nq, cells, std::max(1, (2 * L.rw + 2) / 3), std::max(1, (L.sw + 1) / 2), L.total, false, most);
  return std::max(1, S.nslots);
}

bool same_dims(const qd::WindowHost& a, const qd::WindowHost& b) {  // one layout for both
  return a.n_rows == b.n_rows && a.n_cols == b.n_cols && a.n_short == b.n_short && a.n_edges == b.n_edges &&
         a.row_quads == b.row_quads && a.col_cells == b.col_cells && a.srow_quads == b.srow_quads &&
         a.scol_cells == b.scol_cells;
}

// Shared-memory layouts of every window: shot mode's for one to kShotCtas CTAs
// per SM, the one with its path state in global memory, path mode's.  The ranker
// and the candidate dump (hist) add the quantised history (4 bytes per column of
// degree three or more) to every slot, learned weights the entries' edge ids.
qd_status configure_layouts(qd_decoder* dec, bool hist, const char* who) {
  struct Conf {
    ShotShape sh[kShotCtas];
    PathShape pa[kPathShapes];
    qd::Layout Lg;
    int best, grid_g;
    bool fits;
  };
  const int optin = dec->smem_optin;
  const int nb = dec->kp.nb;
  size_t smem_max = 0;
  std::vector<Conf> cf(dec->wins.size());
  for (size_t w = 0; w < cf.size(); ++w) {
    Conf& c = cf[w];
    if (w && same_dims(dec->wins[w - 1].h, dec->wins[w].h)) {  // interior windows
      c = cf[w - 1];
      continue;
    }
    const auto& h = dec->wins[w].h;
    auto lay = [&](unsigned budget, bool glob = false, qd::GraphPlace place = qd::kGraphShared) {
      return qd::make_slice_layout(slice_dims(h), h.n_rows, h.n_cols, h.n_short, nb, budget, hist, dec->lw_on, glob,
                                   place);
    };
    // CTAs per SM: for large batches the most resident decision-path warps
    // (CTAs x slots a typical shot gets); ties to fewer CTAs, which have room to
    // stage more of the window graph.  Smaller batches: see shot_shape.
    int best = 0;
    c.fits = false;
    c.best = 0;
    for (int n = 1; n <= (dec->lw_on || hist ? 2 : kShotCtas); ++n) {
      const unsigned budget = smem_budget(dec, n);
      ShotShape& s = c.sh[n - 1];
      s.L = lay(budget);
      if (s.L.total > budget) break;  // (the budgets fall)
      s.L.total = budget;  // the slots take what the budget holds
      int blocks = 0;
      s.warps = n == 1 ? kWideWarps : kShotWarps;
      QD_CK(qd::decode_occupancy(0, n, 32 * s.warps, s.L.total, &blocks));
      s.ctas = n;
      s.grid_per_sm = std::max(1, blocks);
      s.wave = typical_slots(s.L, h, s.warps);
      const int resident = std::min(blocks, n) * std::min(s.wave, kShotWarps);
      if (resident > best) {
        best = resident;
        c.best = n - 1;
        c.fits = true;
      }
    }
    // the union region in global memory: eight path slots, shared memory for
    // the persistent part only, no pre-BP staging (its copies need shared memory);
    // a shortened graph too large for that goes to the region as well
    c.Lg = lay(0, true);
    if (c.Lg.U > (unsigned)optin) c.Lg = lay(0, true, qd::kGraphGlobal);
    if (c.Lg.U > (unsigned)optin) {
      set_error(std::string(who) + ": window " + std::to_string(w) + " needs " + std::to_string(c.Lg.U) +
                " B of shared memory even with its path state in global memory (limit " +
                std::to_string(optin) + ")");
      return QD_EUNSUPPORTED;
    }
    int bg = 0;
    QD_CK(qd::decode_occupancy(c.Lg.gg == qd::kGraphGlobal ? 4 : 3, 2, 32 * kShotWarps, c.Lg.U, &bg));
    c.grid_g = std::max(1, bg);
    if (!c.fits) {  // shot mode streams the path state through L2 / HBM
      c.sh[0] = ShotShape{};
      c.sh[0].L = c.Lg;
      c.sh[0].wave = kShotWarps;
      c.sh[0].grid_per_sm = c.grid_g;
    }
    smem_max = std::max<size_t>(smem_max, c.fits ? 0u : c.Lg.U);
    for (int i = 0; i <= c.best && c.fits; ++i) smem_max = std::max<size_t>(smem_max, c.sh[i].L.total);
    for (int i = 0; i < kPathShapes; ++i) {
      PathShape& s = c.pa[i];
      const unsigned budget = smem_budget(dec, 1 << i);
      s.L = lay(budget);
      // learned weights' edge ids in global memory rather than no path mode: one
      // shot of an unshortened [[72,12,6]] (10,1) window takes 2.2 ms so, 28 in shot
      // mode with its paths in global memory
      if (i == 0 && s.L.total > budget && dec->lw_on) s.L = lay(budget, false, qd::kIdsGlobal);
      s.fits = s.L.total <= budget;
      if (!s.fits) break;
      smem_max = std::max<size_t>(smem_max, s.L.total);
      // the largest cluster (8, 4 or 2 CTAs, at most the number of paths) that
      // can be resident, its CTAs splitting the pre-BP of a shot
      for (int C = 8; C >= 2; C >>= 1) {
        if (C > nb || h.n_rows < 2 * C || h.n_cols < 2 * C) continue;
        int ncl = 0;
        if (qd::path_cluster_occupancy(kPathThreads >> i, s.L.total, C, &ncl) != cudaSuccess) {
          (void)cudaGetLastError();
          continue;
        }
        if (ncl >= 1) {
          s.pcl = C;
          break;
        }
      }
    }
  }
  for (size_t w = 0; w < cf.size(); ++w) {
    WinGpu& g = dec->wins[w];
    std::copy(cf[w].sh, cf[w].sh + kShotCtas, g.sh);
    std::copy(cf[w].pa, cf[w].pa + kPathShapes, g.pa);
    g.best = cf[w].best;
    g.Lg = cf[w].Lg;
    g.grid_g = cf[w].grid_g;
    g.fits = cf[w].fits;
  }
  QD_CK_ST(ensure_uscratch(dec, dec->launch_mode == 3));
  // shot mode's snapshot plans (one per window and shape: the first wave is a
  // typical shot's slot count) and one snapshot pool per resident CTA
  size_t cta_bytes = 0;
  int ctas = 0;
  const size_t plan = (size_t)dec->kp.nb * (3 + dec->dmx);
  ForkPlan plans[kWideWarps + 1];  // by wave
  bool have[kWideWarps + 1] = {};
  for (WinGpu& g : dec->wins) {
    std::vector<int16_t> v;
    for (int i = 0; i <= g.best; ++i) {
      ShotShape& s = g.sh[i];
      ForkPlan& F = plans[s.wave];
      if (!have[s.wave]) F = fork_plan(dec->kp, dec->dmx, s.wave);
      have[s.wave] = true;
      s.fork_on = F.on;
      s.fork_nodes = F.n_nodes;
      if (!F.on) continue;
      v.resize(plan * i);
      v.insert(v.end(), F.order.begin(), F.order.end());
      v.insert(v.end(), F.chain.begin(), F.chain.end());
      v.insert(v.end(), F.fnode.begin(), F.fnode.end());
      v.insert(v.end(), F.fdep.begin(), F.fdep.end());
      // node snapshots, then one parking snapshot per path
      cta_bytes = std::max(cta_bytes, (size_t)(F.n_nodes + dec->kp.nb) * (qd::kSnapHeaderBytes + s.L.b_size));
      ctas = std::max(ctas, dec->sm_count * std::max(s.grid_per_sm, g.grid_g));
    }
    if (v.empty()) continue;
    // a plan follows from the form, and one that a captured graph may read is
    // never written again
    int16_t*& d = g.d_fork[layout_form(dec->lw_on, hist)];
    if (!d) {
      QD_CK(cudaMalloc(&d, sizeof(int16_t) * plan * kShotCtas));
      QD_CK(cudaMemcpy(d, v.data(), sizeof(int16_t) * v.size(), cudaMemcpyHostToDevice));
    }
    for (int i = 0; i <= g.best; ++i) g.sh[i].d_fork = d + plan * i;
  }
  if (cta_bytes > dec->snap_cta_bytes || ctas > dec->snap_ctas) {
    const size_t cb = std::max(cta_bytes, dec->snap_cta_bytes);
    const int nc = std::max(ctas, dec->snap_ctas);
    QD_CK_ST(replace_buffer(dec, &dec->d_snap, cb * nc));
    dec->snap_cta_bytes = cb;
    dec->snap_ctas = nc;
  }
  if (dec->P.reuse_msgs) {  // candidate paths' kept values: one set per resident CTA, or per path-mode shot
    int cmax = 0;
    for (const WinGpu& g : dec->wins)
      for (int i = 0; i <= g.best; ++i) cmax = std::max(cmax, dec->sm_count * std::max(g.sh[i].grid_per_sm, g.grid_g));
    const size_t slots = std::max<size_t>(cmax, (size_t)std::min<long long>(dec->max_shots, kPathModeMaxShots));
    if (slots > dec->kpath_slots) {
      QD_CK_ST(replace_buffer(dec, &dec->d_kpath, sizeof(float) * slots * dec->kp.nb * std::max(1, dec->ns_max)));
      dec->kpath_slots = slots;
    }
  }
  dec->smem_max = smem_max;
  dec->hist_on = hist;
  return QD_OK;
}

// Room for `rows` iterations' learned weights of window k in the pre-BP's order;
// the first call makes room in every window, so that a decoder's weights are
// installed window by window without further allocations.  A window that needs
// more later gets at least twice as much (n_pre rows at most, which is all the
// pre-BP reads), so that the replaced buffers together are no larger than the
// last.
qd_status ensure_weight_space(qd_decoder* dec, int k, int rows) {
  for (int i = 0; i < (int)dec->wins.size(); ++i) {
    WinGpu& g = dec->wins[i];
    if (g.wts_rows >= rows || (i != k && g.wts_rows > 0)) continue;
    const int room = std::max(rows, std::min(2 * g.wts_rows, dec->kp.n_pre));
    const size_t per = 128 * (size_t)g.dv.row_quads + 32 * (size_t)g.dv.col_cells;
    QD_CK_ST(replace_buffer(dec, &g.d_wts, sizeof(float) * std::max<size_t>(per * room, 4)));
    g.wts_rows = room;
  }
  return QD_OK;
}

// Lay the windows out again when the need for the quantised history changes.
qd_status update_hist(qd_decoder* dec, const char* who) {
  const bool want = dec->kp.rkq != nullptr || dec->kp.dump != nullptr;
  if (want == dec->hist_on) return QD_OK;
  return configure_layouts(dec, want, who);
}
}  // namespace

extern "C" {

const char* qd_last_error_message(void) { return qd::g_err.c_str(); }

qd_status qd_build_dem(const qd_bb_code* code, const qd_noise* noise, qd_dem** out) {
  QD_REQ(code && noise && out, "qd_build_dem: null argument");
  QD_REQ(code->l >= 1 && code->m >= 1 && code->l * code->m <= 4096, "qd_build_dem: bad l, m");
  QD_REQ(noise->rounds >= 1 && noise->rounds <= 1000, "qd_build_dem: bad rounds");
  QD_REQ(noise->p > 0.0 && noise->p < 0.5, "qd_build_dem: p outside (0, 0.5)");
  std::unique_ptr<qd_dem> d(new (std::nothrow) qd_dem());
  if (!d) return QD_ENOMEM;
  if (!qd::build_dem_host(*code, *noise, d->h)) return QD_EINVAL;
  for (float l : d->h.col_llr)
    if (!(l > std::ldexp(1.0f, -15) && l < 16.0f)) {
      set_error("qd_build_dem: prior LLR outside (2^-15, 16); Eq. (5) would not be exact");
      return QD_EUNSUPPORTED;
    }
  *out = d.release();
  return QD_OK;
}

qd_status qd_build_dem_code_capacity(const qd_bb_code* code, double p_data, double p_synd, qd_dem** out) {
  QD_REQ(code && out, "qd_build_dem_code_capacity: null argument");
  QD_REQ(code->l >= 1 && code->m >= 1 && code->l * code->m <= 4096, "qd_build_dem_code_capacity: bad l, m");
  QD_REQ(p_data > 0.0 && p_data < 0.5, "qd_build_dem_code_capacity: p_data outside (0, 0.5)");
  QD_REQ(p_synd >= 0.0 && p_synd < 0.5, "qd_build_dem_code_capacity: p_synd outside [0, 0.5)");
  std::unique_ptr<qd_dem> d(new (std::nothrow) qd_dem());
  if (!d) return QD_ENOMEM;
  if (!qd::build_dem_code_capacity(*code, p_data, p_synd, d->h)) return QD_EINVAL;
  for (float l : d->h.col_llr)
    if (!(l > std::ldexp(1.0f, -15) && l < 16.0f)) {
      set_error("qd_build_dem_code_capacity: prior LLR outside (2^-15, 16); Eq. (5) would not be exact");
      return QD_EUNSUPPORTED;
    }
  *out = d.release();
  return QD_OK;
}

qd_status qd_dem_info(const qd_dem* d, qd_dem_info_t* o) {
  QD_REQ(d && o, "qd_dem_info: null argument");
  o->n_det = d->h.n_det;
  o->n_cols = d->h.n_cols;
  o->n_obs = d->h.K;
  o->n_blocks = d->h.R + 1;
  o->w = d->h.w;
  o->det_words = (d->h.n_det + 31) / 32;
  o->n_edges = (int)d->h.col_dets.size();
  return QD_OK;
}

qd_status qd_dem_columns(const qd_dem* d, int* col_ptr, int* col_dets, uint32_t* obs, double* prob,
                         float* llr) {
  QD_REQ(d, "qd_dem_columns: null dem");
  const auto& h = d->h;
  if (col_ptr) std::copy(h.col_ptr.begin(), h.col_ptr.end(), col_ptr);
  if (col_dets) std::copy(h.col_dets.begin(), h.col_dets.end(), col_dets);
  if (obs) std::copy(h.col_obs.begin(), h.col_obs.end(), obs);
  if (prob) std::copy(h.col_p.begin(), h.col_p.end(), prob);
  if (llr) std::copy(h.col_llr.begin(), h.col_llr.end(), llr);
  return QD_OK;
}

qd_status qd_dem_window(const qd_dem* d, int W, int F, int k, int merge_h1, int info[7], int* gcols, int* col_ptr,
                        int* col_rows, float* llr) {
  QD_REQ(d && info, "qd_dem_window: null argument");
  QD_REQ(W >= 1 && F >= 1 && F <= W, "qd_dem_window: need 1 <= F <= W");
  QD_REQ(k >= 0 && k < qd::n_windows(d->h, W, F), "qd_dem_window: window out of range");
  QD_REQ(merge_h1 >= 0 && merge_h1 <= 2, "qd_dem_window: merge_h1 must be 0, 1 or 2");
  qd::WindowHost h;
  if (!qd::build_window(d->h, W, F, k, false, h, merge_h1)) return QD_EINVAL;
  const int v[7] = {h.r0, h.n_blocks, h.n_rows, h.n_cols, h.n_edges, h.n_commit, h.last};
  std::copy(v, v + 7, info);
  if (gcols) {
    std::copy(h.gcols.begin(), h.gcols.end(), gcols);
    std::copy(h.col_ptr.begin(), h.col_ptr.end(), col_ptr);
    std::copy(h.col_rows.begin(), h.col_rows.end(), col_rows);
    std::copy(h.llr.begin(), h.llr.end(), llr);
  }
  return QD_OK;
}

qd_status qd_path_plan(const qd_gdg_params* p, int wave, int info[3], int16_t* order, int16_t* chain, int16_t* fnode,
                       int16_t* fdep) {
  QD_REQ(p && info, "qd_path_plan: null argument");
  QD_REQ(p->k_guess >= 0 && p->k_guess <= 5 && wave >= 1, "qd_path_plan: k_guess outside [0, 5] or wave < 1");
  QD_REQ(p->side_max == 0 || (p->side_max >= p->k_guess && p->side_max <= 32), "qd_path_plan: bad side_max");
  qd::KParams k{};
  k.dmax_main = p->d_max_main;
  k.dmax_other = p->d_max_other;
  k.k = p->k_guess;
  k.low_err = p->low_error_mode;
  k.side_max = p->side_max;
  k.reinit = p->reinit_on_split != 0;
  k.nb = (1 << p->k_guess) + (p->side_max > p->k_guess ? p->side_max - p->k_guess : 0);
  int dmx = 0;
  for (int id = 0; id < k.nb; ++id) dmx = std::max(dmx, qd::path_dmax(k, id, qd::path_split(k, id)));
  const ForkPlan F = fork_plan(k, dmx, wave);
  info[0] = k.nb;
  info[1] = dmx;
  info[2] = F.on ? F.n_nodes : -1;
  if (F.on && order) {
    std::copy(F.order.begin(), F.order.end(), order);
    std::copy(F.chain.begin(), F.chain.end(), chain);
    std::copy(F.fnode.begin(), F.fnode.end(), fnode);
    std::copy(F.fdep.begin(), F.fdep.end(), fdep);
  }
  return QD_OK;
}

qd_status qd_dem_destroy(qd_dem* d) {
  if (!d) return QD_OK;
  if (d->d_thr) {
    cudaFree(d->d_cptr);
    cudaFree(d->d_cdet);
    cudaFree(d->d_cobs);
    cudaFree(d->d_thr);
  }
  delete d;
  return QD_OK;
}

qd_status qd_sample_shots(const qd_dem* d, uint64_t seed, uint64_t shot_offset, int64_t n_shots,
                          uint32_t* det_bits, uint32_t* obs_bits, qd_stream_t stream) {
  QD_REQ(d && det_bits && obs_bits, "qd_sample_shots: null argument");
  QD_REQ(n_shots >= 0, "qd_sample_shots: n_shots < 0");
  if (qd_status st = ensure_device(d)) return st;
  QD_CK(qd::launch_sample((cudaStream_t)stream, d->h.n_cols, d->d_thr, d->d_cptr, d->d_cdet, d->d_cobs,
                          (d->h.n_det + 31) / 32, seed, shot_offset, n_shots, det_bits, obs_bits));
  return QD_OK;
}

qd_status qd_decoder_destroy(qd_decoder* dec) {
  if (!dec) return QD_OK;
  for (auto& w : dec->wins) {
    cudaFree(w.d_graph);
    cudaFree(w.d_ccptr);
    cudaFree(w.d_ccdet);
    cudaFree(w.d_ccobs);
    cudaFree(w.d_wthr);
    for (int16_t* p : w.d_fork) cudaFree(p);
    cudaFree(w.d_prev);
    cudaFree(w.d_wts);
  }
  cudaFree(dec->d_snap);
  cudaFree(dec->d_keep);
  cudaFree(dec->d_kpath);
  cudaFree(dec->d_work);
  cudaFree(dec->d_uscratch);
  cudaFree(dec->d_ranker);
  cudaFree(dec->d_path_res);
  cudaFree(dec->d_arrive);
  cudaFree(dec->d_counters);
  cudaFree(dec->d_corr);
  cudaFree(dec->d_det);
  cudaFree(dec->d_obs);
  cudaFree(dec->d_pred);
  cudaFree(dec->d_fail);
  cudaFree(dec->d_resid);
  cudaFree(dec->d_nfail);
  for (void* p : dec->retired) cudaFree(p);
  delete dec;
  return QD_OK;
}

qd_status qd_decoder_create(const qd_dem* dem, const qd_gdg_params* p, int64_t max_shots,
                            qd_decoder** out) {
  QD_REQ(dem && p && out, "qd_decoder_create: null argument");
  QD_REQ(max_shots >= 1, "qd_decoder_create: max_shots < 1");
  QD_REQ(p->W >= 1 && p->F >= 1 && p->F <= p->W, "qd_decoder_create: need 1 <= F <= W");
  QD_REQ(p->n_pre >= 0 && p->iters_per_step >= 1 && p->d_max_main >= 1 && p->d_max_other >= 1,
         "qd_decoder_create: bad iteration counts");
  QD_REQ(p->alpha > 0.0f && p->clip > 0.0f, "qd_decoder_create: alpha and clip must be positive");
  if (p->iters_per_step < 4 || (p->iters_first != 0 && p->iters_first < 4)) {
    set_error("qd_decoder_create: iters_per_step or iters_first < 4 is not implemented on the GPU");
    return QD_EUNSUPPORTED;
  }
  QD_REQ(p->iters_first >= 0, "qd_decoder_create: iters_first < 0");
  QD_REQ(p->merge_h1 >= 0 && p->merge_h1 <= 2, "qd_decoder_create: merge_h1 must be 0, 1 or 2");
  QD_REQ(p->reuse_msgs == 0 || p->reuse_msgs == 1, "qd_decoder_create: reuse_msgs must be 0 or 1");
  QD_REQ(p->fallback >= 0 && p->fallback <= 2, "qd_decoder_create: fallback must be 0, 1 or 2");
  QD_REQ(p->side_max == 0 || (p->side_max >= p->k_guess && p->side_max <= 32),
         "qd_decoder_create: side_max must be 0 or in [k_guess, 32]");
  QD_REQ(p->d_max_other >= p->k_guess, "qd_decoder_create: d_max_other < k_guess");
  if (p->k_guess < 0 || p->k_guess > 5) {
    set_error("qd_decoder_create: k_guess must be in [0, 5]");
    return QD_EUNSUPPORTED;
  }
  if (qd_status st = ensure_device(dem)) return st;
  std::unique_ptr<qd_decoder> dec(new (std::nothrow) qd_decoder());
  if (!dec) return QD_ENOMEM;
  dec->dem = dem;
  dec->P = *p;
  dec->max_shots = max_shots;
  qd::KParams& k = dec->kp;
  k.alpha = p->alpha;
  k.clip = p->clip;
  k.pa_main = p->pa_main;
  k.pa_other = p->pa_other;
  k.pb_main = p->pb_main;
  k.pb_other = p->pb_other;
  k.pb_d1 = p->pb_d1;
  k.pc = p->pc;
  k.pd = p->pd;
  k.n_pre = p->n_pre;
  k.ips = p->iters_per_step;
  k.ips1 = p->iters_first;
  k.fallback = p->fallback;
  k.dmax_main = p->d_max_main;
  k.dmax_other = p->d_max_other;
  k.k = p->k_guess;
  k.low_err = p->low_error_mode;
  k.peel_init = p->peel_at_init;
  k.pc_max_depth = p->pc_max_depth;
  k.n_unsat_min = p->n_unsat_min;
  k.side_max = p->side_max;
  k.reinit = p->reinit_on_split != 0;
  k.nb = (1 << p->k_guess) + (p->side_max > p->k_guess ? p->side_max - p->k_guess : 0);
  dec->dmx = 0;  // the deepest path, by the kernels' own rule (trace sizing)
  for (int id = 0; id < k.nb; ++id) dec->dmx = std::max(dec->dmx, qd::path_dmax(k, id, qd::path_split(k, id)));

  int dev = 0, optin = 0;
  QD_CK(cudaGetDevice(&dev));
  QD_CK(cudaDeviceGetAttribute(&dec->sm_count, cudaDevAttrMultiProcessorCount, dev));
  QD_CK(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));

  const int nwin = qd::n_windows(dem->h, p->W, p->F);
  dec->wins.resize(nwin);
  for (int w = 0; w < nwin; ++w) {
    WinGpu& g = dec->wins[w];
    if (!qd::build_window(dem->h, p->W, p->F, w, p->shorten != 0, g.h, p->merge_h1)) return QD_EINVAL;
    const auto& h = g.h;
    dec->corr_words = std::max(dec->corr_words, (h.n_cols + 31) / 32);
    dec->ns_max = std::max(dec->ns_max, h.n_short);
    dec->sw_max = std::max(dec->sw_max, (h.n_short + 31) / 32);
    if (!qd::build_slices(g.h, w ? &dec->wins[w - 1].h : nullptr)) return QD_EUNSUPPORTED;
    Blob blob;
    auto put = [&](const auto& v) { return blob.put(v); };
    const size_t o_cp = put(h.col_ptr), o_cr = put(h.col_rows), o_rp = put(h.row_ptr), o_re = put(h.row_ent),
                 o_ll = put(h.llr), s_re = put(h.s_rent), s_ce = put(h.s_cent), s_ro = put(h.s_roff),
                 s_co = put(h.s_coff), s_ll = put(h.s_llr), s_rw = put(h.s_row), s_cl = put(h.s_col),
                 s_rf = put(h.s_ref), s_cf = put(h.s_cef);
    QD_CK(blob.upload(&g.d_graph));
    char* b = g.d_graph;
    g.dv = qd::WinDev{h.n_rows, h.n_cols, h.n_edges, h.row0, h.n_short, h.short_edges_max, h.n_rows / h.n_blocks,
                      (const uint16_t*)(b + o_cp), (const uint16_t*)(b + o_cr), (const uint16_t*)(b + o_rp),
                      (const uint32_t*)(b + o_re), (const float*)(b + o_ll), nullptr, 0, 0, nullptr, nullptr,
                      h.last ? h.n_rows : std::min(h.n_rows, dec->P.F * (h.n_rows / h.n_blocks)),
                      h.row_quads, h.col_cells, (const uint16_t*)(b + s_re), (const uint32_t*)(b + s_ce),
                      (const uint16_t*)(b + s_ro), (const uint16_t*)(b + s_co), (const float*)(b + s_ll),
                      (const uint16_t*)(b + s_rw), (const uint16_t*)(b + s_cl),
                      qd::ColClasses{h.cls[0], h.cls[1], h.cls[2], h.cls[3]}, (const uint16_t*)(b + s_rf),
                      (const uint16_t*)(b + s_cf)};
    // committed columns: their full detector sets and observables
    std::vector<int> cc_ptr(1, 0), cc_det;
    std::vector<uint32_t> cc_obs;
    for (int c = 0; c < h.n_commit; ++c) {
      int gc = h.gcols[c];
      for (int e = dem->h.col_ptr[gc]; e < dem->h.col_ptr[gc + 1]; ++e) cc_det.push_back(dem->h.col_dets[e]);
      cc_ptr.push_back((int)cc_det.size());
      cc_obs.push_back(dem->h.col_obs[gc]);
    }
    QD_CK(upload(&g.d_ccptr, cc_ptr));
    QD_CK(upload(&g.d_ccdet, cc_det));
    QD_CK(upload(&g.d_ccobs, cc_obs));
  }
  dec->smem_optin = optin;
  QD_CK(cudaDeviceGetAttribute(&dec->smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
  QD_CK(cudaDeviceGetAttribute(&dec->smem_reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev));
  // the kernels' dynamic shared-memory allowance is the device limit, so
  // decoders of different sizes coexist (the launch asks for what it needs)
  QD_CK(qd::set_decode_smem((size_t)optin));
  if (qd_status st = configure_layouts(dec.get(), false, "qd_decoder_create")) return st;
  dec->trace_bytes = qd::trace_bytes_per_shot(k.nb, dec->dmx, dec->ns_max);
  QD_CK(cudaMalloc(&dec->d_work, sizeof(int) * (nwin + 1)));
  const long long pm_shots = std::min<long long>(max_shots, kPathModeMaxShots);
  QD_CK(cudaMalloc(&dec->d_path_res, qd::path_result_bytes(dec->sw_max) * k.nb * pm_shots));
  QD_CK(cudaMalloc(&dec->d_arrive, sizeof(int) * pm_shots));
  QD_CK(cudaMemset(dec->d_arrive, 0, sizeof(int) * pm_shots));
  QD_CK(cudaMalloc(&dec->d_counters, sizeof(long long) * kCounters));
  QD_CK(cudaMemset(dec->d_counters, 0, sizeof(long long) * kCounters));
  const int dw = (dem->h.n_det + 31) / 32;
  QD_CK(cudaMalloc(&dec->d_corr, sizeof(uint32_t) * (size_t)max_shots * dec->corr_words));
  QD_CK(cudaMalloc(&dec->d_det, sizeof(uint32_t) * (size_t)max_shots * dw));
  QD_CK(cudaMalloc(&dec->d_obs, sizeof(uint32_t) * (size_t)max_shots));
  QD_CK(cudaMalloc(&dec->d_pred, sizeof(uint32_t) * (size_t)max_shots));
  QD_CK(cudaMalloc(&dec->d_fail, sizeof(uint32_t) * (size_t)max_shots));
  QD_CK(cudaMalloc(&dec->d_resid, sizeof(uint32_t) * (size_t)max_shots));
  QD_CK(cudaMalloc(&dec->d_nfail, sizeof(long long)));
  if (p->reuse_msgs) {
    for (const WinGpu& g : dec->wins) dec->keep_ld = std::max(dec->keep_ld, g.h.n_cols);
    QD_CK(cudaMalloc(&dec->d_keep, sizeof(float) * (size_t)max_shots * std::max(1, dec->keep_ld)));
    for (int w = 1; w < nwin; ++w) {
      const auto& a = dec->wins[w - 1].h;
      const auto& b = dec->wins[w].h;
      if (!a.n_cols || !b.n_cols) continue;  // nothing kept across a window without columns
      std::vector<int> at(dem->h.n_cols, -1);
      for (int c = 0; c < a.n_cols; ++c) at[a.gcols[c]] = c;  // a repeated DEM column: its last column
      std::vector<int16_t> prev(b.n_cols);
      for (int c = 0; c < b.n_cols; ++c) prev[c] = (int16_t)at[b.gcols[c]];
      QD_CK(upload(&dec->wins[w].d_prev, prev));
    }
  }
  *out = dec.release();
  return QD_OK;
}

qd_status qd_decoder_n_windows(const qd_decoder* dec, int* n) {
  QD_REQ(dec && n, "null argument");
  *n = (int)dec->wins.size();
  return QD_OK;
}

qd_status qd_decoder_path_info(const qd_decoder* dec, int out[2]) {
  QD_REQ(dec && out, "null argument");
  out[0] = dec->kp.nb;
  out[1] = dec->dmx;
  return QD_OK;
}

qd_status qd_decoder_corr_words(const qd_decoder* dec, int* cw) {
  QD_REQ(dec && cw, "null argument");
  *cw = dec->corr_words;
  return QD_OK;
}

qd_status qd_decoder_trace_bytes(const qd_decoder* dec, size_t* b) {
  QD_REQ(dec && b, "null argument");
  *b = dec->trace_bytes;
  return QD_OK;
}

qd_status qd_window_info(const qd_decoder* dec, int k, qd_window_info_t* o, int* gcols) {
  QD_REQ(dec && o, "null argument");
  QD_REQ(k >= 0 && k < (int)dec->wins.size(), "qd_window_info: window out of range");
  const auto& h = dec->wins[k].h;
  *o = qd_window_info_t{h.r0, h.n_blocks, h.n_rows, h.n_cols, h.n_edges, h.n_commit, h.last, h.n_short};
  if (gcols) std::copy(h.gcols.begin(), h.gcols.end(), gcols);
  return QD_OK;
}

}  // extern "C"

namespace {
// message reuse buffers for window g (keep = nullptr: off)
qd::ReuseDev reuse_dev(const qd_decoder* dec, const WinGpu& g) {
  qd::ReuseDev R{};
  if (!dec->d_keep) return R;
  R.keep = dec->d_keep;
  R.keep_ld = dec->keep_ld;
  R.prev = g.d_prev;
  R.kpath = dec->d_kpath;
  return R;
}

// Path mode's CTA for n_shots shots of window g, as an index into g.pa; -1: shot
// mode.  Path mode runs batches of up to 64 shots.  A path's serial chain is
// what takes the time and 512 threads shorten it most, but only one such CTA
// fits an SM; a batch of several CTAs per SM is faster with smaller ones side by
// side.  Four CTAs of 128 threads pay from three per SM, and a window of at most
// 128 checks gains nothing from more than 256 threads (two lanes per check).
// Every cluster of a shot repeats the pre-BP, so a long one (100 iterations in all
// the figures, against 8 and 16; no preset lies between) with more than nine paths
// per SM is left to shot mode (32 paths, configured: [[144]] W = 4, 38 shots
// 22.9 ms against 28.1 in shot mode, 45 28.6 / 28.6, 64 36.3 / 29.0; 22 paths of the
// paper preset on [[288]] W = 4, 64 shots 13.5 / 23.3).
// All windows of a pass, ms, with 512 x 1 / 256 x 2 / 128 x 4 and in shot mode:
// [[144,12,12]] configured, 2 shots 6.4 / 6.4 / 8.2 / 15.2, 19 shots 16.1 / 9.8 /
// 11.2 / 20.9, 38 shots 26.2 / 15.8 / 12.6 / 18.0, 64 shots 40.3 / 24.4 / 19.6 /
// 18.4; paper preset, 25 shots 6.1 / 4.5 / 5.0 / 11.1, 64 shots 12.5 / 7.8 / 7.0 /
// 12.2; [[72,12,6]], 2 shots 2.45 / 2.26 / 2.47 / 3.9, 64 shots 6.5 / 4.5 / 3.7 /
// 5.0.  (64 configured [[144,12,12]] shots, 6.7 paths per SM, would be 6 % faster
// in shot mode, 64 of the paper preset 1.7 times as slow.)
int path_shape(const qd_decoder* dec, const WinGpu& g, int64_t n_shots) {
  bool path_mode = dec->launch_mode == 2;
  if (dec->launch_mode == 0)
    path_mode = n_shots * 2 <= dec->sm_count &&
                (dec->kp.n_pre < 32 || n_shots * dec->kp.nb <= 9LL * dec->sm_count);
  if (!path_mode || n_shots > std::min<long long>(dec->max_shots, kPathModeMaxShots) || !g.pa[0].fits ||
      (!g.fits && g.pa[0].L.gg != qd::kIdsGlobal))
    return -1;
  int i = 0;
  const long long ctas = n_shots * dec->kp.nb;
  if (g.pa[1].fits && (g.h.n_rows <= 128 || ctas > dec->sm_count)) i = 1;
  if (g.pa[2].fits && ctas > 3LL * dec->sm_count) i = 2;
  return i;
}

// Shot mode for n_shots shots: the fewest CTAs per SM that hold them at once
// (more shared memory, so more path slots and staged graph, and more registers),
// else the large batches'.  150 shots of [[144,12,12]], all windows: configured
// 22.0 ms in the large batches' shape, 18.8 with one CTA per SM; paper preset 14.0
// and 11.2.
const ShotShape& shot_shape(const qd_decoder* dec, const WinGpu& g, int64_t n_shots) {
  int i = 0;
  while (i < g.best && n_shots > (int64_t)(i + 1) * dec->sm_count) ++i;
  return g.sh[i];
}

// shot mode's snapshot plan (pool = nullptr: none, or turned off)
qd::ForkDev fork_dev(const qd_decoder* dec, const ShotShape& g) {
  qd::ForkDev F{};
  // the candidate dump records path 0's every step, so path 0 runs from the root
  if (!dec->fork_on || !g.fork_on || !dec->d_snap || dec->kp.dump) return F;
  const int nb = dec->kp.nb;
  F.order = g.d_fork;
  F.chain = g.d_fork + nb;
  F.fnode = F.chain + (size_t)nb * dec->dmx;
  F.fdep = F.fnode + nb;
  F.pool = dec->d_snap;
  F.cta_bytes = dec->snap_cta_bytes;
  F.n_nodes = g.fork_nodes;
  F.pool_ctas = dec->snap_ctas;
  F.sched = dec->sched_on ? 1 : 0;
  return F;
}
}  // namespace

extern "C" {

qd_status qd_decode_windows(qd_decoder* dec, int k, const uint32_t* det_bits, int64_t n_shots,
                            uint32_t* win_correction, int32_t* status, void* trace, qd_stream_t stream) {
  QD_REQ(dec && det_bits && win_correction, "qd_decode_windows: null argument");
  QD_REQ(k >= 0 && k < (int)dec->wins.size(), "qd_decode_windows: window out of range");
  QD_REQ(n_shots >= 0 && n_shots <= dec->max_shots, "qd_decode_windows: n_shots outside [0, max_shots]");
  if (n_shots == 0) return QD_OK;
  const WinGpu& g = dec->wins[k];
  cudaStream_t st = (cudaStream_t)stream;
  const int dw = (dec->dem->h.n_det + 31) / 32;
  if (g.h.n_cols == 0) {
    // a window without columns decides nothing (the commit tests its residue)
    QD_CK(cudaMemsetAsync(win_correction, 0, sizeof(uint32_t) * (size_t)n_shots * dec->corr_words, st));
    if (status) QD_CK(cudaMemsetAsync(status, 0xFF, sizeof(int32_t) * (size_t)n_shots, st));
    return QD_OK;
  }
  // the path state in global memory when the window does not fit shared memory
  // (or on request)
  const int ps = path_shape(dec, g, n_shots);
  const bool global = ps < 0 && (!g.fits || dec->launch_mode == 3);
  const ShotShape& s = shot_shape(dec, g, global ? INT64_MAX : n_shots);
  const qd::ForkDev fk = fork_dev(dec, s);
  const qd::ReuseDev ru = reuse_dev(dec, g);
  if (g.dv.wts) QD_CK(qd::launch_order_weights(st, g.dv));
  if (global) {
    QD_CK(cudaMemsetAsync(dec->d_work + k, 0, sizeof(int), st));
    const long long grid = std::min<long long>(n_shots, (long long)dec->sm_count * g.grid_g);
    QD_CK(qd::launch_decode(0, 2, (int)grid, 32 * kShotWarps, g.Lg.U, st, dec->kp, g.dv, g.Lg, det_bits, dw, n_shots,
                            win_correction, dec->corr_words, status, (char*)trace, dec->trace_bytes, dec->dmx,
                            dec->ns_max, dec->d_work + k, dec->d_counters, nullptr, nullptr, dec->sw_max,
                            dec->d_uscratch, g.Lg.total - g.Lg.U, 1, 1, &fk, &ru));
    return QD_OK;
  }
  if (ps >= 0) {
    const PathShape& p = g.pa[ps];
    const int cps = path_ctas(dec, p);
    QD_CK(qd::launch_decode(1, 1, (int)(n_shots * cps), kPathThreads >> ps, p.L.total, st, dec->kp, g.dv, p.L,
                            det_bits, dw, n_shots, win_correction, dec->corr_words, status, (char*)trace,
                            dec->trace_bytes, dec->dmx, dec->ns_max, nullptr, dec->d_counters, dec->d_path_res,
                            dec->d_arrive, dec->sw_max, p.L.ids ? dec->d_uscratch : nullptr, p.L.ids, cps,
                            p.pcl, nullptr, &ru));
    return QD_OK;
  }
  QD_CK(cudaMemsetAsync(dec->d_work + k, 0, sizeof(int), st));
  const long long grid = std::min<long long>(n_shots, (long long)dec->sm_count * s.grid_per_sm);
  QD_CK(qd::launch_decode(0, s.ctas, (int)grid, 32 * s.warps, s.L.total, st, dec->kp, g.dv, s.L, det_bits, dw,
                          n_shots, win_correction, dec->corr_words, status, (char*)trace, dec->trace_bytes,
                          dec->dmx, dec->ns_max, dec->d_work + k, dec->d_counters, nullptr, nullptr, dec->sw_max,
                          nullptr, 0, 1, 1, &fk, &ru));
  return QD_OK;
}

qd_status qd_commit_and_slide(qd_decoder* dec, int k, const uint32_t* win_correction, int64_t n_shots,
                              uint32_t* det_bits, uint32_t* obs_pred, uint32_t* residue_fail,
                              qd_stream_t stream) {
  QD_REQ(dec && win_correction && det_bits && obs_pred && residue_fail, "qd_commit_and_slide: null argument");
  QD_REQ(k >= 0 && k < (int)dec->wins.size(), "qd_commit_and_slide: window out of range");
  QD_REQ(n_shots >= 0, "qd_commit_and_slide: n_shots < 0");
  const WinGpu& g = dec->wins[k];
  const int w = dec->dem->h.w;
  QD_CK(qd::launch_commit((cudaStream_t)stream, g.h.n_commit, g.d_ccptr, g.d_ccdet, g.d_ccobs,
                          dec->corr_words, win_correction, n_shots, det_bits, (dec->dem->h.n_det + 31) / 32,
                          obs_pred, residue_fail, g.h.r0 * w, g.h.commit_b1 * w));
  return QD_OK;
}

qd_status qd_evaluate(const uint32_t* obs_pred, const uint32_t* obs_true, const uint32_t* residue_fail,
                      int64_t n_shots, uint32_t* fail, long long* n_fail, qd_stream_t stream) {
  QD_REQ(obs_pred && obs_true && residue_fail, "qd_evaluate: null argument");
  QD_REQ(n_shots >= 0, "qd_evaluate: n_shots < 0");
  QD_CK(qd::launch_evaluate((cudaStream_t)stream, obs_pred, obs_true, residue_fail, n_shots, fail, n_fail));
  return QD_OK;
}

qd_status qd_decode_all(qd_decoder* dec, uint32_t* det_bits, const uint32_t* obs_true, int64_t n_shots,
                        uint32_t* obs_pred, uint32_t* fail, long long* n_fail, qd_stream_t stream) {
  QD_REQ(dec && det_bits && obs_true && obs_pred, "qd_decode_all: null argument");
  QD_REQ(n_shots >= 0 && n_shots <= dec->max_shots, "qd_decode_all: n_shots outside [0, max_shots]");
  if (n_shots == 0) return QD_OK;
  cudaStream_t st = (cudaStream_t)stream;
  QD_CK(cudaMemsetAsync(obs_pred, 0, sizeof(uint32_t) * n_shots, st));
  QD_CK(cudaMemsetAsync(dec->d_resid, 0, sizeof(uint32_t) * n_shots, st));
  for (int k = 0; k < (int)dec->wins.size(); ++k) {
    qd_status s = qd_decode_windows(dec, k, det_bits, n_shots, dec->d_corr, nullptr, nullptr, stream);
    if (s != QD_OK) return s;
    s = qd_commit_and_slide(dec, k, dec->d_corr, n_shots, det_bits, obs_pred, dec->d_resid, stream);
    if (s != QD_OK) return s;
  }
  return qd_evaluate(obs_pred, obs_true, dec->d_resid, n_shots, fail, n_fail, stream);
}

qd_status qd_decode_shots_host(qd_decoder* dec, const uint32_t* det_bits, const uint32_t* obs_true,
                               int64_t n_shots, uint32_t* obs_pred, uint32_t* fail, long long* n_fail,
                               qd_stream_t stream) {
  QD_REQ(dec && det_bits && obs_true, "qd_decode_shots_host: null argument");
  QD_REQ(n_shots >= 0 && n_shots <= dec->max_shots, "qd_decode_shots_host: n_shots outside [0, max_shots]");
  if (n_shots == 0) return QD_OK;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t dw = (dec->dem->h.n_det + 31) / 32;
  QD_CK(cudaMemcpyAsync(dec->d_det, det_bits, sizeof(uint32_t) * dw * n_shots, cudaMemcpyHostToDevice, st));
  QD_CK(cudaMemcpyAsync(dec->d_obs, obs_true, sizeof(uint32_t) * n_shots, cudaMemcpyHostToDevice, st));
  QD_CK(cudaMemsetAsync(dec->d_nfail, 0, sizeof(long long), st));
  qd_status s = qd_decode_all(dec, dec->d_det, dec->d_obs, n_shots, dec->d_pred, dec->d_fail, dec->d_nfail, stream);
  if (s != QD_OK) return s;
  if (obs_pred)
    QD_CK(cudaMemcpyAsync(obs_pred, dec->d_pred, sizeof(uint32_t) * n_shots, cudaMemcpyDeviceToHost, st));
  if (fail) QD_CK(cudaMemcpyAsync(fail, dec->d_fail, sizeof(uint32_t) * n_shots, cudaMemcpyDeviceToHost, st));
  if (n_fail) QD_CK(cudaMemcpyAsync(n_fail, dec->d_nfail, sizeof(long long), cudaMemcpyDeviceToHost, st));
  QD_CK(cudaStreamSynchronize(st));
  return QD_OK;
}

qd_status qd_decoder_set_weights(qd_decoder* dec, int k, const float* w, int T) {
  QD_REQ(dec, "null argument");
  QD_REQ(k >= 0 && k < (int)dec->wins.size(), "qd_decoder_set_weights: window out of range");
  QD_REQ(w == nullptr || T >= 1, "qd_decoder_set_weights: T must be >= 1");
  const int rows = std::min(T, dec->kp.n_pre);  // that the pre-BP reads
  if (w) QD_CK_ST(ensure_weight_space(dec, k, rows));
  const qd::WinDev old = dec->wins[k].dv;
  WinGpu& g = dec->wins[k];
  g.dv.wts = w;
  g.dv.wT = w ? T : 0;
  g.dv.w_rows = w ? rows : 0;
  g.dv.w_row = w ? g.d_wts : nullptr;
  g.dv.w_col = w ? g.d_wts + (size_t)rows * 128 * g.dv.row_quads : nullptr;
  // the layouts keep the shortened edges' full-window ids only while some
  // window has learned weights
  bool want = false;
  for (const WinGpu& g : dec->wins) want = want || g.dv.wts != nullptr;
  if (want != dec->lw_on) {
    dec->lw_on = want;
    if (qd_status st = configure_layouts(dec, dec->hist_on, "qd_decoder_set_weights")) {
      g.dv = old;
      dec->lw_on = !want;
      return st;
    }
  }
  return QD_OK;
}

qd_status qd_decoder_set_ranker(qd_decoder* dec, const float* params) {
  QD_REQ(dec, "null argument");
  if (!params) {
    dec->kp.rkq = nullptr;
    dec->kp.rkb = nullptr;
    return update_hist(dec, "qd_decoder_set_ranker");
  }
  // the grids of the exact first layer (the same rule as the reference model)
  auto grid = [](float x, float scale, float lim) {
    float v = std::rint(x * scale);
    v = v > lim ? lim : (v < -lim ? -lim : v);
    return v / scale;
  };
  std::vector<float> q(644, 0.0f);
  for (int i = 0; i < 641; ++i)
    QD_REQ(std::isfinite(params[i]), "qd_decoder_set_ranker: non-finite parameter");
  for (int i = 0; i < 512; ++i) q[i] = grid(params[i], 64.0f, 128.0f);
  for (int u = 0; u < 64; ++u) q[512 + u] = grid(params[512 + u], 128.0f, 65536.0f);
  for (int u = 0; u < 64; ++u) q[576 + u] = grid(params[576 + u], 64.0f, 128.0f);
  q[640] = params[640];
  std::vector<uint32_t> frag(256);
  for (int t = 0; t < 8; ++t)
    for (int lane = 0; lane < 32; ++lane) {
      const int u = 8 * t + lane / 4, kk = 2 * (lane % 4);
      uint32_t lo, hi;
      memcpy(&lo, &q[u * 8 + kk], 4);
      memcpy(&hi, &q[u * 8 + kk + 1], 4);
      frag[32 * t + lane] = (lo >> 16) | (hi & 0xFFFF0000u);  // exact: 7 significant bits
    }
  if (!dec->d_ranker) QD_CK(cudaMalloc(&dec->d_ranker, 644 * 4 + 256 * 4));
  QD_CK(cudaMemcpy(dec->d_ranker, q.data(), 644 * 4, cudaMemcpyHostToDevice));
  QD_CK(cudaMemcpy((char*)dec->d_ranker + 644 * 4, frag.data(), 256 * 4, cudaMemcpyHostToDevice));
  const float* old_q = dec->kp.rkq;
  const uint32_t* old_b = dec->kp.rkb;
  dec->kp.rkq = (const float*)dec->d_ranker;
  dec->kp.rkb = (const uint32_t*)((char*)dec->d_ranker + 644 * 4);
  if (qd_status st = update_hist(dec, "qd_decoder_set_ranker")) {
    dec->kp.rkq = old_q;
    dec->kp.rkb = old_b;
    return st;
  }
  return QD_OK;
}

qd_status qd_decoder_set_dump(qd_decoder* dec, void* records, int* count, int capacity) {
  QD_REQ(dec, "null argument");
  QD_REQ(!records || (count && capacity >= 0), "qd_decoder_set_dump: need count and capacity >= 0");
  dec->kp.dump = (qd::RankRec*)records;
  dec->kp.dump_n = records ? count : nullptr;
  dec->kp.dump_cap = records ? capacity : 0;
  if (qd_status st = update_hist(dec, "qd_decoder_set_dump")) {
    dec->kp.dump = nullptr;
    dec->kp.dump_n = nullptr;
    dec->kp.dump_cap = 0;
    return st;
  }
  return QD_OK;
}

qd_status qd_decoder_launch_info(const qd_decoder* dec, int k, int out[8]) {
  QD_REQ(dec && out, "null argument");
  QD_REQ(k >= 0 && k < (int)dec->wins.size(), "qd_decoder_launch_info: window out of range");
  const WinGpu& g = dec->wins[k];
  const ShotShape& s = g.sh[g.best];
  const PathShape& p = g.pa[0];
  out[0] = (int)s.L.total;
  out[1] = 32 * s.warps;
  out[2] = s.grid_per_sm;
  out[3] = (int)p.L.total;
  out[4] = kPathThreads;
  out[5] = dec->sm_count;
  out[6] = p.pcl;
  out[7] = path_ctas(dec, p);
  return QD_OK;
}

qd_status qd_decoder_set_launch(qd_decoder* dec, int mode) {
  QD_REQ(dec, "null argument");
  QD_REQ(mode >= 0 && mode <= 3, "qd_decoder_set_launch: mode must be 0, 1, 2 or 3");
  if (mode == 3) QD_CK_ST(ensure_uscratch(dec, true));
  dec->launch_mode = mode;
  return QD_OK;
}

qd_status qd_decoder_counters(qd_decoder* dec, long long out[5]) {
  QD_REQ(dec && out, "null argument");
  QD_CK(cudaMemcpy(out, dec->d_counters, sizeof(long long) * 5, cudaMemcpyDeviceToHost));
  return QD_OK;
}

qd_status qd_decoder_counters_ex(qd_decoder* dec, long long* out, int n) {
  QD_REQ(dec && out, "null argument");
  QD_REQ(n >= 1 && n <= kCounters, "qd_decoder_counters_ex: n outside [1, 8]");
  QD_CK(cudaMemcpy(out, dec->d_counters, sizeof(long long) * n, cudaMemcpyDeviceToHost));
  return QD_OK;
}

qd_status qd_decoder_set_fork(qd_decoder* dec, int on) {
  QD_REQ(dec, "null argument");
  QD_REQ(on >= 0 && on <= 2, "qd_decoder_set_fork: on must be 0, 1 or 2");
  dec->fork_on = on != 0;
  dec->sched_on = on == 2;
  return QD_OK;
}

qd_status qd_decoder_reset_counters(qd_decoder* dec, qd_stream_t stream) {
  QD_REQ(dec, "null argument");
  QD_CK(cudaMemsetAsync(dec->d_counters, 0, sizeof(long long) * kCounters, (cudaStream_t)stream));
  return QD_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Allocation-free decode + commit (qd_decode_commit_static).
//
// The per-shot window corrections and the work-queue counter that
// qd_decode_windows / qd_commit_and_slide keep in decoder-owned or
// caller-owned device buffers live here in one fixed array that is part of
// the library image.  Every GPU that loads the library holds these
// QD_STATIC_SCRATCH_BYTES until the process exits.
namespace {
constexpr size_t kStaticScratchBytes = QD_STATIC_SCRATCH_BYTES;
constexpr size_t kStaticHeader = 256;  // the work counter, then padding to the corrections' alignment
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

std::mutex g_static_mu;
void* g_static_addr[256] = {};  // device address of g_static_scratch, per device ordinal

// The array's name in host code is only a host-side stand-in; the device
// address must come from the runtime, once per device, with that device current.
qd_status static_scratch_address(void** out) {
  int dev = 0;
  QD_CK(cudaGetDevice(&dev));
  QD_REQ(dev >= 0 && dev < 256, "qd_decode_commit_static: device ordinal out of range");
  std::lock_guard<std::mutex> lk(g_static_mu);
  if (!g_static_addr[dev]) {
    void* p = nullptr;
    QD_CK(cudaGetSymbolAddress(&p, g_static_scratch));
    g_static_addr[dev] = p;
  }
  *out = g_static_addr[dev];
  return QD_OK;
}
}  // namespace

extern "C" qd_status qd_decode_commit_static(qd_decoder* dec, int k, uint32_t* det_bits, int64_t n_shots,
                                             uint32_t* obs_pred, uint32_t* residue_fail,
                                             qd_stream_t stream) {
  QD_REQ(dec && det_bits && obs_pred && residue_fail, "qd_decode_commit_static: null argument");
  QD_REQ(k >= 0 && k < (int)dec->wins.size(), "qd_decode_commit_static: window out of range");
  QD_REQ(n_shots >= 0, "qd_decode_commit_static: n_shots < 0");
  const size_t need = kStaticHeader + sizeof(uint32_t) * (size_t)n_shots * dec->corr_words;
  if (need > kStaticScratchBytes) {
    set_error("qd_decode_commit_static: " + std::to_string(n_shots) + " shots need " +
              std::to_string(need) + " B of static scratch, more than the library's fixed " +
              std::to_string(kStaticScratchBytes) + " B; use at most " +
              std::to_string((kStaticScratchBytes - kStaticHeader) / (sizeof(uint32_t) * dec->corr_words)) +
              " shots per call");
    return QD_EINVAL;
  }
  if (n_shots == 0) return QD_OK;
  QD_REQ(!dec->d_keep || n_shots <= dec->max_shots, "qd_decode_commit_static: n_shots > max_shots with message reuse");
  void* base = nullptr;
  if (qd_status st = static_scratch_address(&base)) return st;
  int* work = (int*)base;
  uint32_t* corr = (uint32_t*)((char*)base + kStaticHeader);
  const WinGpu& g = dec->wins[k];
  const qd::ReuseDev ru = reuse_dev(dec, g);
  cudaStream_t st = (cudaStream_t)stream;
  const int dw = (dec->dem->h.n_det + 31) / 32;
  if (g.h.n_cols > 0) {
    // the launch shape qd_decode_windows would take; every buffer it needs
    // besides the corrections and the work counter was allocated with the
    // decoder (path results and arrival counters, global union regions), and
    // the work counters go to the decoder's own (qd_decoder_counters)
    const bool global = !g.fits || dec->launch_mode == 3;
    const int ps = path_shape(dec, g, n_shots);
    if (g.dv.wts) QD_CK(qd::launch_order_weights(st, g.dv));
    if (ps >= 0) {
      const PathShape& p = g.pa[ps];
      const int cps = path_ctas(dec, p);
      QD_CK(qd::launch_decode(1, 1, (int)(n_shots * cps), kPathThreads >> ps, p.L.total, st, dec->kp, g.dv, p.L,
                              det_bits, dw, n_shots, corr, dec->corr_words, nullptr, nullptr, 0, dec->dmx, dec->ns_max,
                              nullptr, dec->d_counters, dec->d_path_res, dec->d_arrive, dec->sw_max,
                              p.L.ids ? dec->d_uscratch : nullptr, p.L.ids, cps, p.pcl, nullptr, &ru));
    } else {
      // the array keeps the previous call's contents: the work counter restarts at 0
      QD_CK(cudaMemsetAsync(work, 0, sizeof(int), st));
      const ShotShape& s = shot_shape(dec, g, global ? INT64_MAX : n_shots);
      const qd::ForkDev fk = fork_dev(dec, s);
      const qd::Layout& L = global ? g.Lg : s.L;
      const long long grid =
          std::min<long long>(n_shots, (long long)dec->sm_count * (global ? g.grid_g : s.grid_per_sm));
      QD_CK(qd::launch_decode(0, s.ctas, (int)grid, 32 * (global ? kShotWarps : s.warps), global ? L.U : L.total, st,
                              dec->kp, g.dv, L, det_bits, dw, n_shots, corr, dec->corr_words, nullptr, nullptr, 0,
                              dec->dmx, dec->ns_max, work, dec->d_counters, nullptr, nullptr, dec->sw_max,
                              global ? dec->d_uscratch : nullptr, global ? L.total - L.U : 0, 1, 1, &fk, &ru));
    }
  }
  const int w = dec->dem->h.w;
  QD_CK(qd::launch_commit(st, g.h.n_commit, g.d_ccptr, g.d_ccdet, g.d_ccobs, dec->corr_words, corr, n_shots,
                          det_bits, dw, obs_pred, residue_fail, g.h.r0 * w, g.h.commit_b1 * w));
  return QD_OK;
}

// ---------------------------------------------------------------------------
// Batched window steps over several decoders (codes / window sizes).
struct qd_batch {
  std::vector<qd_decoder*> mem;
  int n_steps = 0, sm_count = 0, optin = 0;
  size_t budget2 = 0;  // dynamic shared bytes that leave room for two CTAs per SM
  struct Step {
    int warps = 1, blocks = 1;
    size_t budget = 0, smem = 0;
    unsigned q_off = 0;
    std::vector<qd::Layout> L;  // per member (unused where the member has no such window)
    std::vector<int> form;      // per member: what its layout was made for (member_form)
    std::vector<char> own;      // per member: decoded by a launch of its own (see batch_plan)
  };
  std::vector<Step> steps;
  int* d_work = nullptr;  // one counter per step
  std::vector<qd::ForkDev> forks;  // per member: the current step's path-scheduling plan
};

namespace {
int member_form(const qd_decoder* d) { return layout_form(d->lw_on, d->hist_on); }

// CTAs of `warps` warps with at most `budget` bytes of dynamic shared memory:
// each member's layout takes as many path slots (<= warps) as fit.  A shape is
// for windows whose plain CSC and CSR arrays leave room for a slot (make_layout);
// in slices a few of those do not fit (unshortened windows with learned weights,
// one size per code: [[72,12,6]] (5,1) on half an SM), and such a member is
// decoded by its own launch in the same step.
qd_status batch_plan(qd_batch* b, int j, int warps, size_t budget) {
  qd_batch::Step S;
  S.L.assign(b->mem.size(), qd::Layout{});
  S.own.assign(b->mem.size(), 0);
  for (const qd_decoder* d : b->mem) S.form.push_back(member_form(d));
  unsigned mx = 0;
  for (size_t i = 0; i < b->mem.size(); ++i) {
    const qd_decoder* d = b->mem[i];
    if (j >= (int)d->wins.size()) continue;
    const auto& h = d->wins[j].h;
    const unsigned room = budget > 64 ? (unsigned)(budget - 32) & ~15u : 0u;
    S.L[i] = qd::make_slice_layout(slice_dims(h), h.n_rows, h.n_cols, h.n_short, d->kp.nb, room, d->hist_on, d->lw_on,
                                   false);
    if (S.L[i].total > room) {
      const unsigned plain = qd::make_layout(h.n_rows, h.n_cols, h.n_edges, h.n_short, h.short_edges_max, d->kp.nb, 1,
                                             false, d->hist_on, d->lw_on).total;
      if (qd::al16(plain) + 32 <= budget) {
        S.own[i] = 1;
        continue;
      }
      set_error("qd_batch: member " + std::to_string(i) + " window " + std::to_string(j) + " needs " +
                std::to_string(S.L[i].total + 32) + " B of shared memory with one path slot (budget " +
                std::to_string(budget) + ")");
      return QD_EUNSUPPORTED;
    }
    S.L[i].total = room;  // its slots take what the budget holds
    mx = std::max(mx, S.L[i].total);
  }
  S.q_off = qd::al16(mx);
  S.smem = S.q_off + 32;  // work slot, then the staging mbarrier and its flag
  S.warps = warps;
  S.budget = budget;
  int blocks = 0;
  QD_CK(qd::batch_occupancy(32 * warps, S.smem, &blocks));
  S.blocks = std::max(1, blocks);
  b->steps[j] = S;
  return QD_OK;
}

// The member table of step j; returns the number of members with work.
int batch_members(qd_batch* b, int j, uint32_t* const* det, const int64_t* n, uint32_t* const* obs_pred,
                  uint32_t* const* resid, std::vector<qd::BatchMember>& out) {
  out.clear();
  // heavier windows first, so the tail of the persistent launch is short
  std::vector<int> order;
  for (size_t i = 0; i < b->mem.size(); ++i)
    if (j < (int)b->mem[i]->wins.size() && n[i] > 0) order.push_back((int)i);
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
    return b->mem[x]->wins[j].h.n_edges > b->mem[y]->wins[j].h.n_edges;
  });
  for (int i : order) {
    qd_decoder* d = b->mem[i];
    const WinGpu& g = d->wins[j];
    qd::BatchMember m{};
    m.P = &d->kp;
    m.W = &g.dv;
    m.L = &b->steps[j].L[i];
    m.det = det[i];
    m.det_words = (d->dem->h.n_det + 31) / 32;
    m.n = n[i];
    m.corr = d->d_corr;
    m.corr_words = d->corr_words;
    m.dmx = d->dmx;
    m.ns_max = d->ns_max;
    m.sw_max = d->sw_max;
    m.counters = d->d_counters;
    m.n_commit = g.h.n_commit;
    m.cptr = g.d_ccptr;
    m.cdet = g.d_ccdet;
    m.cobs = g.d_ccobs;
    m.obs_pred = obs_pred ? obs_pred[i] : nullptr;
    m.resid = resid ? resid[i] : nullptr;
    const int w = d->dem->h.w;
    m.b0 = g.h.r0 * w;
    m.b1 = g.h.commit_b1 * w;
    b->forks.resize(b->mem.size());
    b->forks[i] = fork_dev(d, g.sh[g.best]);
    m.fork = &b->forks[i];
    m.who = i;
    out.push_back(m);
  }
  return (int)out.size();
}

qd_status batch_decode(qd_batch* b, int j, const std::vector<qd::BatchMember>& all, cudaStream_t st) {
  const qd_batch::Step& S = b->steps[j];
  // windows without columns decide nothing; their commits still test the residue
  std::vector<qd::BatchMember> m;
  for (const auto& x : all) {
    if (x.W->n_cols == 0) continue;
    if (S.own[x.who]) QD_CK_ST(qd_decode_windows(b->mem[x.who], j, x.det, x.n, x.corr, nullptr, nullptr, st));
    else m.push_back(x);
  }
  if (m.empty()) return QD_OK;
  long long tot = 0;
  for (const auto& x : m) tot += x.n;
  QD_CK(cudaMemsetAsync(b->d_work + j, 0, sizeof(int), st));
  for (const auto& x : m)
    if (x.W->wts) QD_CK(qd::launch_order_weights(st, *x.W));
  const long long grid = std::min<long long>(tot, (long long)b->sm_count * S.blocks);
  QD_CK(qd::launch_decode_batch(st, (int)grid, 32 * S.warps, S.smem, S.q_off, b->d_work + j, m.data(),
                                (int)m.size()));
  return QD_OK;
}
}  // namespace

extern "C" {

qd_status qd_batch_create(qd_decoder* const* members, int n_members, qd_batch** out) {
  QD_REQ(members && out, "qd_batch_create: null argument");
  QD_REQ(n_members >= 1 && n_members <= qd::kMaxBatch,
         "qd_batch_create: need 1 <= n_members <= " + std::to_string(qd::kMaxBatch));
  std::unique_ptr<qd_batch> b(new (std::nothrow) qd_batch());
  if (!b) return QD_ENOMEM;
  for (int i = 0; i < n_members; ++i) {
    QD_REQ(members[i], "qd_batch_create: null member");
    if (members[i]->P.reuse_msgs) {
      set_error("qd_batch_create: message reuse between windows is not supported in batched steps");
      return QD_EUNSUPPORTED;
    }
    b->mem.push_back(members[i]);
    b->n_steps = std::max(b->n_steps, (int)members[i]->wins.size());
  }
  int dev = 0;
  QD_CK(cudaGetDevice(&dev));
  QD_CK(cudaDeviceGetAttribute(&b->sm_count, cudaDevAttrMultiProcessorCount, dev));
  QD_CK(cudaDeviceGetAttribute(&b->optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  QD_CK(qd::set_decode_smem((size_t)b->optin));
  int per_sm = 0, reserved = 0;
  QD_CK(cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
  QD_CK(cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev));
  b->budget2 = (size_t)std::max(0, per_sm / 2 - reserved);
  b->steps.resize(b->n_steps);
  // default shape: 8 warps, two CTAs per SM when every member fits a slot
  for (int j = 0; j < b->n_steps; ++j)
    if (batch_plan(b.get(), j, kShotWarps, b->budget2) != QD_OK)
      QD_CK_ST(batch_plan(b.get(), j, kShotWarps, (size_t)b->optin));
  QD_CK(cudaMalloc(&b->d_work, sizeof(int) * std::max(1, b->n_steps)));
  *out = b.release();
  return QD_OK;
}

qd_status qd_batch_destroy(qd_batch* b) {
  if (!b) return QD_OK;
  cudaFree(b->d_work);
  delete b;
  return QD_OK;
}

qd_status qd_batch_n_steps(const qd_batch* b, int* n) {
  QD_REQ(b && n, "null argument");
  *n = b->n_steps;
  return QD_OK;
}

qd_status qd_batch_set_shape(qd_batch* b, int step, int warps, int ctas_per_sm) {
  QD_REQ(b, "null argument");
  QD_REQ(step >= 0 && step < b->n_steps, "qd_batch_set_shape: step out of range");
  QD_REQ(warps >= 1 && warps <= kShotWarps, "qd_batch_set_shape: warps must be in [1, 8]");
  QD_REQ(ctas_per_sm == 1 || ctas_per_sm == 2, "qd_batch_set_shape: ctas_per_sm must be 1 or 2");
  const qd_batch::Step keep = b->steps[step];
  if (qd_status st = batch_plan(b, step, warps, ctas_per_sm == 2 ? b->budget2 : (size_t)b->optin)) {
    b->steps[step] = keep;
    return st;
  }
  return QD_OK;
}

qd_status qd_batch_info(const qd_batch* b, int step, int out[4]) {
  QD_REQ(b && out, "null argument");
  QD_REQ(step >= 0 && step < b->n_steps, "qd_batch_info: step out of range");
  const auto& S = b->steps[step];
  out[0] = S.warps;
  out[1] = (int)S.smem;
  out[2] = S.blocks;
  int active = 0;
  for (auto* d : b->mem) active += step < (int)d->wins.size();
  out[3] = active;
  return QD_OK;
}

qd_status qd_batch_step(qd_batch* b, int step, uint32_t* const* det_bits, const int64_t* n_shots,
                        uint32_t* const* obs_pred, uint32_t* const* residue_fail, qd_stream_t stream) {
  QD_REQ(b && det_bits && n_shots && obs_pred && residue_fail, "qd_batch_step: null argument");
  QD_REQ(step >= 0 && step < b->n_steps, "qd_batch_step: step out of range");
  for (size_t i = 0; i < b->mem.size(); ++i) {
    QD_REQ(n_shots[i] >= 0 && n_shots[i] <= b->mem[i]->max_shots,
           "qd_batch_step: n_shots of member " + std::to_string(i) + " outside [0, max_shots]");
    QD_REQ(n_shots[i] == 0 || (det_bits[i] && obs_pred[i] && residue_fail[i]),
           "qd_batch_step: null buffer of member " + std::to_string(i));
  }
  // weights or a ranker installed (or removed) since the step was planned
  for (size_t i = 0; i < b->mem.size(); ++i)
    if (b->steps[step].form[i] != member_form(b->mem[i])) {
      const int warps = b->steps[step].warps;
      const size_t budget = b->steps[step].budget;
      if (batch_plan(b, step, warps, budget) != QD_OK) QD_CK_ST(batch_plan(b, step, warps, (size_t)b->optin));
      break;
    }
  std::vector<qd::BatchMember> m;
  if (!batch_members(b, step, det_bits, n_shots, obs_pred, residue_fail, m)) return QD_OK;
  cudaStream_t st = (cudaStream_t)stream;
  if (qd_status s = batch_decode(b, step, m, st)) return s;
  QD_CK(qd::launch_commit_batch(st, m.data(), (int)m.size()));
  return QD_OK;
}

qd_status qd_batch_autotune(qd_batch* b, int step, uint32_t* const* det_bits, const int64_t* n_shots, int reps,
                            qd_stream_t stream, float* best_ms) {
  QD_REQ(b && det_bits && n_shots, "qd_batch_autotune: null argument");
  QD_REQ(step >= 0 && step < b->n_steps, "qd_batch_autotune: step out of range");
  QD_REQ(reps >= 1, "qd_batch_autotune: reps < 1");
  for (size_t i = 0; i < b->mem.size(); ++i)
    QD_REQ(n_shots[i] >= 0 && n_shots[i] <= b->mem[i]->max_shots, "qd_batch_autotune: n_shots outside range");
  std::vector<qd::BatchMember> m;
  if (!batch_members(b, step, det_bits, n_shots, nullptr, nullptr, m)) return QD_OK;
  cudaStream_t st = (cudaStream_t)stream;
  cudaEvent_t e0, e1;
  QD_CK(cudaEventCreate(&e0));
  QD_CK(cudaEventCreate(&e1));
  const qd_batch::Step keep = b->steps[step];
  float best = 0.0f;
  int pick_w = 0;
  size_t pick_b = 0;
  qd_status st_out = QD_OK;
  const size_t budgets[2] = {b->budget2, (size_t)b->optin};
  for (int w = kShotWarps; w >= 4 && st_out == QD_OK; --w)
    for (size_t bud : budgets) {
      if (batch_plan(b, step, w, bud) != QD_OK) continue;
      // the member table points at this step's layouts, which batch_plan rebuilt
      batch_members(b, step, det_bits, n_shots, nullptr, nullptr, m);
      if ((st_out = batch_decode(b, step, m, st)) != QD_OK) break;  // warm-up
      cudaError_t e = cudaEventRecord(e0, st);
      for (int r = 0; r < reps && e == cudaSuccess; ++r)
        if ((st_out = batch_decode(b, step, m, st)) != QD_OK) break;
      if (st_out != QD_OK) break;
      if (e == cudaSuccess) e = cudaEventRecord(e1, st);
      if (e == cudaSuccess) e = cudaEventSynchronize(e1);
      float ms = 0.0f;
      if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
      if (e != cudaSuccess) {
        set_error(std::string("qd_batch_autotune: ") + cudaGetErrorString(e));
        st_out = QD_ECUDA;
        break;
      }
      ms /= reps;
      if (!pick_w || ms < best) {
        best = ms;
        pick_w = w;
        pick_b = bud;
      }
    }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (st_out != QD_OK || !pick_w) {
    b->steps[step] = keep;
    return st_out;
  }
  QD_CK_ST(batch_plan(b, step, pick_w, pick_b));
  if (best_ms) *best_ms = best;
  return QD_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Learned weighted min-sum: training on window samples.
struct qd_wms {
  qd::WmsGraph G{};
  qd::WmsSlices S{};
  int k = 0;
  uint32_t* d_thr = nullptr;
  char* d_graph = nullptr;    // the arrays of S
  char* d_scratch = nullptr;  // check records by iteration, per CTA
  int* d_work = nullptr;
  int grid = 0;
  size_t smem = 0;
};

extern "C" {

qd_status qd_wms_create(const qd_decoder* dec, int k, int T, int ckpt, qd_wms** out) {
  QD_REQ(dec && out, "qd_wms_create: null argument");
  QD_REQ(k >= 0 && k < (int)dec->wins.size(), "qd_wms_create: window out of range");
  QD_REQ(T >= 1 && T <= 1000 && ckpt >= 1 && ckpt <= T, "qd_wms_create: need 1 <= ckpt <= T");
  std::unique_ptr<qd_wms> m(new (std::nothrow) qd_wms());
  if (!m) return QD_ENOMEM;
  const WinGpu& g = dec->wins[k];
  m->k = k;
  m->G = qd::WmsGraph{g.h.n_rows, g.h.n_cols, g.h.n_edges, (g.h.n_rows + 31) / 32, T, ckpt,
                      g.dv.col_ptr, g.dv.col_rows, g.dv.row_ptr, g.dv.row_ent, g.dv.llr, dec->P.clip};
  std::vector<uint32_t> thr(g.h.n_cols);
  for (int c = 0; c < g.h.n_cols; ++c) thr[c] = dec->dem->h.col_thr[g.h.gcols[c]];
  QD_CK(upload(&m->d_thr, thr));
  int optin = 0, dev = 0;
  QD_CK(cudaGetDevice(&dev));
  QD_CK(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  if (qd::wms_window_bytes(m->G.ne, m->G.nc, m->G.rw) > (size_t)optin) {
    set_error("qd_wms_create: window too large for shared memory");
    return QD_EUNSUPPORTED;
  }
  const qd::WmsHost H = qd::build_wms(g.h);
  Blob b;
  const size_t o_ro = b.put(H.roff), o_co = b.put(H.coff), o_rc = b.put(H.rcell), o_rl = b.put(H.rcol),
               o_re = b.put(H.reid), o_ce = b.put(H.cent), o_ei = b.put(H.ceid), o_ll = b.put(g.h.s_llr),
               o_rw = b.put(H.row), o_cl = b.put(H.col);
  QD_CK(b.upload(&m->d_graph));
  auto u16 = [&](size_t o) { return (const uint16_t*)(m->d_graph + o); };
  m->S = qd::WmsSlices{m->G.nr, m->G.nc, m->G.ne, m->G.rw, T, (int)H.roff.size() - 1, (int)H.coff.size() - 1,
                       g.h.col_cells, u16(o_ro), u16(o_co), u16(o_rc), u16(o_rl), u16(o_re),
                       (const uint32_t*)(m->d_graph + o_ce), u16(o_ei), (const float*)(m->d_graph + o_ll), u16(o_rw),
                       u16(o_cl), dec->P.clip, 0};
  m->smem = qd::wms_smem_bytes(m->S);
  QD_CK(qd::wms_set_smem((size_t)optin));  // the device limit: contexts of different sizes coexist
  int blocks = 0;
  QD_CK(qd::wms_occupancy(m->smem, &blocks));
  m->grid = dec->sm_count * std::max(1, blocks);
  if (qd::wms_scratch_per_cta(m->S) * m->grid > qd::kWmsKeepBytes) m->S.seg = ckpt;
  QD_CK(cudaMalloc(&m->d_scratch, qd::wms_scratch_per_cta(m->S) * m->grid));
  QD_CK(cudaMalloc(&m->d_work, sizeof(int)));
  *out = m.release();
  return QD_OK;
}

qd_status qd_wms_destroy(qd_wms* m) {
  if (!m) return QD_OK;
  cudaFree(m->d_thr);
  cudaFree(m->d_graph);
  cudaFree(m->d_scratch);
  cudaFree(m->d_work);
  delete m;
  return QD_OK;
}

qd_status qd_wms_info(const qd_wms* m, int out[6]) {
  QD_REQ(m && out, "null argument");
  out[0] = m->G.nr;
  out[1] = m->G.nc;
  out[2] = m->G.ne;
  out[3] = m->G.T;
  out[4] = m->G.ckpt;
  out[5] = m->G.rw;
  return QD_OK;
}

qd_status qd_wms_sample(qd_wms* m, uint64_t seed, uint64_t offset, int64_t n, uint32_t* synd, qd_stream_t stream) {
  QD_REQ(m && synd && n >= 0, "qd_wms_sample: bad argument");
  QD_CK(qd::launch_wms_sample((cudaStream_t)stream, m->G, m->d_thr, seed, offset, n, 1u + (unsigned)m->k, synd,
                              nullptr, 0, 0, nullptr, 0));
  return QD_OK;
}

static qd_status wms_run(qd_wms* m, const float* w, const uint32_t* synd, int64_t n, int backward, float scale,
                         float* grad_w, float* loss, float* post, qd_stream_t stream) {
  QD_REQ(m && w && synd && n >= 0, "qd_wms: bad argument");
  if (n == 0) return QD_OK;
  cudaStream_t st = (cudaStream_t)stream;
  QD_CK(cudaMemsetAsync(m->d_work, 0, sizeof(int), st));
  const int grid = (int)std::min<long long>(n, m->grid);
  QD_CK(qd::launch_wms(st, grid, m->smem, m->S, w, synd, n, backward, scale, grad_w, loss, post, m->d_scratch,
                       m->d_work));
  return QD_OK;
}

qd_status qd_wms_loss(qd_wms* m, const float* w, const uint32_t* synd, int64_t n, float* loss, float* post,
                      qd_stream_t stream) {
  QD_REQ(loss, "qd_wms_loss: loss is required");
  return wms_run(m, w, synd, n, 0, 0.0f, nullptr, loss, post, stream);
}

qd_status qd_wms_grad(qd_wms* m, const float* w, const uint32_t* synd, int64_t n, float grad_scale, float* grad_w,
                      float* loss, qd_stream_t stream) {
  QD_REQ(grad_w, "qd_wms_grad: grad_w is required");
  return wms_run(m, w, synd, n, 1, grad_scale, grad_w, loss, nullptr, stream);
}

qd_status qd_window_sample(qd_decoder* dec, int k, uint64_t seed, uint64_t offset, int64_t n, uint32_t* det_bits,
                           uint32_t* fault_bits, qd_stream_t stream) {
  QD_REQ(dec && det_bits && n >= 0, "qd_window_sample: bad argument");
  QD_REQ(k >= 0 && k < (int)dec->wins.size(), "qd_window_sample: window out of range");
  WinGpu& g = dec->wins[k];
  if (!g.d_wthr) {
    std::vector<uint32_t> thr(g.h.n_cols);
    for (int c = 0; c < g.h.n_cols; ++c) thr[c] = dec->dem->h.col_thr[g.h.gcols[c]];
    QD_CK(upload(&g.d_wthr, thr));
  }
  const qd::WmsGraph G{g.h.n_rows, g.h.n_cols, g.h.n_edges, (g.h.n_rows + 31) / 32, 1, 1,
                       g.dv.col_ptr, g.dv.col_rows, g.dv.row_ptr, g.dv.row_ent, g.dv.llr, dec->P.clip};
  QD_CK(qd::launch_wms_sample((cudaStream_t)stream, G, g.d_wthr, seed, offset, n, 1u + (unsigned)k, nullptr,
                              det_bits, (dec->dem->h.n_det + 31) / 32, g.h.row0, fault_bits, dec->corr_words));
  return QD_OK;
}

qd_status qd_ranker_eval(const float* params, const void* records, const uint8_t* labels, int64_t n, int quantize,
                         float pos_weight, float grad_scale, float* grad, float* loss, float* score,
                         qd_stream_t stream) {
  QD_REQ(params && records && n >= 0, "qd_ranker_eval: bad argument");
  QD_REQ(!(grad || loss) || labels, "qd_ranker_eval: labels are required for grad and loss");
  QD_CK(qd::launch_ranker((cudaStream_t)stream, params, (const qd::RankRec*)records, labels, n, quantize,
                          pos_weight, grad_scale, grad, loss, score));
  return QD_OK;
}

qd_status qd_set_zero(void* dst, size_t bytes, qd_stream_t stream) {
  QD_REQ(dst || bytes == 0, "qd_set_zero: null pointer");
  if (bytes) QD_CK(cudaMemsetAsync(dst, 0, bytes, (cudaStream_t)stream));
  return QD_OK;
}

qd_status qd_adam_step(float* w, const float* g, float* m1, float* m2, int64_t n, float lr, float beta1, float beta2,
                       float eps, int step, qd_stream_t stream) {
  QD_REQ(w && g && m1 && m2 && n >= 0 && step >= 1, "qd_adam_step: bad argument");
  QD_CK(qd::launch_adam((cudaStream_t)stream, w, g, m1, m2, n, lr, beta1, beta2, eps, step));
  return QD_OK;
}

}  // extern "C"
