// gdg_kernel.cuh -- shared definitions of the window decoder (host and device).
//
// Message representation.  Min-sum (Eq. (1)) sends from check j to variable i
//   mu_{j->i} = (-1)^{s_j} * (alpha * min_{i' != i} |mu_{i'->j}|) * prod_{i' != i} sign(mu_{i'->j})
// which only depends on the check's two smallest |mu| (min1, min2), the edge
// holding min1 (amin), the sign parity of all its inputs xor s_j, and the sign
// of the receiving edge's own input.  The kernel keeps exactly that per check
// in one 16-byte record (the signs as one bit per edge), instead of two FP32
// messages per edge.  The VN->CN message of Eq. (3) is recomputed where it is
// needed as clip(Lambda_i^(t) - mu_{j->i}), the same FP32 operations the
// explicit form performs, so every value is bit-identical to it.  All FP32
// operations are __fadd_rn / __fsub_rn / __fmul_rn (never contracted).
//
// Graph format.  Checks and columns are numbered by descending degree, and the
// entries of 32 consecutive ones (a slice, one per lane of a warp) are stored
// lane by lane, entry u of every lane side by side (a check's four at a time),
// each slice as wide as its first node's degree (check slices rounded up to a
// multiple of four).  A warp
// walks a slice with conflict-free loads, one trip count for all lanes and no
// bounds test: the places past a node's degree hold a dummy whose value
// changes nothing (a column with posterior +inf, a check record with message
// +0).
//   check entry:  the column, or (shortened graph) its posterior's byte offset
//   column entry: check << 16 | position of the edge among the check's entries
#pragma once
#include <cstddef>
#include <cstdint>

namespace qd {

constexpr int kMaxBatch = 16;  // decoders in one batched launch

struct KParams {
  float alpha, clip, pa_main, pa_other, pb_main, pb_other, pb_d1, pc, pd;
  int n_pre, ips, dmax_main, dmax_other, k, low_err, peel_init, pc_max_depth, n_unsat_min;
  int nb;        // decision paths: 2^k tree + side branches
  int side_max;  // side branches split off the main branch at D_split = k .. side_max (0: none)
  int reinit;    // 1: a path continuing from another's snapshot restarts its messages there
  int ips1;      // BP iterations of the first decimation step (0: ips)
  int fallback;  // output when no path converges: 0 path 0, 1 fewest unsatisfied checks, 2 committed ones first
  // learned decimation ranker (NULL: the argmin of Alg. 1): rkq = the
  // grid-rounded W1[64][8], b1[64], W2[64], b2; rkb[t][lane] = the BF16 pair
  // (W1[8t + lane/4][2 (lane%4)], W1[8t + lane/4][2 (lane%4) + 1]), the B
  // fragment of an m16n8k8 MMA for hidden units 8t..8t+7
  const float* rkq;
  const uint32_t* rkb;
  // candidate dump of path 0 (ranker training data; NULL: off)
  struct RankRec* dump;
  int* dump_n;
  int dump_cap;
};

// One ranker candidate (layout of qd_rank_rec_t): features, shot, window
// column, selection depth, path; flags bit 0 = [L <= 0], bit 1 = selected.
struct RankRec {
  float x[8];
  int32_t shot, wcol;
  int16_t depth, path;
  int32_t flags;
};

// Side-branch split depth of path `id` (Fig. 2): 0 for the main and tree
// branches.  With side branches, id 1 (contrary only at D = k) is the one
// splitting at D = k and ids 2^k.. split at D = k + 1 ...
__host__ __device__ inline int path_split(const KParams& P, int id) {
  if (P.side_max <= 0) return 0;
  const int nt = 1 << P.k;
  if (id >= nt) return P.k + 1 + (id - nt);
  return (id == 1 && P.k >= 1) ? P.k : 0;
}

// Depth after whose decimation path `id` restarts its messages (reinit
// reading: side branches at their split, odd tree ids at D = k); 0: never.
__host__ __device__ inline int path_reinit(const KParams& P, int id, int split) {
  if (!P.reinit) return 0;
  if (split) return split;
  return (id >= 1 && (id & 1) && P.k >= 1) ? P.k : 0;
}

// D_max of path `id` with side-branch split `split` (Fig. 2): the main
// branch's own; a side branch runs as many steps past its split as a tree
// branch runs past depth k.
__host__ __device__ inline int path_dmax(const KParams& P, int id, int split) {
  return id == 0 ? P.dmax_main : (split ? split + (P.dmax_other - P.k) : P.dmax_other);
}

// Shot-mode queue order: the main branch, side branches from the deepest
// split down, then the tree branches -- the longest paths first when the main
// branch's D_max is the largest (the circuit-level presets; the code-capacity
// tree's deepest side branches outlast its main branch).  The order only
// schedules the paths; every result is kept by path id.
__host__ __device__ inline int path_at(const KParams& P, int pos) {
  const int nside = P.nb - (1 << P.k);
  if (pos == 0) return 0;
  if (pos <= nside) return P.nb - pos;
  return pos - nside;
}

// Column slices by width: [0, n4) at least four wide, [n4, n3) three, [n3, n2)
// two, [n2, n1) one.
struct ColClasses {
  int n4, n3, n2, n1;
};

// One window's Tanner graph in global memory (read-only for all shots).
struct WinDev {
  int n_rows, n_cols, n_edges, row0, n_short, es_max, rows_per_block;
  const uint16_t *col_ptr, *col_rows, *row_ptr;
  const uint32_t* row_ent;  // CSR entry: CSC edge id | (column << 16)
  const float* llr;
  // learned weighted min-sum: wts[(min(t, wT) - 1) * n_edges + e] replaces
  // alpha at iteration t (counted from message initialisation); NULL = alpha
  const float* wts;
  int wT;
  // the first w_rows iterations' (all that the pre-BP reads) in the order of
  // s_rent / s_cent (order_weights_kernel)
  int w_rows;
  float *w_row, *w_col;
  int n_commit_rows;      // rows [0, n_commit_rows) are the ones the window commits
  // the graph in slices (see the top of the file), checks and columns by label
  int row_quads, col_cells;    // slice totals per lane: check entries in fours, column entries
  const uint16_t* s_rent;  // [4 * 32 * row_quads]
  const uint32_t* s_cent;  // [32 * col_cells]
  const uint16_t *s_roff, *s_coff;   // slice starts, in fours / in entries per lane
  const float* s_llr;                // priors by column label
  const uint16_t *s_row, *s_col;     // label -> window row / window column
  ColClasses cls;
  const uint16_t *s_ref, *s_cef;     // full-window edge of each check / column entry (learned weights)
};

// Shot mode's plan for resuming decision paths from snapshots of shared
// prefixes (see ForkCtx in gdg_kernel.cu): the queue order, and for every path
// p and depth D the snapshot node of p after the BP of step D
// (chain[p * dmx + D - 1], -1: none).  Snapshots of CTA b live at
// pool + b * cta_bytes, nodes `stride` bytes apart; pool = nullptr: no
// snapshots, the path-queue order of path_at.
// node flags, then path states, live in the shot-mode CTA's 512-byte reduction area
constexpr int kMaxForkNodes = 64;
constexpr unsigned kSnapHeaderBytes = 32;  // a snapshot's header, before the copy of the slot
// fnode / fdep: each path's planned snapshot node (-1: none) and its depth;
// sched != 0: preemption at step boundaries, each path's parking snapshot
// after the n_nodes node snapshots of the CTA's pool.
struct ForkDev {
  const int16_t* order;
  const int16_t* chain;
  const int16_t* fnode;
  const int16_t* fdep;
  char* pool;
  size_t cta_bytes;
  int n_nodes, pool_ctas, sched;
};

// Message reuse between windows (see DecodeArgs::keep); keep = nullptr: off.
struct ReuseDev {
  float* keep;
  int keep_ld;
  const int16_t* prev;
  float* kpath;
};

// A window's Tanner graph for the learned weighted min-sum (training kernels).
struct WmsGraph {
  int nr, nc, ne, rw, T, ckpt;
  const uint16_t *col_ptr, *col_rows, *row_ptr;
  const uint32_t* row_ent;  // CSC edge id | column << 16
  const float* llr;
  float clip;
};

// The same in slices for the training kernel (labels of WinDev; every check's
// entries in ascending edge order, which decides ties and the order of the
// loss's products; check slices exactly as wide as their first check).
struct WmsSlices {
  int nr, nc, ne, rw, T;
  int nrs, ncs, col_cells;       // check and column slices, column entries per lane
  const uint16_t *roff, *coff;   // slice starts, in entries per lane
  const uint16_t *rcell, *rcol, *reid;  // check entry: the edge's column cell, column label, edge id
  const uint32_t* cent;          // column entry: check label << 16 | position
  const uint16_t* ceid;          // its edge id
  const float* llr;              // by column label
  const uint16_t *row, *col;     // label -> window row (0 for the padding), window column
  float clip;
  // check records kept for the backward pass: every iteration's (0), or every
  // seg-th iteration's and those of one segment of seg iterations at a time
  int seg;
  __host__ __device__ int segs() const { return (T + seg - 1) / seg; }
  __host__ __device__ int records() const { return seg ? segs() - 1 + seg : T; }  // iterations there is room for
  // where iteration t's record goes in the forward pass, -1: it is not kept
  __host__ __device__ int slot_forward(int t) const {
    if (!seg) return t - 1;
    const int n = segs();
    return t > (n - 1) * seg ? slot_backward(t) : (t % seg ? -1 : t / seg - 1);
  }
  // where it is when its segment is gone through backwards
  __host__ __device__ int slot_backward(int t) const { return seg ? segs() - 1 + (t - 1) % seg : t - 1; }
};

// Compressed state of one check node: its two smallest |input| (bounded by the
// clip), each negated when the sign parity xor s_j is 1 and, in the plain
// decoder, multiplied by alpha; sg: the inputs' signs, position p at bit 31 - p
// (p < 32); am: the position of the smallest input (low six bits) and the
// signs of positions 32 .. 57, position p at bit 63 - p.
struct __align__(16) CNState {
  float m1, m2;
  uint32_t sg, am;
};
// Most entries a check may have.  A detector of these codes' circuits touches
// at most 35 columns: the fault classes of a round are the same for every
// choice of A and B (three terms each), and coinciding terms only merge them.
constexpr int kMaxRowDeg = 51;
// Edge id of a dummy (a window has fewer than 65535 edges).
constexpr uint16_t kNoEdge = 0xFFFF;
// Flag of a shortened graph's column slice starts (s_coff) when some check has
// more than 32 entries, so that signs may be in the second word.
constexpr uint16_t kWideSlice = 0x8000;

struct BranchTrace {
  int32_t status, depth, iters, pad;
  double pm;
};
struct StepTrace {
  int16_t g;
  int8_t value, pad;
  int16_t n_agg, n_peel;
};

// Result of one decision path in the path-per-CTA launch (global scratch).
__host__ __device__ inline size_t path_result_bytes(int sw) { return (16 + 4 * (size_t)sw + 15) & ~(size_t)15; }

// Sizes of a window's graph in slices, and bounds on those of its shortened
// graphs.
struct SliceDims {
  int row_quads, col_cells;    // the window's, as WinDev
  int srow_quads, scol_cells;  // the shortened graph's, at most
};
__host__ __device__ inline unsigned al16(unsigned x) { return (x + 15u) & ~15u; }
__host__ __device__ inline unsigned up32(unsigned x) { return (x + 31u) & ~31u; }

// Shared-memory layout of one CTA (byte offsets), identical on host and device.
struct Layout {
  // persistent
  unsigned sbits, cbits, sel, s_colptr, s_colrows, s_rowptr, s_rowent, s_llr, s_vdeg, s_efull, s_cperm, s_vperm, rowcnt,
      res_status, res_pm, res_ebits, red, misc;
  // window graph staged in shared memory (path mode only; 0 bytes otherwise)
  unsigned g_colptr, g_colrows, g_rowptr, g_rowent, g_llr, g_bytes;
  unsigned U;  // start of the union region
  // pre-BP (relative to U; make_slice_layout: to V)
  unsigned p_post, p_key, p_cns, p_sign, p_par, p_sort, p_end;
  // the window graph staged for the pre-BP loop in otherwise idle union bytes
  // (overwritten by the sort that follows); pre_stage = 0: none
  unsigned pre_stage, q_colptr, q_colrows, q_rowptr, q_rowent, q_llr, q_vperm;
  // one path slot (relative to the slot base)
  unsigned b_post, b_acc, b_hfl, b_status, b_sign, b_cns, b_deg, b_sp, b_unsat, b_hq, b_size;
  unsigned total;
  int rw, cw, sw, sortn, nslots;
  // slices: the shortened graph's fixed arrays, and where its entries and the
  // path slots start (s_dyn; laid out per shot, see SlotPlan; U: the slots'
  // start at the latest); the staged window graph (q_rent .. q_sllr; pre_stage
  // has a bit for each array that is staged)
  unsigned s_roff, s_coff, s_cls, s_dyn, plan, p_scr;
  unsigned q_rent, q_cent, q_roff, q_coff, q_sllr;
  // The pre-BP's arrays start at V, where the shortened graph and the path
  // slots begin: neither exists before the pre-BP has ended.
  unsigned V;
  // GraphPlace; with kGraphGlobal s_dyn and SlotPlan::U are relative to the union
  // region in global memory, with kIdsGlobal the shortened entries' edge ids take
  // `ids` bytes of global memory
  unsigned gg, ids;
  unsigned hist, lwe;  // bytes of quantised history per column of degree >= 3; 1: learned weights' edge ids
};
// Where the shortened graph's entries lie: in shared memory; with the union region
// in global memory; in shared memory, but for the edge ids of learned weights.
enum GraphPlace { kGraphShared = 0, kGraphGlobal = 1, kIdsGlobal = 2 };
enum { kStageRent = 1, kStageCent = 2, kStageLlr = 4, kStageOff = 8 };

// A shot's part of the layout: the entries of its shortened graph, then its
// path slots, sized by the graph the shot has (its non-empty check slices,
// its columns of degree three or more), not by the largest there could be:
// 671 edges against a bound of 2304 for [[144,12,12]] (3,1) windows.
struct SlotPlan {
  unsigned rent, cent, ref, cef, U;
  unsigned b_acc, b_hfl, b_status, b_cns, b_deg, b_sp, b_unsat, b_hq, b_size;
  int nslots, rwz;  // path slots that fit; non-empty check slices
  unsigned ids;     // kIdsGlobal: bytes of edge ids
};


// nq, ncell: the shortened graph's check entries in fours and column entries
// (per lane); rwz, n3: its non-empty check slices, its column slices of width
// three or more; end: the bytes there are (glob: of the union region, which
// then holds only the slots); the slots' number is at most `most`.
__host__ __device__ inline SlotPlan slot_plan(const Layout& L, int nq, int ncell, int rwz, int n3, unsigned end,
                                              bool glob, int most) {
  SlotPlan S{};
  const unsigned nsp = 32u * L.sw;
  unsigned o = L.s_dyn;
  S.rent = o; o = al16(o + 512u * nq);
  S.cent = o; o = al16(o + 128u * ncell);
  unsigned& at = L.gg == kIdsGlobal ? S.ids : o;
  S.ref = at; at = al16(at + (L.lwe ? 256u * nq : 0u));
  S.cef = at; at = al16(at + (L.lwe ? 64u * ncell : 0u));
  S.U = o;
  unsigned b = al16(4u * (nsp + 1));  // posteriors and the dummy column's
  S.b_acc = b; b += 128u * n3;
  S.b_hfl = b; b += 32u * n3;
  S.b_status = b; b = al16(b + nsp);
  S.b_cns = b; b += 16u * (32u * rwz + 1);
  S.b_deg = b; b = al16(b + 32u * L.rw);
  S.b_sp = b; b = al16(b + 4u * L.rw);
  S.b_unsat = b; b = al16(b + 4u * L.rw);
  S.b_hq = b; b = al16(b + 32u * L.hist * n3);
  S.b_size = b;
  const unsigned from = glob && L.gg != kGraphGlobal ? 0u : S.U;  // the slots' start
  const unsigned room = end > from ? end - from : 0u;
  const int n = (int)(room / b);
  S.nslots = n < most ? n : most;
  S.rwz = rwz;
  return S;
}

// Layout of the decode kernels for a CTA with `budget` bytes of shared memory.
// The pre-BP scratch and as much of the window graph as fits beside it share
// their bytes with the shortened graph and the path slots that follow.  The
// ranking's sort buffer lies past the keys it is filled from and past the
// shortened graph's fixed arrays, which are written from it; the shortening's
// scratch (p_scr), in use while the entries are written, past the graph at its
// largest.
// total: what the window needs at least (one slot), or with what is staged;
// past the budget the window does not fit.  ub_glob: pre-BP scratch and slots
// live in a region of global memory (eight slots), the shortened graph stays
// in shared memory, total - U is the region's size.  place = kGraphGlobal
// (with ub_glob): the shortened graph's entries start that region, the pre-BP scratch and, once
// it is dead, the slots follow; for windows whose entries at their largest do
// not fit shared memory (padded to slices they take up to twice the bytes of
// plain CSC and CSR arrays: an unshortened [[144,12,12]] window of nine rounds,
// or one of 17 rounds with learned weights).  kIdsGlobal (without ub_glob): see
// GraphPlace; for path mode, where one path has the CTA for itself.
__host__ __device__ inline Layout make_slice_layout(const SliceDims& D, int nr, int nc, int ns, int nb, unsigned budget,
                                                    bool ranker, bool lw, bool ub_glob,
                                                    GraphPlace place = kGraphShared) {
  Layout L{};
  const bool graph_glob = place == kGraphGlobal;
  L.gg = place;
  L.rw = (nr + 31) / 32;
  L.cw = (nc + 31) / 32;
  L.sw = (ns + 31) / 32;
  // keys sorted: the kept columns', selected first, or all when that takes as many
  int sn = 1;
  while (sn < ns) sn <<= 1;
  L.sortn = sn;
  L.hist = ranker ? 4u : 0u;
  L.lwe = lw ? 1u : 0u;
  const unsigned nrp = up32(nr), ncp = up32(nc), nsp = up32(ns);
  unsigned o = 0;
  L.sbits = o; o = al16(o + 4u * L.rw);
  L.cbits = o; o = al16(o + 4u * L.cw);
  L.res_status = o; o = al16(o + 4u * nb);
  L.res_pm = o; o = al16(o + 8u * nb);
  L.res_ebits = o; o = al16(o + 4u * L.sw * nb);
  L.red = o; o = al16(o + 16u * 32);
  L.misc = o; o = al16(o + 64u);
  L.plan = o; o = al16(o + (unsigned)sizeof(SlotPlan));
  L.V = o;
  L.sel = o; o = al16(o + 2u * ns);
  L.s_roff = o; o = al16(o + 2u * (L.rw + 1));
  L.s_coff = o; o = al16(o + 2u * (L.sw + 1));
  L.s_cls = o; o = al16(o + 16u);
  L.s_llr = o; o = al16(o + 4u * nsp);
  L.s_vdeg = o; o = al16(o + nsp);
  L.s_cperm = o; o = al16(o + 2u * nr);
  L.s_vperm = o; o = al16(o + 2u * ns);
  L.s_dyn = graph_glob ? 0u : o;
  const SlotPlan S = slot_plan(L, D.srow_quads, D.scol_cells, L.rw, L.sw, 0u, ub_glob, 0);  // the largest
  L.U = graph_glob ? o : S.U;
  L.ids = S.ids;
  L.b_size = S.b_size;
  const unsigned p0 = ub_glob ? 0u : L.V;  // where the pre-BP scratch starts
  unsigned u = graph_glob ? S.U : 0u;      // relative to it
  L.p_post = u; u = al16(u + 4u * (ncp + 1));
  L.p_key = u; u = al16(u + 4u * ncp);
  L.p_cns = u; u = al16(u + 16u * (nrp + 1));
  L.p_par = u; u = al16(u + 8u * L.rw);
  const unsigned own = u;
  unsigned srt = al16(L.p_key + 4u * ncp);
  if (!ub_glob && srt < L.s_dyn - L.V) srt = L.s_dyn - L.V;
  if (ub_glob) srt = own;
  L.p_sort = srt;
  const unsigned sort_end = al16(srt + 8u * sn);
  // degrees by rank, check labels, check degrees
  L.p_scr = ub_glob ? srt : L.U - L.V;
  const unsigned scr_end = al16(L.p_scr + 4u * (nsp + 2u * nrp));
  L.p_end = own > sort_end ? own : sort_end;
  if (scr_end > L.p_end) L.p_end = scr_end;
  if (ub_glob) {
    const unsigned slots = (graph_glob ? S.U : 0u) + 8u * L.b_size;
    L.total = L.U + (slots > L.p_end ? slots : L.p_end);
    return L;
  }
  unsigned end = L.U + L.b_size > p0 + L.p_end ? L.U + L.b_size : p0 + L.p_end;
  const unsigned lim = budget > end ? budget : end;
  unsigned q = own;
  auto put = [&](unsigned& at, unsigned bytes, unsigned bit) {
    if (p0 + q + bytes > lim) return;
    at = q;
    q = al16(q + bytes);
    L.pre_stage |= bit;
  };
  if (p0 + q + al16(2u * (L.rw + 1)) + al16(2u * (L.cw + 1)) <= lim) {
    L.q_roff = q; q = al16(q + 2u * (L.rw + 1));
    L.q_coff = q; q = al16(q + 2u * (L.cw + 1));
    L.pre_stage |= kStageOff;
  }
  put(L.q_cent, 128u * D.col_cells, kStageCent);
  put(L.q_rent, 256u * D.row_quads, kStageRent);
  put(L.q_sllr, 4u * ncp, kStageLlr);
  if (p0 + q > end) end = p0 + q;
  L.total = end;
  return L;
}

// The layout with one sign byte per edge and plain CSC / CSR arrays.  No kernel
// takes it: it says which windows a batched step accepts (batch_plan), and the
// layout checks compare the layouts in slices with it.
// lw: the shortened edges' full-window edge ids (s_efull) are kept, which
// only learned weights read
__host__ __device__ inline Layout make_layout(int nr, int nc, int ne, int ns, int es, int nb,
                                              int nslots, bool stage_graph = false, bool ranker = false,
                                              bool lw = true) {
  Layout L{};
  L.rw = (nr + 31) / 32;
  L.cw = (nc + 31) / 32;
  L.sw = (ns + 31) / 32;
  L.nslots = nslots;
  int sn = 1;
  while (sn < nc) sn <<= 1;
  L.sortn = sn;
  unsigned o = 0;
  L.sbits = o; o = al16(o + 4u * L.rw);
  L.cbits = o; o = al16(o + 4u * L.cw);
  L.sel = o; o = al16(o + 2u * ns);
  L.s_colptr = o; o = al16(o + 2u * (ns + 1));
  L.s_colrows = o; o = al16(o + 2u * es);
  L.s_rowptr = o; o = al16(o + 2u * (nr + 1));
  L.s_rowent = o; o = al16(o + 4u * es);
  L.s_llr = o; o = al16(o + 4u * ns);
  L.s_vdeg = o; o = al16(o + 1u * ns);
  L.s_efull = o; o = al16(o + (lw ? 2u * es : 0u));
  L.s_cperm = o; o = al16(o + 2u * nr);
  L.s_vperm = o; o = al16(o + 2u * ns);
  L.rowcnt = o; o = al16(o + 4u * (nr + 1));
  L.res_status = o; o = al16(o + 4u * nb);
  L.res_pm = o; o = al16(o + 8u * nb);
  L.res_ebits = o; o = al16(o + 4u * L.sw * nb);
  L.red = o; o = al16(o + 16u * 32);
  L.misc = o; o = al16(o + 64u);
  const unsigned g0 = o;
  if (stage_graph) {
    L.g_colptr = o; o = al16(o + 2u * (nc + 1));
    L.g_colrows = o; o = al16(o + 2u * ne);
    L.g_rowptr = o; o = al16(o + 2u * (nr + 1));
    L.g_rowent = o; o = al16(o + 4u * ne);
    L.g_llr = o; o = al16(o + 4u * nc);
  }
  L.g_bytes = o - g0;
  L.U = o;
  unsigned u = 0;
  L.p_post = u; u = al16(u + 4u * nc);
  L.p_key = u; u = al16(u + 4u * nc);
  L.p_cns = u; u = al16(u + 16u * nr);
  L.p_sign = u; u = al16(u + 1u * ne);
  L.p_par = u; u = al16(u + 8u * L.rw);
  L.p_sort = u; u = al16(u + 8u * sn);
  L.p_end = u;
  unsigned b = 0;
  L.b_post = b; b = al16(b + 4u * ns);
  L.b_acc = b; b = al16(b + 4u * ns);
  L.b_hfl = b; b = al16(b + 1u * ns);
  L.b_status = b; b = al16(b + 1u * ns);
  L.b_sign = b; b = al16(b + 1u * es);
  L.b_cns = b; b = al16(b + 16u * nr);
  L.b_deg = b; b = al16(b + 4u * nr);
  L.b_sp = b; b = al16(b + 4u * L.rw);
  L.b_unsat = b; b = al16(b + 4u * L.rw);
  L.b_hq = b; b = al16(b + (ranker ? 4u * ns : 0u));
  L.b_size = b;
  unsigned ub = L.p_end > b * (unsigned)nslots ? L.p_end : b * (unsigned)nslots;
  if (!stage_graph) {
    unsigned q = L.p_sort;
    L.q_colptr = q; q = al16(q + 2u * (nc + 1));
    L.q_colrows = q; q = al16(q + 2u * ne);
    L.q_rowptr = q; q = al16(q + 2u * (nr + 1));
    L.q_rowent = q; q = al16(q + 4u * ne);
    L.q_llr = q; q = al16(q + 4u * nc);
    L.q_vperm = q; q = al16(q + 2u * nc);
    L.pre_stage = q <= ub ? 1u : 0u;
  }
  L.total = L.U + ub;
  return L;
}

}  // namespace qd
