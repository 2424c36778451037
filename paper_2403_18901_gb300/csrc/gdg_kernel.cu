// gdg_kernel.cu -- the window decoder, sampler, commit and evaluation kernels.
//
// decode, per shot:
//   a1  window syndrome: bits [row0, row0 + n_rows) of the shot's detectors
//   a2  pre-BP: n_pre flooding min-sum iterations on the full window
//       (Eq. (1)-(4)); a check node by one lane (shot mode) or a lane group
//       (path mode), a variable node by one thread; early stop when H e = s
//       (Sec. II-A), tested inside the next check pass
//   a3  ranking key ((h0+h1)+h2)+h3 of the last four posteriors, the 2w'
//       columns of least (key, column) selected and sorted (Sec. III); the
//       shortened matrix is rebuilt in shared memory with its checks and
//       columns numbered in processing order (descending degree)
//   a4-a7 GDG decision paths (Alg. 2 on the 2^k tree and the side branches of
//       Fig. 2): BP steps of iters_per_step iterations, SELECT-VN (Alg. 1)
//       with aggressive decimation (Alg. 3), guess value by the path id,
//       peeling
//   a8  minimum path metric Eq. (5) over converged paths, ties to the lowest id;
//       without a converged path, path 0 or (fallback rules) the estimate with
//       the fewest unsatisfied (committed, then all) checks
//   (message reuse between windows, optional) the output path's final
//       posteriors kept per window column; the next window's pre-BP starts
//       its first VN->CN messages from them
//
// Two launch shapes run the same path code:
//   shot mode (throughput): persistent CTAs of 8 or 12 warps take shots from
//     a work counter; after the CTA-wide pre-BP the warps take decision paths
//     from a shared-memory queue in a host-planned order, one warp per path;
//     paths resume from snapshots of the prefixes they share with earlier
//     paths, and at every step boundary a warp parks its path for a waiting
//     one with more steps left (snapshots in a per-CTA pool in global memory;
//     see ForkCtx);
//   path mode (latency, small batches): one CTA per (shot, path), of fewer
//     threads and more to an SM the more there are; the path
//     CTAs of a shot form a thread-block cluster that splits the pre-BP over
//     distributed shared memory, each CTA then ranks, shortens and runs its
//     one path with all its threads, stores the result in global scratch,
//     and the last CTA of the shot to arrive (atomic counter, no waiting)
//     picks the winner.
// Every wait is a CTA, warp or cluster barrier, except the bulk-copy
// mbarrier, whose wait is bounded; the path scheduler never waits (a path
// whose snapshot is not ready starts from an earlier one or from the root).
#include <cuda_runtime.h>
#include <math_constants.h>

#include <cfloat>
#include <cstdint>
#include <type_traits>

#include "gdg_kernel.cuh"
#include "qdec_internal.h"

namespace qd {
namespace dev {

constexpr unsigned FULL = 0xffffffffu;
enum { BR_CONVERGED = 0, BR_MAXDEPTH = 1, BR_CONTRADICTION = 2, BR_NOCAND = 3, BR_INTERNAL = 4 };
constexpr int kNone = 0x7fffffff;

// The posterior a decimated VN stores, and that of the dummy column: a check's
// input from it is +inf whatever its message (finite), so it never is the
// smallest or second smallest, has sign 0 and no hard decision.
__device__ __forceinline__ float dead_post() { return CUDART_INF_F; }

__device__ __forceinline__ float flip_sign(float x, uint32_t s) {  // s: the sign at bit 31, other bits 0
  return __uint_as_float(__float_as_uint(x) ^ s);
}

// Eq. (1): mu_{j->i} from the check's record for the edge at position p of
// its entries (low six bits of e); w: the learned weight.  wide: the position
// may be past 31.
template <bool LW>
__device__ __forceinline__ float c2v(const CNState& c, uint32_t e, bool wide, float w) {
  float m = ((c.am ^ e) & 63u) ? c.m1 : c.m2;
  uint32_t sg = c.sg;
  if (wide && (e & 32u)) sg = c.am;
  m = flip_sign(m, __funnelshift_l(0u, sg, e) & 0x80000000u);  // shift by e mod 32
  return LW ? __fmul_rn(w, m) : m;
}

// The maximum, NaN if an operand is NaN (fmaxf returns the other operand then).
__device__ __forceinline__ float max_or_nan(float x, float y) {
  float m;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(x), "f"(y));
  return m;
}

// The inputs a check has seen: two smallest magnitudes, the position of the
// smallest, the parity of the hard decisions it read (bit 31).  The two
// smallest and so every message do not depend on the order of the inputs.
struct CheckAcc {
  float m1, m2;
  uint32_t am, hp;
};

// One input at position u: posterior pv, the previous iteration's record (its
// argmin position oam, two magnitudes, this edge's sign osg at bit 31); before
// the first iteration that record is zero, and so is the message.  Returns the
// bits of v, whose sign the caller collects.  The clip of Eq. (3) bounds every
// magnitude alike, so it is applied to the two smallest at the end.  A
// posterior is never -0 (its prior is positive and x + y = -0 only for
// x = y = -0), nor is the difference of two messages, so the sign bit is the
// comparison with 0, and pv <= 0 is the sign of pv's bits minus one.
template <bool LW>
__device__ __forceinline__ uint32_t check_input(CheckAcc& A, float pv, uint32_t u, uint32_t oam, float om1, float om2,
                                                uint32_t osg, float w, bool first) {
  float m = flip_sign(u == oam ? om2 : om1, osg & 0x80000000u);
  if (LW) m = __fmul_rn(w, m);
  float v = __fsub_rn(pv, m);
  // (an infinite weight: no message before the first iteration, and a dead
  // input stays one)
  if (LW && (first || pv == CUDART_INF_F)) v = pv;
  // (v is NaN where an infinite message met an infinite posterior -- no clip, or
  // learned weights that are not finite.  Such an input counts as +inf: the
  // comparison does not hold, the maximum is NaN and fminf returns its other
  // operand.)
  const float a = fabsf(v);
  A.am = a < A.m1 ? u : A.am;
  A.m2 = fminf(A.m2, max_or_nan(A.m1, a));
  A.m1 = fminf(A.m1, a);
  A.hp ^= __float_as_uint(pv) - 1u;
  return __float_as_uint(v);
}

// The columns of four check entries.  The window graph keeps 16-bit column
// labels (it is staged in shared memory whole, and twice the bytes would cost
// resident CTAs); a shortened graph keeps byte offsets, one instruction less
// per entry.
__device__ __forceinline__ void four_posts(const uint2& e, const char* post, float (&p)[4]) {
  const float* f = (const float*)post;
  p[0] = f[e.x & 0xFFFFu];
  p[1] = f[e.x >> 16];
  p[2] = f[e.y & 0xFFFFu];
  p[3] = f[e.y >> 16];
}
__device__ __forceinline__ void four_posts(const uint4& e, const char* post, float (&p)[4]) {
  p[0] = *(const float*)(post + e.x);
  p[1] = *(const float*)(post + e.y);
  p[2] = *(const float*)(post + e.z);
  p[3] = *(const float*)(post + e.w);
}

// Four inputs at positions u .. u + 3; osg: the old signs, position u at bit
// 31.  The new signs are shifted into sg, one bit each.
template <bool LW>
__device__ __forceinline__ void check_four(CheckAcc& A, const float (&p)[4], uint32_t u, uint32_t oam, float om1,
                                           float om2, uint32_t osg, const float (&w)[4], bool first, uint32_t& sg) {
  sg = __funnelshift_l(check_input<LW>(A, p[0], u, oam, om1, om2, osg, w[0], first), sg, 1);
  sg = __funnelshift_l(check_input<LW>(A, p[1], u + 1, oam, om1, om2, osg << 1, w[1], first), sg, 1);
  sg = __funnelshift_l(check_input<LW>(A, p[2], u + 2, oam, om1, om2, osg << 2, w[2], first), sg, 1);
  sg = __funnelshift_l(check_input<LW>(A, p[3], u + 3, oam, om1, om2, osg << 3, w[3], first), sg, 1);
}

// The record of a check from its inputs and the syndrome bit: magnitudes
// bounded by the clip (an only input gets the clip itself, the minimum over
// the empty set; the first iteration's inputs are priors, not clipped).
template <bool LW>
__device__ __forceinline__ CNState check_record(const CheckAcc& A, uint32_t sg0, uint32_t sg1, uint32_t sbit, bool first,
                                                float alpha, float clip) {
  const float lim = first ? FLT_MAX : clip;
  float m1 = A.m1 == CUDART_INF_F ? clip : fminf(A.m1, lim);
  float m2 = A.m2 == CUDART_INF_F ? clip : fminf(A.m2, lim);
  if (!LW) {
    m1 = __fmul_rn(alpha, m1);
    m2 = __fmul_rn(alpha, m2);
  }
  const uint32_t par = (uint32_t)(__popc(sg0 ^ sg1) + (int)sbit) << 31;
  return CNState{flip_sign(m1, par), flip_sign(m2, par), sg0, (sg1 & ~63u) | A.am};
}

// Learned weights' view of one iteration: entry i's weight is w[ef[i]] (its row
// of the weights, the entries' full-window edges), or w[i] where the weights
// have been put in entry order (ef = nullptr; a type of its own, so that each
// loop is compiled for one of the two).  A column's dummy has no edge and the
// weight 0 (its message has to be +0, which an infinite weight would not give);
// a check's dummies are dead inputs, whatever their weight.
struct LwEdge {
  const float* w;
  const uint16_t* ef;
  __device__ __forceinline__ float one(int i) const {
    const uint32_t e = ef[i];
    return e == kNoEdge ? 0.0f : w[e];
  }
  __device__ __forceinline__ void four(int i, float (&x)[4]) const {
    const uint2 e = *(const uint2*)(ef + i);
    x[0] = w[e.x & 0xFFFFu];
    x[1] = w[e.x >> 16];
    x[2] = w[e.y & 0xFFFFu];
    x[3] = w[e.y >> 16];
  }
};
struct LwOrdered {
  const float* w;
  __device__ __forceinline__ float one(int i) const { return w[i]; }
  __device__ __forceinline__ void four(int i, float (&x)[4]) const {
    const float4 v = *(const float4*)(w + i);
    x[0] = v.x;
    x[1] = v.y;
    x[2] = v.z;
    x[3] = v.w;
  }
};
template <bool LW, class Lw>
__device__ __forceinline__ void lw_four(const Lw& r, int i, bool first, float (&w)[4]) {
  w[0] = w[1] = w[2] = w[3] = 0.0f;
  if (LW && !first) r.four(i, w);
}

// Check-node update of Eq. (1) of one check by one lane.  ent: the lane's
// entries, four at a time, `nq` times, 32 lanes apart (ei: the index of the
// first entry, for the learned weights' edge ids); post: posteriors; rec: its
// record, the previous iteration's on entry.  Returns at bit 31 the parity of
// the hard decisions read, xor the syndrome bit: the test H e = s of the
// iteration before.  What bounds it: issue, ALU instructions above all (half
// rate, about 11 of 14 per entry), and the latency of entry and posterior
// loads, which four entries at a time overlap; the posterior gathers' bank
// conflicts come next.  With a sign byte and an edge id per edge, a NaN test
// and the clip on every input and ragged rows, 5000 shots of [[144,12,12]]
// took 450 ms; in slices, with the signs as bits of the record and the clip on
// the two minima, 354 ms (with all that followed, 231).
template <bool LW, class E, class Lw>
__device__ __forceinline__ uint32_t check_lane(const E* ent, int nq, const char* post, CNState* rec, uint32_t sbit,
                                               float alpha, float clip, const Lw& lw, int ei, bool first) {
  CNState oc = *rec;
  if (first) oc = CNState{0.0f, 0.0f, 0u, 0u};
  const uint32_t oam = oc.am & 63u;
  uint32_t osg = oc.sg;
  CheckAcc A{CUDART_INF_F, CUDART_INF_F, 0u, 0u};
  uint32_t sg0 = 0u, sg1 = 0u;
#pragma unroll 1
  for (int q0 = 0; q0 < nq; q0 += 8) {  // 32 positions to a sign word
    const int q1 = min(nq, q0 + 8);
    uint32_t sg = 0u;
#pragma unroll 1
    for (int q = q0; q < q1; ++q) {
      float w[4];
      lw_four<LW>(lw, ei + 128 * q, first, w);
      float p[4];
      four_posts(ent[32 * q], post, p);
      check_four<LW>(A, p, 4 * q, oam, oc.m1, oc.m2, osg, w, first, sg);
      osg <<= 4;
    }
    sg <<= (32 - 4 * (q1 - q0)) & 31;  // the first position to bit 31
    if (q0 == 0) sg0 = sg;
    else sg1 = sg;
    osg = oc.am;
  }
  *rec = check_record<LW>(A, sg0, sg1, sbit, first, alpha, clip);
  return (A.hp ^ (sbit << 31)) & 0x80000000u;
}

// The same by tpc neighbouring lanes (fours sub, sub + tpc, ...); every lane
// of the group ends with the record.
template <bool LW, class E, class Lw>
__device__ __forceinline__ CNState check_group(const E* ent, int nq, const char* post, CNState oc, uint32_t sbit,
                                               float alpha, float clip, bool first, const Lw& lw, int ei, int sub,
                                               int tpc, bool wide, uint32_t& unsat) {
  if (first) oc = CNState{0.0f, 0.0f, 0u, 0u};
  const uint32_t oam = oc.am & 63u;
  CheckAcc A{CUDART_INF_F, CUDART_INF_F, 0u, 0u};
  uint32_t sg0 = 0u, sg1 = 0u;
#pragma unroll 1
  for (int q = sub; q < nq; q += tpc) {
    float w[4];
    lw_four<LW>(lw, ei + 128 * q, first, w);
    const int sh = (4 * q) & 31;
    uint32_t sg = 0u;
    float p[4];
    four_posts(ent[32 * q], post, p);
    check_four<LW>(A, p, 4 * q, oam, oc.m1, oc.m2, (q < 8 ? oc.sg : oc.am) << sh, w, first, sg);
    if (q < 8) sg0 |= sg << (28 - sh);
    else sg1 |= sg << (28 - sh);
  }
#pragma unroll 1
  for (int off = tpc >> 1; off; off >>= 1) {
    const float x1 = __shfl_xor_sync(FULL, A.m1, off), x2 = __shfl_xor_sync(FULL, A.m2, off);
    const uint32_t xa = __shfl_xor_sync(FULL, A.am, off);
    A.hp ^= __shfl_xor_sync(FULL, A.hp, off);
    sg0 |= __shfl_xor_sync(FULL, sg0, off);
    if (wide) sg1 |= __shfl_xor_sync(FULL, sg1, off);
    A.m2 = fminf(fminf(A.m2, x2), fmaxf(A.m1, x1));
    // equal minima: either position gives the same messages, but every lane of
    // the group has to take the same one
    A.am = x1 < A.m1 || (x1 == A.m1 && xa < A.am) ? xa : A.am;
    A.m1 = fminf(A.m1, x1);
  }
  unsat |= (A.hp ^ (sbit << 31)) & 0x80000000u;
  return check_record<LW>(A, sg0, sg1, sbit, first, alpha, clip);
}

// The parity of a check's hard decisions, at bit 31.
template <class E>
__device__ __forceinline__ uint32_t check_parity(const E* ent, int nq, const char* post) {
  uint32_t hp = 0u;
#pragma unroll 1
  for (int q = 0; q < nq; ++q) {
    float p[4];
    four_posts(ent[32 * q], post, p);
    hp ^= ((__float_as_uint(p[0]) - 1u) ^ (__float_as_uint(p[1]) - 1u)) ^
          ((__float_as_uint(p[2]) - 1u) ^ (__float_as_uint(p[3]) - 1u));
  }
  return hp & 0x80000000u;
}

// What the variable pass walks: this lane's view of the column slices.
template <class Lw>
struct ColView {
  ColClasses K;
  const uint32_t* cent;
  const uint16_t* coff;
  const float* llr;
  const int8_t* status;  // nullptr: every column is active
  const char* cns;
  Lw lw;
  int lane, st;  // the group takes every st-th slice
};

// p + the messages of N entries of this lane's column from cell c0 on, in
// ascending check order (Eq. (2); a dummy adds +0): N record gathers in flight.
template <bool LW, bool WIDE, int N, class Lw>
__device__ __forceinline__ float add_messages(const ColView<Lw>& V, float p, int c0) {
  uint32_t e[N];
  CNState c[N];
  float w[N];
#pragma unroll
  for (int x = 0; x < N; ++x) {
    e[x] = V.cent[32 * (c0 + x) + V.lane];
    w[x] = LW ? V.lw.one(32 * (c0 + x) + V.lane) : 0.0f;
  }
#pragma unroll
  for (int x = 0; x < N; ++x) c[x] = *(const CNState*)(V.cns + (e[x] >> 12));
#pragma unroll
  for (int x = 0; x < N; ++x) p = __fadd_rn(p, c2v<LW>(c[x], e[x], WIDE, w[x]));
  return p;
}

// The variable pass over column slices first, first + st, ...: put(s, p) takes
// the posterior of this lane's column of slice s.  WIDE: edges may have
// positions past 31 (the widest slices always allow it).  A loop per width, so
// that trip counts and offsets are constants, and one slice a trip: two or four
// slices at once overlap more gathers, but the larger loop and the repeated
// slices at its end cost more (2000 shots of [[144,12,12]], three CTAs per SM:
// 106.6 ms with four slices of width one at once, 102.8 ms so; one loop for all
// widths, 126 ms).
template <bool LW, bool WIDE, class Lw, class Put>
__device__ __forceinline__ void column_pass(const ColView<Lw>& V, int first, Put put) {
  constexpr int kLow = kWideSlice - 1;
  const ColClasses& K = V.K;
  int s = first;
  auto active = [&]() { return !V.status || V.status[32 * s + V.lane] == -1; };  // (asked for before the gathers)
#pragma unroll 1
  for (; s < K.n4; s += V.st) {
    int c0 = V.coff[s] & kLow;
    const int c1 = V.coff[s + 1] & kLow;
    float p = V.llr[32 * s + V.lane];
#pragma unroll 1
    for (; c0 + 3 <= c1; c0 += 3) p = add_messages<LW, true, 3>(V, p, c0);
#pragma unroll 1
    for (; c0 < c1; ++c0) p = add_messages<LW, true, 1>(V, p, c0);
    if (active()) put(s, p);
  }
  auto narrow = [&](auto width, int end, int b) {  // cells from b + N s on
    constexpr int N = decltype(width)::value;
#pragma unroll 1
    for (; s < end; s += V.st) {
      const bool act = active();
      const float p = add_messages<LW, WIDE, N>(V, V.llr[32 * s + V.lane], b + N * s);
      if (act) put(s, p);
    }
  };
  narrow(std::integral_constant<int, 3>{}, K.n3, (V.coff[K.n4] & kLow) - 3 * K.n4);
  narrow(std::integral_constant<int, 2>{}, K.n2, (V.coff[K.n3] & kLow) - 2 * K.n3);
  narrow(std::integral_constant<int, 1>{}, K.n1, (V.coff[K.n2] & kLow) - K.n2);
}

__device__ __forceinline__ uint32_t bit_of(const uint32_t* w, int j) { return (w[j >> 5] >> (j & 31)) & 1u; }

// ---- bulk asynchronous copies global -> shared (TMA, cp.async.bulk) ----
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// A CTA's staging state: its mbarrier (one arrival + transaction bytes per
// phase), the parity of the phase in flight, a shared flag that turns the
// bulk path off after a wait ran out, and the counter such events go to.
struct Stager {
  uint64_t* bar;
  int* off;
  long long* err;
  unsigned phase;
};

__device__ __forceinline__ Stager stager_init(char* where, long long* err) {
  Stager st{(uint64_t*)where, (int*)(where + 8), err, 0u};
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(st.bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    *st.off = 0;
  }
  __syncthreads();
  return st;
}

struct StagePiece {
  void* dst;
  const void* src;
  unsigned bytes;
};

// Copies the pieces into shared memory, all threads calling: one bulk copy
// per piece issued by thread 0, completion tracked on the mbarrier, every
// thread waiting with a bound of ~2^31 cycles.  Pieces that are not 16-byte
// aligned in address and size, an empty list, or a wait that ran out (counted
// in *err; the bulk path then stays off for this CTA) use plain loads.
template <int n>
__device__ __forceinline__ void stage_pieces(Stager& st, const StagePiece (&pc)[n]) {
  bool aligned = true;
  unsigned tot = 0;
#pragma unroll
  for (int i = 0; i < n; ++i) {
    aligned = aligned && (((smem_u32(pc[i].dst) | (unsigned)(uintptr_t)pc[i].src | pc[i].bytes) & 15u) == 0u);
    tot += pc[i].bytes;
  }
  __syncthreads();  // every earlier access to these bytes has finished
  if (aligned && tot > 0 && !*st.off) {
    if (threadIdx.x == 0) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(st.bar)), "r"(tot)
                   : "memory");
#pragma unroll
      for (int i = 0; i < n; ++i)
        if (pc[i].bytes)
          asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                           smem_u32(pc[i].dst)),
                       "l"(pc[i].src), "r"(pc[i].bytes), "r"(smem_u32(st.bar))
                       : "memory");
    }
    unsigned ok = 0;
    const long long t0 = clock64();
#pragma unroll 1
    while (!ok && clock64() - t0 < (1ll << 31)) {
      asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                   : "=r"(ok)
                   : "r"(smem_u32(st.bar)), "r"(st.phase)
                   : "memory");
    }
    st.phase ^= 1u;
    if (__syncthreads_and(ok != 0)) return;
    if (threadIdx.x == 0) {
      *st.off = 1;
      atomicAdd((unsigned long long*)st.err, 1ull);
    }
  }
#pragma unroll
  for (int i = 0; i < n; ++i) {
    const uint16_t* s16 = (const uint16_t*)pc[i].src;
    uint16_t* d16 = (uint16_t*)pc[i].dst;
#pragma unroll 1
    for (unsigned x = threadIdx.x; x < pc[i].bytes / 2; x += blockDim.x) d16[x] = s16[x];
  }
  __syncthreads();
}

// Learned weights of iteration t (1-based): w[min(t, T)], never a row before
// the first.
__device__ __forceinline__ const float* weight_row(const float* wts, int wT, int wE, int t) {
  const int row = t < 1 ? 0 : (t < wT ? t : wT) - 1;
  return wts + (size_t)row * wE;
}

// order-preserving map of a float to uint32 (-0 and +0 equal)
__device__ __forceinline__ uint32_t ordkey(float f) {
  if (f == 0.0f) f = 0.0f;
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Lanes per check of a decision path run by a whole CTA: two where that takes
// one round of threads / lanes checks, else one.  A shortened graph's checks
// have a few entries each, so more lanes mostly add reduction steps (one
// [[144,12,12]] shot, 11 windows, when this was chosen: 8.0 ms with up to eight
// lanes in two rounds, 6.9 ms with four in one, 6.7 ms with two; 5.9 ms with the
// steps that followed).
__host__ __device__ inline int path_lanes_per_check(int threads, int n_checks) {
  return threads / 2 >= n_checks ? 2 : 1;
}

// lexicographic (value, index) minimum over the warp
__device__ __forceinline__ void warp_argmin(float& v, int& k) {
#pragma unroll
  for (int off = 16; off; off >>= 1) {
    const float xv = __shfl_xor_sync(FULL, v, off);
    const int xk = __shfl_xor_sync(FULL, k, off);
    if (xv < v || (xv == v && xk < k)) {
      v = xv;
      k = xk;
    }
  }
}

__device__ __forceinline__ int warp_incl_scan(int v, int lane) {
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(FULL, v, off);
    if (lane >= off) v += y;
  }
  return v;
}

// ---- cooperative groups of threads that run one decision path ----
struct WarpGrp {  // one warp
  int rank;
  static constexpr int size = 32;
  static constexpr bool kWarp = true;
  __device__ void sync() const { __syncwarp(); }
  __device__ bool all(bool p) const { return __all_sync(FULL, p); }
  __device__ bool any(bool p) const { return __any_sync(FULL, p); }
  __device__ unsigned min_u(unsigned v) const { return __reduce_min_sync(FULL, v); }
  __device__ int sum_i(int v) const { return (int)__reduce_add_sync(FULL, (unsigned)v); }
  __device__ long long sum_ll(long long v) const {
#pragma unroll
    for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(FULL, v, off);
    return v;
  }
  __device__ double sum_d(double v) const {
#pragma unroll
    for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(FULL, v, off);
    return v;
  }
  __device__ void argmin(float& v, int& k) const { warp_argmin(v, k); }
  // SELECT-VN's reductions in one: two lexicographic argmins and a count;
  // every lane's shared-memory writes are visible after it
  __device__ void select_reduce(float& bv, int& bk, float& tv, int& tk, int& n) const {
    warp_argmin(bv, bk);
    warp_argmin(tv, tk);
    n = (int)__reduce_add_sync(FULL, (unsigned)n);
    __syncwarp();
  }
};

struct CtaGrp {  // the whole CTA; every member must call every primitive
  int rank, size;
  static constexpr bool kWarp = false;
  char* red;  // >= 32 * 16 bytes of shared memory
  __device__ void sync() const { __syncthreads(); }
  __device__ bool all(bool p) const { return __syncthreads_and(p) != 0; }
  __device__ bool any(bool p) const { return __syncthreads_or(p) != 0; }
  // Reductions: each warp's result through shared memory, then every warp
  // reduces the (at most 32) results again, one per lane: a loop over them
  // would be as many shared-memory round trips in a row.
  template <class T>
  __device__ T exchange(T v, T none) const {
    T* r = (T*)red;
    __syncthreads();
    if ((rank & 31) == 0) r[rank >> 5] = v;
    __syncthreads();
    return (rank & 31) < (size >> 5) ? r[rank & 31] : none;
  }
  __device__ unsigned min_u(unsigned v) const {
    return __reduce_min_sync(FULL, exchange(__reduce_min_sync(FULL, v), 0xFFFFFFFFu));
  }
  __device__ int sum_i(int v) const {
    return (int)__reduce_add_sync(FULL, exchange(__reduce_add_sync(FULL, (unsigned)v), 0u));
  }
  template <class T>
  __device__ T sum(T v) const {
#pragma unroll
    for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(FULL, v, off);
    v = exchange(v, (T)0);
#pragma unroll
    for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(FULL, v, off);
    return v;
  }
  __device__ long long sum_ll(long long v) const { return sum(v); }
  __device__ double sum_d(double v) const { return sum(v); }
  __device__ void argmin(float& v, int& k) const {
    warp_argmin(v, k);
    const unsigned long long x =
        exchange(((unsigned long long)__float_as_uint(v) << 32) | (unsigned)k,
                 ((unsigned long long)__float_as_uint(CUDART_INF_F) << 32) | (unsigned)kNone);
    v = __uint_as_float((unsigned)(x >> 32));
    k = (int)(unsigned)x;
    warp_argmin(v, k);
  }
  // SELECT-VN's reductions in one exchange: two lexicographic argmins and a
  // count, for at most 16 warps (the path-mode CTA); every thread's
  // shared-memory writes are visible after it
  __device__ void select_reduce(float& bv, int& bk, float& tv, int& tk, int& n) const {
    warp_argmin(bv, bk);
    warp_argmin(tv, tk);
    n = (int)__reduce_add_sync(FULL, (unsigned)n);
    uint4* r = (uint4*)red;
    int* r_n = (int*)(red + 256);
    const int lane = rank & 31;
    __syncthreads();
    if (lane == 0) {
      r[rank >> 5] = make_uint4(__float_as_uint(bv), (unsigned)bk, __float_as_uint(tv), (unsigned)tk);
      r_n[rank >> 5] = n;
    }
    __syncthreads();
    const bool in = lane < (size >> 5);
    const uint4 x = in ? r[lane] : make_uint4(__float_as_uint(CUDART_INF_F), (unsigned)kNone,
                                              __float_as_uint(CUDART_INF_F), (unsigned)kNone);
    bv = __uint_as_float(x.x);
    bk = (int)x.y;
    tv = __uint_as_float(x.z);
    tk = (int)x.w;
    warp_argmin(bv, bk);
    warp_argmin(tv, tk);
    n = (int)__reduce_add_sync(FULL, in ? (unsigned)r_n[lane] : 0u);
  }
};

// The shortened graph in slices (gdg_kernel.cuh).
struct ShortG {
  int nr, ns, rw, cw;  // checks, columns, and their slices
  int rwz;             // non-empty check slices
  const uint32_t *rent, *cent;  // rent: byte offsets of the columns' posteriors
  const uint16_t *roff, *coff;
  const float* llr;
  const uint8_t* vdeg;
  const uint32_t* sbits;
  const uint16_t *ref, *cef;  // full-window edge of each check / column entry (learned weights)
  const ColClasses* cls;
  const float* wts;
  int wT, wE;
  int rpb;  // window rows per block (block of a column = its first row / rpb)
  const uint16_t* sel;    // short column -> window column
  // Checks and short columns are numbered by descending degree (ties by
  // window row / rank); these map a label back to the window row and to the
  // ranked column, whose order decides every tie.
  const uint16_t* cperm;
  const uint16_t* vperm;
  int ncr;  // window rows [0, ncr) are the ones the window commits

  __device__ __forceinline__ int col_slice(int k) const { return (int)(coff[k >> 5] & (kWideSlice - 1)); }
  // check label of column k's u-th entry (u < vdeg[k])
  __device__ __forceinline__ const uint32_t* col_ents(int k) const { return cent + col_slice(k) * 32 + (k & 31); }
};

struct Slot {
  float *post, *acc;
  uint8_t* hfl;
  int8_t* status;
  CNState* cns;
  uint8_t* deg;  // active VNs per check
  uint32_t *sp, *unsat;
  int8_t* hq;  // ranker only: the last four posteriors as round(2 clamp(x, 63.5)), oldest first
};

__device__ __forceinline__ Slot make_slot(char* base, const SlotPlan& S) {
  return Slot{(float*)base,                 (float*)(base + S.b_acc),      (uint8_t*)(base + S.b_hfl),
              (int8_t*)(base + S.b_status), (CNState*)(base + S.b_cns),    (uint8_t*)(base + S.b_deg),
              (uint32_t*)(base + S.b_sp),   (uint32_t*)(base + S.b_unsat), (int8_t*)(base + S.b_hq)};
}

// Fix column k to v while other lanes fix others; returns its degree.
__device__ __forceinline__ int decimate_atomic(const ShortG& G, const Slot& B, int k, int v) {
  B.status[k] = (int8_t)v;
  B.post[k] = dead_post();
  const uint32_t* ce = G.col_ents(k);
  const int d = G.vdeg[k];
#pragma unroll 1
  for (int u = 0; u < d; ++u) {
    const int j = (int)(ce[32 * u] >> 16);
    atomicSub((uint32_t*)B.deg + (j >> 2), 1u << (8 * (j & 3)));  // counts stay >= 0: no borrow
    if (v) atomicXor(&B.sp[j >> 5], 1u << (j & 31));
  }
  return d;
}

__device__ __forceinline__ int decimate_one(const ShortG& G, const Slot& B, int k, int v) {
  B.status[k] = (int8_t)v;
  B.post[k] = dead_post();
  const uint32_t* ce = G.col_ents(k);
  const int d = G.vdeg[k];
#pragma unroll 1
  for (int u = 0; u < d; ++u) {
    const int r = (int)(ce[32 * u] >> 16);
    B.deg[r] -= 1;
    if (v) B.sp[r >> 5] ^= 1u << (r & 31);
  }
  return d;
}

// Peeling (Sec. IV): repeatedly fix the lone active VN of a degree-one check
// to the check's current syndrome; a check left with no active VN and
// syndrome 1 is a contradiction.  One check at a time, always the lowest-index
// degree-one check, after testing every check for a contradiction (this order
// also fixes the partial state of a path killed by a contradiction).
// Returns #peeled, -1 (contradiction) or -2 (inconsistent degree count);
// subtracts the edges of the peeled VNs from rank 0's `act`.
template <class Grp>
__device__ int peel(const ShortG& G, const Slot& B, const Grp& g, int& act) {
  int npeel = 0;
#pragma unroll 1
  for (int guard = 0; guard <= G.ns + 1; ++guard) {
    bool contra = false;
    int cand = kNone;  // (window row << 16) | label of the lowest degree-one check
#pragma unroll 1
    for (int x = g.rank; x < 8 * G.rw; x += g.size) {  // four checks' counts at a time
      const uint32_t d4 = ((const uint32_t*)B.deg)[x];
      const uint32_t low = d4 & 0xFEFEFEFEu;
      if (!((low - 0x01010101u) & ~low & 0x80808080u)) continue;  // none is 0 or 1 (a borrow only adds hits)
      const uint32_t s4 = B.sp[x >> 3] >> (4 * (x & 7));
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        const int d = (int)((d4 >> (8 * y)) & 0xFFu), j = 4 * x + y;
        if (d == 0) {
          if ((s4 >> y) & 1u) contra = true;  // (the padding's syndrome bits are 0)
        } else if (d == 1) {
          cand = min(cand, ((int)G.cperm[j] << 16) | j);
        }
      }
    }
    if (g.any(contra)) return -1;
    const int jc = (int)g.min_u((unsigned)cand);
    if (jc == kNone) return npeel;
    const int j = jc & 0xFFFF;
    int found = kNone;
    const uint32_t* re = G.rent + (int)G.roff[j >> 5] * 128 + 4 * (j & 31);
    const int width = 4 * (int)(G.roff[(j >> 5) + 1] - G.roff[j >> 5]);
#pragma unroll 1
    for (int u = g.rank; u < width; u += g.size) {
      const int i = (int)(re[128 * (u >> 2) + (u & 3)] >> 2);
      if (i < G.ns && B.status[i] == -1) found = i;  // (the dummy column is no VN)
    }
    const int i = (int)g.min_u((unsigned)found);
    if (i == kNone) return -2;
    const int v = (int)bit_of(B.sp, j);
    g.sync();
    if (g.rank == 0) act -= decimate_one(G, B, i, v);
    g.sync();
    ++npeel;
  }
  return -2;
}

// ---- learned decimation ranker (replaces the argmin of Alg. 1) ----
// score = W2 . relu(W1 x + b1) + b2 over the candidate features
//   x = (L/4, h0, h1, h2, h3 on the 1/2 grid clamped to +-63.5, #unsatisfied
//        neighbour checks (<= 127), static degree, block of the first
//        detector (<= 255)).
// With W1 on the 2^-6 grid in [-2, 2] and b1 on the 2^-7 grid in [-512, 512] every layer-1
// partial sum is a multiple of 2^-7 below 2^13: the BF16 tensor-core product
// with FP32 accumulation is exact, in any order.  Layer 2 runs in FP32 in one
// fixed order per candidate: s_q = sum over t = 0..7, c = 0..1 of
// W2[u] h[u], u = 8t + 2q + c (lane q of the quad that holds those units in
// the MMA accumulator layout), score = ((s_0 + s_1) + (s_2 + s_3)) + b2.

__device__ __forceinline__ float qfeat(float x) {
  return (float)__float2int_rn(2.0f * fminf(fmaxf(x, -63.5f), 63.5f)) * 0.5f;
}
__device__ __forceinline__ int8_t qhist(float x) { return (int8_t)__float2int_rn(2.0f * fminf(fmaxf(x, -63.5f), 63.5f)); }

// two BF16-exact floats as a packed pair (low half = first)
__device__ __forceinline__ uint32_t bf16x2_exact(float lo, float hi) {
  return (__float_as_uint(lo) >> 16) | (__float_as_uint(hi) & 0xFFFF0000u);
}

// D = A B + C, m16n8k8, BF16 inputs, FP32 accumulate
__device__ __forceinline__ void mma_m16n8k8_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0, float c0,
                                                 float c1) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%7,%8,%9,%10};\n"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(b0), "f"(c0), "f"(c1), "f"(c0), "f"(c1));
}

__device__ __forceinline__ bool ranker_candidate(const ShortG& G, const Slot& B, int k) {
  return k < G.ns && B.status[k] == -1 && G.vdeg[k] > 2;
}

// Features 2 tig and 2 tig + 1 of short column k (zero for a non-candidate).
__device__ __forceinline__ uint32_t ranker_pair(const ShortG& G, const Slot& B, int k, bool cand, int tig) {
  if (!cand) return 0u;
  float lo, hi;
  const uint32_t h4 = *(const uint32_t*)(B.hq + 4 * k);
  const float hv0 = (float)(int8_t)(h4 & 0xFF) * 0.5f, hv1 = (float)(int8_t)((h4 >> 8) & 0xFF) * 0.5f;
  const float hv2 = (float)(int8_t)((h4 >> 16) & 0xFF) * 0.5f, hv3 = (float)(int8_t)(h4 >> 24) * 0.5f;
  if (tig == 0) {
    lo = qfeat(__fmul_rn(B.acc[k], 0.25f));
    hi = hv0;
  } else if (tig == 1) {
    lo = hv1;
    hi = hv2;
  } else if (tig == 2) {
    int nus = 0;
    const uint32_t* ce = G.col_ents(k);
#pragma unroll 1
    for (int u = 0; u < G.vdeg[k]; ++u) nus += bit_of(B.unsat, (int)(ce[32 * u] >> 16));
    lo = hv3;
    hi = (float)min(nus, 127);
  } else {
    lo = (float)G.vdeg[k];
    hi = (float)min(G.cperm[*G.col_ents(k) >> 16] / G.rpb, 255);
  }
  return bf16x2_exact(lo, hi);
}

// Highest score over the candidates (ties to the lowest ranked column), as
// (-score, (ranked column << 16) | label) for the group's lexicographic
// argmin.  Each warp of the group scores tiles of 16 consecutive labels;
// every lane of the group calls.
template <class Grp>
__device__ void ranker_select(const KParams& P, const ShortG& G, const Slot& B, const Grp& g, float& nv, int& nk) {
  const int lane = g.rank & 31, wid = g.rank >> 5, nw = g.size >> 5;
  const int gi = lane >> 2, tig = lane & 3, qb = lane & ~3;
  const float* b1 = P.rkq + 512;
  const float* w2 = P.rkq + 576;
  const float b2 = P.rkq[640];
  nv = CUDART_INF_F;
  nk = kNone;
#pragma unroll 1
  for (int t0 = 16 * wid; t0 < G.ns; t0 += 16 * nw) {
    const int r0 = t0 + gi, r1 = r0 + 8;
    const bool c0 = ranker_candidate(G, B, r0), c1 = ranker_candidate(G, B, r1);
    const uint32_t a0 = ranker_pair(G, B, r0, c0, tig), a1 = ranker_pair(G, B, r1, c1, tig);
    float s0 = 0.0f, s1 = 0.0f;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int u = 8 * t + 2 * tig;
      float d[4];
      mma_m16n8k8_bf16(d, a0, a1, P.rkb[32 * t + lane], b1[u], b1[u + 1]);
      const float wa = w2[u], wb = w2[u + 1];
      s0 = __fadd_rn(s0, __fmul_rn(wa, d[0] > 0.0f ? d[0] : 0.0f));
      s0 = __fadd_rn(s0, __fmul_rn(wb, d[1] > 0.0f ? d[1] : 0.0f));
      s1 = __fadd_rn(s1, __fmul_rn(wa, d[2] > 0.0f ? d[2] : 0.0f));
      s1 = __fadd_rn(s1, __fmul_rn(wb, d[3] > 0.0f ? d[3] : 0.0f));
    }
    float q[4], p[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      q[i] = __shfl_sync(FULL, s0, qb + i);
      p[i] = __shfl_sync(FULL, s1, qb + i);
    }
    const float sc0 = __fadd_rn(__fadd_rn(__fadd_rn(q[0], q[1]), __fadd_rn(q[2], q[3])), b2);
    const float sc1 = __fadd_rn(__fadd_rn(__fadd_rn(p[0], p[1]), __fadd_rn(p[2], p[3])), b2);
    // ties to the lowest ranked column: (column << 16) | label
    if (c0) {
      const int pk = ((int)G.vperm[r0] << 16) | r0;
      if (-sc0 < nv || (-sc0 == nv && pk < nk)) {
        nv = -sc0;
        nk = pk;
      }
    }
    if (c1) {
      const int pk = ((int)G.vperm[r1] << 16) | r1;
      if (-sc1 < nv || (-sc1 == nv && pk < nk)) {
        nv = -sc1;
        nk = pk;
      }
    }
  }
  g.argmin(nv, nk);
}

// Records of every candidate of this step (path 0 only), in any order.
template <class Grp>
__device__ void dump_candidates(const KParams& P, const ShortG& G, const Slot& B, const Grp& g, long long shot, int D,
                                int gsel) {
#pragma unroll 1
  for (int k = g.rank; k < G.ns; k += g.size) {
    if (!ranker_candidate(G, B, k)) continue;
    const uint32_t h4 = *(const uint32_t*)(B.hq + 4 * k);
    int nus = 0;
    const uint32_t* ce = G.col_ents(k);
#pragma unroll 1
    for (int u = 0; u < G.vdeg[k]; ++u) nus += bit_of(B.unsat, (int)(ce[32 * u] >> 16));
    const float L = B.acc[k];
    const int pos = atomicAdd(P.dump_n, 1);
    if (pos >= P.dump_cap) continue;
    RankRec r;
    r.x[0] = qfeat(__fmul_rn(L, 0.25f));
    r.x[1] = (float)(int8_t)(h4 & 0xFF) * 0.5f;
    r.x[2] = (float)(int8_t)((h4 >> 8) & 0xFF) * 0.5f;
    r.x[3] = (float)(int8_t)((h4 >> 16) & 0xFF) * 0.5f;
    r.x[4] = (float)(int8_t)(h4 >> 24) * 0.5f;
    r.x[5] = (float)min(nus, 127);
    r.x[6] = (float)G.vdeg[k];
    r.x[7] = (float)min(G.cperm[*G.col_ents(k) >> 16] / G.rpb, 255);
    r.shot = (int32_t)shot;
    r.wcol = G.sel[G.vperm[k]];
    r.depth = (int16_t)D;
    r.path = 0;
    r.flags = (L <= 0.0f ? 1 : 0) | (k == gsel ? 2 : 0);
    P.dump[pos] = r;
  }
}

// Eq. (5): the summed priors of the path's estimate (decimated values and the
// hard decisions of the active VNs), in FP64 (exact: every prior lies in
// (2^-15, 16), so every partial sum is exact in any order).
template <class Grp>
__device__ double path_metric(const ShortG& G, const Slot& B, const Grp& g) {
  double s = 0.0;
#pragma unroll 1
  for (int k = g.rank; k < G.ns; k += g.size) {
    const int st8 = B.status[k];
    if (st8 == 1 || (st8 == -1 && B.post[k] <= 0.0f)) s += (double)G.llr[k];
  }
  return g.sum_d(s);
}

// H e = s for the current decisions (Eq. (4), decimated VNs through s'):
// writes every check's unsatisfied bit to B.unsat, for every lane of the group
// to read once it has returned, and returns whether any is unsatisfied.  Checks
// in label order, one per lane.
template <class Grp>
__device__ bool parity_pass(const ShortG& G, const Slot& B, const Grp& g) {
  bool any = false;
#pragma unroll 1
  for (int s = g.rank >> 5; s < G.rw; s += g.size >> 5) {
    const int lane = g.rank & 31;
    const uint32_t sw = B.sp[s];
    if (s >= G.rwz) {  // checks without columns
      if (lane == 0) B.unsat[s] = sw;
      any |= sw != 0u;
      continue;
    }
    const uint32_t hp = (((sw >> lane) & 1u) << 31) ^
                        check_parity((const uint4*)G.rent + (int)G.roff[s] * 32 + lane,
                                     (int)G.roff[s + 1] - (int)G.roff[s], (const char*)B.post);
    const unsigned m = __ballot_sync(FULL, (hp >> 31) != 0u);
    if (lane == 0) B.unsat[s] = m;
    any |= m != 0u;
  }
  if constexpr (Grp::kWarp) __syncwarp();  // (a warp's vote orders no memory, a CTA's is a barrier)
  return g.any(any);
}

struct PathOut {
  int* status;
  double* pm;
  uint32_t* ebits;
  BranchTrace* btr;
  StepTrace* st;
  int8_t* fstat;
  long long* visits;  // accumulates active edge visits, the path's shared prefix included
  long long* exec;    // accumulates the active edge visits this launch executed (nullable)
  long long shot;
  float* keep;        // message reuse: this path's final values by label (nullable)
};

// Shot mode's shared path prefixes.  Paths that made the same decisions at
// depths 1..D-1 are in the same state after the BP of step D (that BP does
// not depend on the path: both P_A flags of Alg. 3 are kept), so a path can
// resume there from a snapshot another path left instead of recomputing the
// prefix from the root.  A snapshot is a 32-byte header (depth, iterations,
// iterations since the messages were initialised, the `first` flag, the
// producing path, the active edges, the prefix's edge visits) and a copy of
// the slot.
//
// Preemption (sched): the paths of a shot outnumber the warps, and the main
// branch is the longest, so a fixed assignment leaves warps idle at the end
// of the shot.  At every step boundary a warp compares the steps its path
// has left with those of the waiting paths -- parked paths, and queued paths
// whose planned snapshot is ready -- and when one has more than one step
// more, it parks its own path (a snapshot of the same form in the path's own
// buffer) and switches to it: longest remaining work first.  Path states
// (sched words): 0 queued, 1 running, 2 | D << 8 parked after the BP of
// step D, 3 done.
struct ForkCtx {
  const char* src;       // snapshot to resume from (nullptr: from the root)
  const int16_t* chain;  // this path's snapshot node by depth (index D - 1), -1: none; nullptr: no snapshots
  int* flags;            // per node: 0 free, 1 being written, 2 ready
  char* pool;            // this CTA's snapshots, `stride` bytes apart: nodes, then one per path
  unsigned stride;
  char* slot;            // this warp's slot and its size
  unsigned slot_bytes;
  const StepTrace* st0;  // the shot's step records (path p at st0 + p * dmx), or nullptr
  unsigned* sched;       // per path state word (nullptr: no preemption)
  const int16_t* fnode;  // per path: its planned snapshot node (-1: none) and that node's depth
  const int16_t* fdep;
  int n_nodes;
};
constexpr unsigned kSnapHeader = kSnapHeaderBytes;
enum { PS_QUEUED = 0, PS_RUNNING = 1, PS_PARKED = 2, PS_DONE = 3 };

// Snapshot of a path's state after the BP of step D (all lanes of the group).
template <class Grp>
__device__ void write_snapshot(char* dst, const ForkCtx& F, const Grp& g, int D, int iters, int tw, bool first,
                               int producer, int act, long long vs) {
  if (g.rank == 0) {
    int* h = (int*)dst;
    __stcg(h, D);
    __stcg(h + 1, iters);
    __stcg(h + 2, tw);
    __stcg(h + 3, first ? 1 : 0);
    __stcg(h + 4, producer);
    __stcg(h + 5, act);
    __stcg((long long*)(dst + 24), vs);
  }
  const uint4* s4 = (const uint4*)F.slot;
  uint4* d4 = (uint4*)(dst + kSnapHeader);
#pragma unroll 4
  for (unsigned x = g.rank; x < F.slot_bytes / 16u; x += g.size) __stcg(d4 + x, s4[x]);
  __threadfence();  // the snapshot and this path's decision records before its flag
  g.sync();
}

// The waiting path with the most steps left, if more than `least` (every lane
// of the warp looks at a path; the lowest id among equals): a parked path, or
// a queued one whose planned snapshot is ready.  -1: none; w: its state word.
__device__ __forceinline__ int longest_waiting(const KParams& P, const ForkCtx& F, int lane, int least, unsigned& w) {
  unsigned key = 0, kw = 0;
#pragma unroll 1
  for (int p = lane; p < P.nb; p += 32) {
    const unsigned x = *(volatile unsigned*)&F.sched[p];
    int at = 0;
    if ((x & 3u) == PS_PARKED) at = (int)(x >> 8);
    else if (x == PS_QUEUED && F.fnode[p] >= 0 && *(volatile int*)&F.flags[F.fnode[p]] == 2) at = F.fdep[p];
    if (!at) continue;
    const int rem = path_dmax(P, p, path_split(P, p)) - at + 1;
    const unsigned k = rem > least ? ((unsigned)rem << 8) | (255u - (unsigned)p) : 0u;
    if (k > key) {
      key = k;
      kw = x;
    }
  }
  const unsigned best = __reduce_max_sync(FULL, key);
  if (!best) return -1;
  const int c = 255 - (int)(best & 255u);
  w = __shfl_sync(FULL, kw, c & 31);
  return c;
}

// Check-node update of Eq. (1) over the active VNs of one decision path; a
// warp takes a slice with one check per lane, a CTA tpc lanes per check.  Each
// check also takes the parity of its active VNs' hard decisions (Eq. (4)) from
// the posteriors it reads: for it >= 2 this pass is the convergence test
// H e = s of the previous iteration (Sec. II-A).  Returns whether this lane saw
// an unsatisfied check.
template <bool LW>
__device__ __forceinline__ bool check_pass_warp(const KParams& P, const ShortG& G, const Slot& B, int lane, bool first,
                                                int tw) {
  LwEdge lw{nullptr, G.ref};
  if (LW && !first) lw.w = weight_row(G.wts, G.wT, G.wE, tw);
  uint32_t unsat = 0u;
  int r0 = 0;
#pragma unroll 1
  for (int s = 0; s < G.rwz; ++s) {
    const int r1 = G.roff[s + 1];
    unsat |= check_lane<LW>((const uint4*)G.rent + r0 * 32 + lane, r1 - r0, (const char*)B.post, B.cns + 32 * s + lane,
                            (B.sp[s] >> lane) & 1u, P.alpha, P.clip, lw, (r0 * 32 + lane) * 4, first);
    r0 = r1;
  }
  // checks without columns are unsatisfied when their syndrome bit is set
#pragma unroll 1
  for (int s = G.rwz + lane; s < G.rw; s += 32) unsat |= B.sp[s];
  return unsat != 0u;
}

template <bool LW>
__device__ __forceinline__ bool check_pass_cta(const KParams& P, const ShortG& G, const Slot& B, int R, int S, int tpc,
                                               bool first, int tw) {
  LwEdge lw{nullptr, G.ref};
  if (LW && !first) lw.w = weight_row(G.wts, G.wT, G.wE, tw);
  const int nrp = 32 * G.rwz, per = S / tpc, sub = R & (tpc - 1);
  uint32_t unsat = 0u;
#pragma unroll 1
  for (int s = G.rwz + R; s < G.rw; s += S) unsat |= B.sp[s];  // checks without columns
#pragma unroll 1
  for (int b = 0; b < nrp; b += per) {
    const int j0 = b + R / tpc;
    const int j = j0 < nrp ? j0 : nrp - 1, s = j >> 5;
    const int r0 = G.roff[s], nq = j0 < nrp ? (int)G.roff[s + 1] - r0 : 0;
    const uint32_t sbit = (B.sp[s] >> (j & 31)) & 1u;
    uint32_t u = 0u;
    const CNState rec =
        check_group<LW>((const uint4*)G.rent + r0 * 32 + (j & 31), nq, (const char*)B.post, B.cns[j], sbit, P.alpha,
                        P.clip, first, lw, (r0 * 32 + (j & 31)) * 4, sub, tpc, (G.coff[0] & kWideSlice) != 0, u);
    if (sub == 0 && j0 < nrp) {
      B.cns[j] = rec;
      unsat |= u;
    }
  }
  return unsat != 0u;
}

// One decision path of Alg. 2 on the shortened window, run by group g.
// LW: learned per-edge weights instead of alpha (compiled separately so the
// plain decoder carries no weight lookups).
// Returns -1 when the path is finished, or (preemption) the path this group
// switches to after parking this one; *claimed is the state word it took.
template <bool LW, class Grp>
__device__ int run_path(const KParams& P, const ShortG& G, const Slot& B, int id, const Grp& g,
                        const PathOut& out, int dmx, const ForkCtx& F, unsigned* claimed = nullptr) {
  const int nr = G.nr, ns = G.ns, R = g.rank, S = g.size;
  // Fig. 2: main branch (id 0), tree branches, side branches (split > 0),
  // which keep the main-branch thresholds up to and including their split
  const int split = path_split(P, id);
  const int d_reinit = path_reinit(P, id, split);
  const int dmax = path_dmax(P, id, split);
  auto main_rules = [&](int D) { return id == 0 || (split && D <= split); };
  int status = BR_MAXDEPTH, depth = 0, iters = 0;
  int tw = 0;  // iterations since the messages were (re)initialised (learned weights)
  long long visits = 0, inherited = 0;  // executed here / the resumed prefix's (lane 0)
  int act = 0;  // active edges, summed over the lanes (each subtracts what it decimates)
  double pm = CUDART_INF;
  bool first = true;
  int D0 = 1;  // first depth of this run: resumed runs start at its SELECT-VN
  if (F.src) {
    // resume from a snapshot taken after the BP of step D0 by a path with the
    // same decisions at depths 1..D0-1
    const int* h = (const int*)F.src;
    D0 = __ldcg(h);
    iters = __ldcg(h + 1);
    tw = __ldcg(h + 2);
    first = __ldcg(h + 3) != 0;
    const int producer = __ldcg(h + 4);
    if (R == 0) act = __ldcg(h + 5);
    if (R == 0) inherited = __ldcg((const long long*)(F.src + 24));
    const uint4* s4 = (const uint4*)(F.src + kSnapHeader);
    uint4* d4 = (uint4*)F.slot;
#pragma unroll 4
    for (unsigned x = R; x < F.slot_bytes / 16u; x += S) d4[x] = __ldcg(s4 + x);  // (in flight together)
    // a path resumed from its own parking snapshot keeps its records
    if (out.st && producer != id) {  // the decision records of the shared prefix are the producer's
      const StepTrace* ps = F.st0 + (size_t)producer * dmx;
#pragma unroll 1
      for (int q = R; q < dmx; q += S) {
        StepTrace r{-2, -1, 0, 0, 0};
        if (q < D0 - 1) {
          const uint2 v = __ldcg((const uint2*)(ps + q));
          memcpy(&r, &v, sizeof(r));
        }
        out.st[q] = r;
      }
    }
    g.sync();
  } else {
    const int nrp = 32 * G.rw, nsp = 32 * G.cw;
#pragma unroll 1
    for (int k = R; k <= nsp; k += S) {  // (past ns: no VN; nsp: the dummy column)
      if (k < nsp) B.status[k] = k < ns ? -1 : 0;
      B.post[k] = k < ns ? G.llr[k] : dead_post();  // t = 0: mu_{i->j} = Lambda_i (Sec. II-A)
      if (k < ns) act += G.vdeg[k];
    }
#pragma unroll 1
    for (int j = R; j < nrp; j += S) {
      // active VNs of the check: its entries that are not the dummy column
      int d = 0;
      if (j < 32 * G.rwz) {
        const uint4* re = (const uint4*)G.rent + (int)G.roff[j >> 5] * 32 + (j & 31);
        const int nq = (int)(G.roff[(j >> 5) + 1] - G.roff[j >> 5]);
        const uint32_t dum = 4u * nsp;
#pragma unroll 1
        for (int q = 0; q < nq; ++q) {
          const uint4 e = re[32 * q];
          d += (int)(e.x < dum) + (int)(e.y < dum) + (int)(e.z < dum) + (int)(e.w < dum);
        }
      }
      B.deg[j] = (uint8_t)d;
    }
    if (R == 0) B.cns[32 * G.rwz] = CNState{0.0f, 0.0f, 0u, 0u};  // the dummy check: message +0
#pragma unroll 1
    for (int base = 0; base < nr; base += S) {  // the window syndrome by check label
      const int j = base + R;
      const unsigned m = __ballot_sync(FULL, j < nr && bit_of(G.sbits, G.cperm[j]));
      if ((R & 31) == 0 && base + R < nr) B.sp[(base + R) >> 5] = m;
    }
    if (out.st)
#pragma unroll 1
      for (int q = R; q < dmx; q += S) out.st[q] = StepTrace{-2, -1, 0, 0, 0};
    g.sync();
    if (P.peel_init) {
      const int np = peel(G, B, g, act);
      if (np < 0) {
        status = np == -1 ? BR_CONTRADICTION : BR_INTERNAL;
        goto done;
      }
    }
  }
#pragma unroll 1
  for (int D = D0; D <= dmax; ++D) {
    depth = D;
    if (!(F.src && D == D0)) {  // (a resumed run's snapshot holds its first step's BP)
    const int ips = (D == 1 && P.ips1 > 0) ? P.ips1 : P.ips;  // the first step may have its own length
#pragma unroll 1
    for (int it = 1; it <= ips; ++it) {
      // ---- check-node update, Eq. (1), and the previous iteration's H e = s ----
      bool unsat;
      if constexpr (Grp::kWarp) {
        unsat = check_pass_warp<LW>(P, G, B, R, first, tw);
        __syncwarp();
      } else {
        unsat = check_pass_cta<LW>(P, G, B, R, S, path_lanes_per_check(S, 32 * G.rwz), first, tw);
      }
      visits += act;
      if (!g.any(unsat) && it >= 2) {  // the previous iteration's decisions satisfy H e = s
        status = BR_CONVERGED;
        pm = path_metric(G, B, g);
        goto done;
      }
      // ---- variable-node update, Eq. (2)-(3); history of Sec. IV-A ----
      const bool hist = it > ips - 4;
      const bool hist0 = it == ips - 3;
      // variables in label order; a decimated column runs the loop too and stores nothing
      LwEdge lw{nullptr, G.cef};
      if (LW) lw.w = weight_row(G.wts, G.wT, G.wE, tw + 1);
      const int lane = R & 31;
      ColView<LwEdge> V{*G.cls, G.cent, G.coff, G.llr, B.status, (const char*)B.cns, lw, lane, S >> 5};
      const int n3 = V.K.n3;
      // (a check past 32 entries: every slice goes one at a time)
      if ((G.coff[0] & kWideSlice) != 0) V.K.n4 = V.K.n3 = V.K.n2 = V.K.n1;
      column_pass<LW, false>(V, R >> 5, [&](int s, float p) { B.post[32 * s + lane] = p; });
      // the history of Sec. IV-A, for the columns a decimation step looks at:
      // SELECT-VN's and Alg. 3's candidates have degree three or more
      if (hist)
#pragma unroll 1
        for (int s = R >> 5; s < n3; s += V.st) {
          const int k = 32 * s + lane;
          if (B.status[k] != -1) continue;
          const float p = B.post[k];
          if (P.rkq || P.dump) B.hq[4 * k + (it - (ips - 3))] = qhist(p);
          // both P_A tests of Alg. 3 (main branch: bit 1, other branches: bit 4),
          // so that the step's BP does not depend on the path
          const uint8_t f = (uint8_t)((p <= 0.0f) | ((p < P.pa_main) << 1) | ((p > P.pc) << 2) | ((p > P.pd) << 3) |
                                      ((p < P.pa_other) << 4));
          if (hist0) {
            B.acc[k] = p;
            B.hfl[k] = f;
          } else {
            B.acc[k] = __fadd_rn(B.acc[k], p);
            B.hfl[k] &= f;
          }
        }
      g.sync();
      ++iters;
      ++tw;
      first = false;
    }
    // the step's last iteration: its own convergence test, which also leaves
    // the unsatisfied-check words for Alg. 3 and the ranker
    if (!parity_pass(G, B, g)) {
      status = BR_CONVERGED;
      pm = path_metric(G, B, g);
      goto done;
    }
    // a snapshot here for paths queued later that share the decisions so far
    // (the first path to get here writes it)
    if (F.chain && F.chain[D - 1] >= 0) {
      const int n = F.chain[D - 1];
      int won = 0;
      if (R == 0) won = atomicCAS(&F.flags[n], 0, 1) == 0;
      if (g.any(won != 0)) {
        write_snapshot(F.pool + (size_t)n * F.stride, F, g, D, iters, tw, first, id, g.sum_i(act),
                       g.sum_ll(visits + inherited));
        if (R == 0) atomicExch(&F.flags[n], 2);
      }
    }
    }
    // preemption point: switch to a waiting path with more steps left (not
    // right where this run resumed)
    if (F.sched && D < dmax && !(F.src && D == D0)) {
      unsigned cw = 0;
      int c = longest_waiting(P, F, R, dmax - D + 2, cw);  // more than one step more than this path's
      if (c >= 0) {
        int won = 0;
        if (R == 0) won = atomicCAS(&F.sched[c], cw, (unsigned)PS_RUNNING) == cw;
        if (!g.any(won != 0)) c = -1;
      }
      if (c >= 0) {
        if (claimed) *claimed = cw;
        // park: this path resumes from its own snapshot after the BP of step D
        const long long own = g.sum_ll(visits);
        write_snapshot(F.pool + (size_t)(F.n_nodes + id) * F.stride, F, g, D, iters, tw, first, id, g.sum_i(act),
                       g.sum_ll(visits + inherited));
        if (R == 0) {
          atomicExch(&F.sched[id], (unsigned)PS_PARKED | ((unsigned)D << 8));
          if (out.exec) atomicAdd((unsigned long long*)out.exec, (unsigned long long)own);
        }
        g.sync();
        return c;
      }
    }
    if (D == dmax) break;  // no decimation after the last BP step
    {
      // ---- SELECT-VN (Alg. 1) with AGG-DEC (Alg. 3) ----
      const float PBd = (D == 1) ? P.pb_d1 : (main_rules(D) ? P.pb_main : P.pb_other);
      const uint8_t pa_bit = main_rules(D) ? 2 : 16;
      // bk, tk: (ranked column << 16) | label, so that ties go to the lowest
      // ranked column (the oracle's index order) whatever the label order
      float bL = CUDART_INF_F, tL = CUDART_INF_F;
      int bk = kNone, tk = kNone, nagg = 0;
      const int n3 = min(ns, 32 * G.cls->n3);  // (labels by descending degree)
#pragma unroll 1
      for (int k = R; k < n3; k += S) {
        if (B.status[k] != -1 || G.vdeg[k] <= 2) continue;
        const float L = B.acc[k];
        const uint8_t fl = B.hfl[k];
        if (!P.low_err) {
          int nus = 0;
          const uint32_t* ce = G.col_ents(k);
#pragma unroll 1
          for (int u = 0; u < G.vdeg[k]; ++u) nus += bit_of(B.unsat, (int)(ce[32 * u] >> 16));
          int bdec = -1;
          if ((fl & pa_bit) && L < PBd) bdec = 1;
          else if (((fl & 4) && D <= P.pc_max_depth) || ((fl & 8) && nus >= P.n_unsat_min)) bdec = 0;
          if (bdec >= 0) {
            act -= decimate_atomic(G, B, k, bdec);
            ++nagg;
            continue;
          }
        }
        if (P.rkq) continue;
        const int pk = ((int)G.vperm[k] << 16) | k;
        if (L < bL || (L == bL && pk < bk)) {
          bL = L;
          bk = pk;
        }
        if ((fl & 1) && (L < tL || (L == tL && pk < tk))) {
          tL = L;
          tk = pk;
        }
      }
      if (P.rkq) {
        g.sync();  // the aggressive decisions are visible
        ranker_select(P, G, B, g, bL, bk);
        if (bk != kNone) bL = B.acc[bk & 0xFFFF];  // f keeps the rule of Alg. 1: [L <= 0]
        nagg = g.sum_i(nagg);
        g.sync();
      } else {
        g.select_reduce(bL, bk, tL, tk, nagg);
      }
      int gsel, f;
      if (tk != kNone) {
        gsel = tk & 0xFFFF;
        f = 1;
      } else if (bk != kNone) {
        gsel = bk & 0xFFFF;
        f = bL <= 0.0f ? 1 : 0;
      } else {
        if (out.st && R == 0) out.st[D - 1] = StepTrace{-1, -1, 0, (int16_t)nagg, 0};
        status = BR_NOCAND;
        goto done;
      }
      if (P.dump && id == 0) {
        dump_candidates(P, G, B, g, out.shot, D, gsel);
        g.sync();
      }
      int v = f;
      if (split) {
        if (D == split) v = 1 - f;  // the one contrary decision of a side branch
      } else if (D <= P.k) {
        v = ((id >> (P.k - D)) & 1) ? 1 - f : f;  // b + (-1)^b f
      }
      if (R == 0) act -= decimate_one(G, B, gsel, v);
      g.sync();
      const int np = peel(G, B, g, act);
      if (out.st && R == 0)
        out.st[D - 1] = StepTrace{(int16_t)G.vperm[gsel], (int8_t)v, 0, (int16_t)nagg, (int16_t)(np < 0 ? -1 : np)};
      if (np < 0) {
        status = np == -1 ? BR_CONTRADICTION : BR_INTERNAL;
        goto done;
      }
      if (D == d_reinit) {  // mu_{i->j} = Lambda_i again: the next pass reads the priors
#pragma unroll 1
        for (int k = R; k < ns; k += S)
          if (B.status[k] == -1) B.post[k] = G.llr[k];
        tw = 0;
        first = true;
        g.sync();
      }
    }
  }
done:
  // the estimate by ranked column (bit vperm[k] for label k)
#pragma unroll 1
  for (int x = R; x < (ns + 31) >> 5; x += S) out.ebits[x] = 0u;
  g.sync();
#pragma unroll 1
  for (int k = R; k < ns; k += S) {
    const int s8 = B.status[k];
    const int kr = G.vperm[k];
    if (s8 == 1 || (s8 == -1 && B.post[k] <= 0.0f)) atomicOr(&out.ebits[kr >> 5], 1u << (kr & 31));
    if (out.fstat) out.fstat[kr] = (int8_t)s8;
  }
  // The fallback key of a path that did not converge (the window's output
  // when no path converges is the least key, ties to the lowest id): rule 1
  // counts the unsatisfied checks of its estimate, rule 2 those among the
  // committed rows first (key = committed * (nr + 1) + all).  It takes the
  // place of the path metric, which only a converged path has.
  double fkey = CUDART_INF;
  if (status != BR_CONVERGED && P.fallback) {
    parity_pass(G, B, g);
    g.sync();
    long long nu = 0;
#pragma unroll 1
    for (int j = R; j < G.nr; j += S)
      if (bit_of(B.unsat, j)) nu += (P.fallback == 2 && G.cperm[j] < G.ncr) ? (long long)G.nr + 2 : 1;
    fkey = (double)g.sum_ll(nu);
  }
  // message reuse: what this path would leave the next window if it is the
  // window's output path (converged, path 0, or any path under a fallback
  // rule): the final posterior of each active column, +-clip for a decimated one
  if (out.keep && (status == BR_CONVERGED || id == 0 || P.fallback))
#pragma unroll 1
    for (int k = R; k < ns; k += S) {
      const int s8 = B.status[k];
      out.keep[k] = s8 == -1 ? B.post[k] : (s8 ? -P.clip : P.clip);
    }
  visits = g.sum_ll(visits);
  if (R == 0) {
    *out.status = status;
    *out.pm = status == BR_CONVERGED ? pm : fkey;
    if (out.btr) *out.btr = BranchTrace{status, depth, iters, 0, status == BR_CONVERGED ? pm : CUDART_INF};
    atomicAdd((unsigned long long*)out.visits, (unsigned long long)(visits + inherited));
    if (out.exec) atomicAdd((unsigned long long*)out.exec, (unsigned long long)visits);
    if (F.sched) atomicExch(&F.sched[id], (unsigned)PS_DONE);
  }
  g.sync();
  return -1;
}

// Trace layout of one shot: int32 head[4]; BranchTrace[nb]; StepTrace[nb][dmx];
// int8 final_status[nb][ns_max]; uint16 short columns[ns_max].
__host__ __device__ inline size_t trace_off_br() { return 16; }
__host__ __device__ inline size_t trace_off_st(int nb) { return 16 + sizeof(BranchTrace) * nb; }
__host__ __device__ inline size_t trace_off_fs(int nb, int dmx) {
  return trace_off_st(nb) + sizeof(StepTrace) * (size_t)nb * dmx;
}
__host__ __device__ inline size_t trace_off_sel(int nb, int dmx, int nsm) {
  return (trace_off_fs(nb, dmx) + (size_t)nb * nsm + 1) & ~(size_t)1;
}
__host__ __device__ inline size_t trace_bytes(int nb, int dmx, int nsm) {
  return (trace_off_sel(nb, dmx, nsm) + 2 * (size_t)nsm + 15) & ~(size_t)15;
}

struct DecodeArgs {
  KParams P;
  WinDev W;
  Layout L;
  const uint32_t* det;
  int det_words;
  long long n_shots;
  uint32_t* corr;
  int corr_words;
  int32_t* status_out;
  char* trace;
  size_t tr_bytes;
  int dmx, ns_max;
  int* work;            // shot mode: work counter
  long long* counters;  // [0] pre-BP edge-iterations, [1] GDG edge visits, [2] pre-BP converged,
                        // [3] GDG windows, [4] bulk staging waits that ran out
  char* path_res;       // path mode: results [shot][path]
  int* arrive;          // path mode: per-shot arrival counters (0 between launches)
  int sw_max;
  // windows too large for shared memory: the union region (pre-BP scratch and
  // path slots) of CTA b lives at uglob + b * ubytes in global memory
  // (L2-resident at these sizes) instead of after the persistent part
  char* uglob;
  size_t ubytes;
  // path mode: CTAs per shot (the paths, then idle CTAs up to a whole number
  // of clusters, which only help with the pre-BP)
  int cps;
  // executed GDG edge visits (nullable; counters[1] counts every path's
  // whole run, resumed prefixes included)
  long long* exec;
  ForkDev F;  // shot mode: snapshots of shared path prefixes
  // message reuse between windows (nullptr: off): keep[shot * keep_ld + c]
  // what the output path of this window ends with for window column c (NaN:
  // nothing), read by the next window through prev[c] (this window's column
  // -> the previous window's, -1: none; nullptr for the first window);
  // kpath[(slot * nb + path) * ns_max + label] each candidate path's values
  // (slot: the CTA in shot mode, the shot in path mode)
  float* keep;
  int keep_ld;
  const int16_t* prev;
  float* kpath;
};

// UG (a template parameter, so that shared-memory kernels keep shared-memory
// instructions for every union access): 1: the region lives in global memory;
// 2: the shortened graph's entries as well, at its start (kGraphGlobal); 3: only
// the entries' edge ids (kIdsGlobal).
template <int UG>
__device__ __forceinline__ char* union_base(const DecodeArgs& A, char* sm, const SlotPlan& S) {
  if (UG == 1 || UG == 2) return A.uglob + (size_t)blockIdx.x * A.ubytes + (UG == 2 ? S.U : 0u);
  return sm + S.U;
}
// What the entries' offsets are relative to: SlotPlan::rent and cent, and ref and cef.
template <int UG>
__device__ __forceinline__ char* graph_base(const DecodeArgs& A, char* sm) {
  return UG == 2 ? A.uglob + (size_t)blockIdx.x * A.ubytes : sm;
}
template <int UG>
__device__ __forceinline__ char* ids_base(const DecodeArgs& A, char* sm) {
  return UG >= 2 ? A.uglob + (size_t)blockIdx.x * A.ubytes : sm;
}
// The pre-BP scratch: the union region in global memory, else the bytes of the
// shortened graph and the path slots, which do not exist yet.
template <int UG>
__device__ __forceinline__ char* prebp_base(const DecodeArgs& A, char* sm) {
  if (UG == 1 || UG == 2) return A.uglob + (size_t)blockIdx.x * A.ubytes;
  return sm + A.L.V;
}

// One window step of several decoders in one launch (kernel parameter).
struct BatchArgs {
  int n_seg;
  unsigned q_off;  // shared-memory offset of the launch's own work slot
  int* work;
  long long seg_end[kMaxBatch];  // cumulative shot counts
  DecodeArgs seg[kMaxBatch];
};

// Commit (Eq. (10)) + residue test (Eq. (11)) of one decoder's window.
struct CommitArgs {
  int n_commit;
  const int *cptr, *cdet;
  const uint32_t* cobs;
  int corr_words;
  const uint32_t* corr;
  long long n;
  uint32_t* det;
  int det_words;
  uint32_t *obs_pred, *resid;
  int b0, b1;
};
struct CommitBatch {
  int n_seg;
  long long seg_end[kMaxBatch];
  CommitArgs seg[kMaxBatch];
};

// ---- ascending sort of n = 2^m 64-bit keys in shared memory (all threads) ----
// A bitonic network.  Every stage of stride < 256 runs in registers: a warp
// holds a segment of 256 keys, lane L the keys L + 32 r (r < 8), so strides
// 32..128 pair two registers of a lane and strides 1..16 two lanes (shuffles).
// Strides >= 256 pass through shared memory, up to three stages per pass.
// Keys that differ sort the same under any correct network.
__device__ __forceinline__ unsigned long long shfl_u64(unsigned long long v, int m) {
  const unsigned lo = __shfl_xor_sync(FULL, (unsigned)v, m), hi = __shfl_xor_sync(FULL, (unsigned)(v >> 32), m);
  return ((unsigned long long)hi << 32) | lo;
}

// stride 32 RJ: registers r and r | RJ of a lane
template <int RJ>
__device__ __forceinline__ void reg_stage(unsigned long long (&v)[8], int base, int lane, int kk) {
#pragma unroll
  for (int r = 0; r < 8; ++r)
    if (!(r & RJ)) {
      const bool up = ((base + 32 * r + lane) & kk) == 0;
      const unsigned long long a = v[r], b = v[r | RJ];
      const bool sw = (a > b) == up;
      v[r] = sw ? b : a;
      v[r | RJ] = sw ? a : b;
    }
}

// the stages of block size kk with strides j0 >= j >= 1 (j0 < 256) of one
// register segment whose first key has global index base
__device__ __forceinline__ void seg_stages(unsigned long long (&v)[8], int base, int lane, int kk, int j0) {
#pragma unroll 1
  for (int j = j0; j > 0; j >>= 1) {
    if (j == 128) {
      reg_stage<4>(v, base, lane, kk);
    } else if (j == 64) {
      reg_stage<2>(v, base, lane, kk);
    } else if (j == 32) {
      reg_stage<1>(v, base, lane, kk);
    } else {
      const bool low = (lane & j) == 0;
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const unsigned long long o = shfl_u64(v[r], j);
        const bool up = ((base + 32 * r + lane) & kk) == 0;
        const bool keep_min = low == up;
        v[r] = keep_min ? (o < v[r] ? o : v[r]) : (o > v[r] ? o : v[r]);
      }
    }
  }
}

// M stages of strides j, j/2, ..., j/2^(M-1) (all >= 256) through shared memory
template <int M>
__device__ __forceinline__ void smem_stages(unsigned long long* s, int n, int kk, int j) {
  const int b1 = __ffs(j) - 1;
#pragma unroll 1
  for (int g = threadIdx.x; g < (n >> M); g += blockDim.x) {
    int base = g;
#pragma unroll
    for (int q = M - 1; q >= 0; --q) {  // zero bits at b1-M+1 .. b1, lowest first
      const int b = b1 - q;
      base = ((base >> b) << (b + 1)) | (base & ((1 << b) - 1));
    }
    const bool up = (base & kk) == 0;
    unsigned long long v[1 << M];
#pragma unroll
    for (int t = 0; t < (1 << M); ++t) {
      int off = 0;
#pragma unroll
      for (int l = 0; l < M; ++l) off += ((t >> l) & 1) * (j >> (M - 1 - l));
      v[t] = s[base + off];
    }
#pragma unroll
    for (int l = M - 1; l >= 0; --l)  // bit l of t <-> stride j >> (M - 1 - l), largest first
#pragma unroll
      for (int t = 0; t < (1 << M); ++t)
        if (!((t >> l) & 1)) {
          const unsigned long long a = v[t], b = v[t | (1 << l)];
          const bool sw = (a > b) == up;
          v[t] = sw ? b : a;
          v[t | (1 << l)] = sw ? a : b;
        }
#pragma unroll
    for (int t = 0; t < (1 << M); ++t) {
      int off = 0;
#pragma unroll
      for (int l = 0; l < M; ++l) off += ((t >> l) & 1) * (j >> (M - 1 - l));
      s[base + off] = v[t];
    }
  }
}

// Call with every thread; s holds n keys (n a power of two); returns after a barrier.
__device__ void block_sort_u64(unsigned long long* s, int n) {
  const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = NT >> 5;
  if (n < 256) {  // tiny windows: the plain network
#pragma unroll 1
    for (int kk = 2; kk <= n; kk <<= 1)
#pragma unroll 1
      for (int jj = kk >> 1; jj > 0; jj >>= 1) {
#pragma unroll 1
        for (int i = tid; i < n; i += NT) {
          const int ixj = i ^ jj;
          if (ixj > i) {
            const unsigned long long a = s[i], b = s[ixj];
            if ((a > b) == ((i & kk) == 0)) {
              s[i] = b;
              s[ixj] = a;
            }
          }
        }
        __syncthreads();
      }
    return;
  }
  // every block size up to 256 inside the segments
#pragma unroll 1
  for (int sg = warp; sg < (n >> 8); sg += nw) {
    const int base = sg << 8;
    unsigned long long v[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = s[base + 32 * r + lane];
#pragma unroll 1
    for (int kk = 2; kk <= 256; kk <<= 1) seg_stages(v, base, lane, kk, kk >> 1);
#pragma unroll
    for (int r = 0; r < 8; ++r) s[base + 32 * r + lane] = v[r];
  }
  __syncthreads();
#pragma unroll 1
  for (int kk = 512; kk <= n; kk <<= 1) {
    int j = kk >> 1;
#pragma unroll 1
    for (; j >= 256 * 4; j >>= 3) {  // three stages, all of stride >= 256
      smem_stages<3>(s, n, kk, j);
      __syncthreads();
    }
    if (j >= 512) {
      smem_stages<2>(s, n, kk, j);
      __syncthreads();
    } else if (j == 256) {
      smem_stages<1>(s, n, kk, j);
      __syncthreads();
    }
#pragma unroll 1
    for (int sg = warp; sg < (n >> 8); sg += nw) {
      const int base = sg << 8;
      unsigned long long v[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) v[r] = s[base + 32 * r + lane];
      seg_stages(v, base, lane, kk, 128);
#pragma unroll
      for (int r = 0; r < 8; ++r) s[base + 32 * r + lane] = v[r];
    }
    __syncthreads();
  }
}

// ---- thread-block clusters: distributed shared memory ----
__device__ __forceinline__ unsigned cl_size() {
  unsigned n;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(n));
  return n;
}
__device__ __forceinline__ unsigned cl_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// every thread of every CTA of the cluster; orders the shared-memory writes
// before it with the reads (local or remote) after it
__device__ __forceinline__ void cl_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the address of `p` (a shared-memory location of this CTA) in CTA `rank`
__device__ __forceinline__ unsigned cl_map(const void* p, unsigned rank) {
  unsigned a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void cl_st_f32(unsigned a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void cl_st_u32(unsigned a, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void cl_st_cns(unsigned a, const CNState& c) {
  asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(__float_as_uint(c.m1)),
               "r"(__float_as_uint(c.m2)), "r"(c.sg), "r"(c.am)
               : "memory");
}

// The pre-BP's arrays and graph, all by label.
struct PreBp {
  float *post, *key;
  CNState* cns;
  const uint32_t* sp;  // the window syndrome
  const uint16_t* rent;
  const uint32_t* cent;
  const uint16_t *roff, *coff;
  const float* llr;
};

// The pre-BP's variable pass (Eq. (2)) over the column slices first, first + st, ...
template <bool LW, class Put>
__device__ __forceinline__ void prebp_columns(const WinDev& W, const PreBp& X, int t, int first, int st, int lane,
                                              Put put) {
  LwOrdered lw{nullptr};
  if (LW) lw.w = weight_row(W.w_col, W.wT, 32 * W.col_cells, t);
  const ColView<LwOrdered> V{W.cls, X.cent, X.coff, X.llr, nullptr, (const char*)X.cns, lw, lane, st};
  column_pass<LW, true>(V, first, put);
}

__device__ __forceinline__ float prebp_key(const KParams& P, const PreBp& X, int l, int t, int tk0, float p) {
  if (t != tk0) return __fadd_rn(X.key[l], p);
  if (P.n_pre >= 4) return p;
  const float li = X.llr[l];
  float s = li;
#pragma unroll 1
  for (int r = 1; r < 4 - P.n_pre; ++r) s = __fadd_rn(s, li);
  return __fadd_rn(s, p);
}

// a2 split over the CTAs of a cluster (path mode, one cluster per shot): CTA
// r owns the r-th slice of the checks and of the variables, runs the check
// pass of Eq. (1) for its checks and the variable pass of Eq. (2)-(3) for its
// variables.  A remote load costs a round trip of ~1200 cycles (a cluster
// barrier ~470), so values only travel as stores: each CTA pushes the records
// of its checks, its posteriors (and ranking keys) and its "unsatisfied" flag
// into every CTA's shared memory before the barrier that ends the pass, and
// both passes read locally.  Two cluster barriers per iteration separate the
// passes, so every value read was written in the pass before, and after the
// last one no CTA touches another's shared memory.
// The arithmetic of every message and posterior is that of the single-CTA
// loop; at the end every CTA holds the whole posterior and key.  Returns t as
// the loop leaves it; conv and t_conv as in the caller.
template <bool LW>
__device__ int prebp_cluster(const DecodeArgs& A, const WinDev& W, const PreBp& X, char* sm, bool& conv, int& t_conv) {
  const KParams& P = A.P;
  const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31;
  const int nr = W.n_rows, nc = W.n_cols;
  const unsigned C = cl_size(), r = cl_rank();
  // flags[8 * parity + c]: CTA c found an unsatisfied check (in the reduction
  // scratch of the path phase, idle until the pre-BP ends)
  int* flags = (int*)(sm + A.L.red);
  const int sc = (nr + (int)C - 1) / (int)C, sv = (nc + (int)C - 1) / (int)C;
  const int jb = min(nr, (int)r * sc), je = min(nr, jb + sc);
  const int ib = min(nc, (int)r * sv), ie = min(nc, ib + sv);
  int tpc = 1;  // lanes per check: the most (<= 16) that take the slice in one round
  while (tpc < 16 && 2 * tpc * max(1, je - jb) <= NT) tpc <<= 1;
  const int sub = tid & (tpc - 1), per = NT / tpc;
  const int tk0 = P.n_pre - 3 > 1 ? P.n_pre - 3 : 1;
  const bool rwide = X.roff[1] - X.roff[0] > 8;  // the first slice is the widest
  cl_sync();  // every CTA of the cluster runs and has set up its arrays
  int t;
  for (t = 1; t <= P.n_pre; ++t) {
    LwOrdered lw{nullptr};
    if (LW && t > 1) lw.w = weight_row(W.w_row, W.wT, 128 * W.row_quads, t - 1);
    uint32_t unsat = 0u;
    for (int b = jb; b < je; b += per) {
      const int j0 = b + tid / tpc;
      const bool real = j0 < je;
      const int j = real ? j0 : je - 1, s = j >> 5;
      const int r0 = X.roff[s], nq = real ? (int)X.roff[s + 1] - r0 : 0;
      uint32_t u = 0u;
      const CNState rec = check_group<LW>((const uint2*)X.rent + r0 * 32 + (j & 31), nq, (const char*)X.post, X.cns[j],
                                          (X.sp[s] >> (j & 31)) & 1u, P.alpha, P.clip, t == 1, lw,
                                          (r0 * 32 + (j & 31)) * 4, sub, tpc, rwide, u);
      if (real) {
        for (int c = sub; c < (int)C; c += tpc) cl_st_cns(cl_map(&X.cns[j], (unsigned)c), rec);
        unsat |= u;
      }
    }
    const int lu = __syncthreads_or(unsat != 0u);
    if (tid < (int)C) cl_st_u32(cl_map(&flags[8 * (t & 1) + (int)r], (unsigned)tid), (uint32_t)lu);
    cl_sync();  // check records and flags of pass t, in every CTA
    const bool any = __any_sync(FULL, lane < (int)C && flags[8 * (t & 1) + lane] != 0);
    if (!any && t >= 2) {  // iteration t-1 satisfies H e = s in every slice
      conv = true;
      t_conv = t - 1;
      break;
    }
    LwOrdered lc{nullptr};
    if (LW) lc.w = weight_row(W.w_col, W.wT, 32 * W.col_cells, t);
    for (int i = ib + tid; i < ie; i += NT) {
      const int q = i >> 5, c0 = X.coff[q] & (kWideSlice - 1), n = (int)(X.coff[q + 1] & (kWideSlice - 1)) - c0;
      const int ei = c0 * 32 + (i & 31);
      float p = X.llr[i];
#pragma unroll 3
      for (int u = 0; u < n; ++u) {
        const uint32_t e = X.cent[ei + 32 * u];
        p = __fadd_rn(p, c2v<LW>(*(const CNState*)((const char*)X.cns + (e >> 12)), e, true,
                                 LW ? lc.one(ei + 32 * u) : 0.0f));
      }
      for (unsigned c = 0; c < C; ++c)  // every CTA reads the whole posterior in its check pass
        cl_st_f32(cl_map(&X.post[i], c), p);
      if (t >= tk0) {
        const float kv = prebp_key(P, X, i, t, tk0, p);
        for (unsigned c = 0; c < C; ++c) cl_st_f32(cl_map(&X.key[i], c), kv);
      }
    }
    cl_sync();  // posteriors (and keys) of pass t, in every CTA
  }
  return t;
}

// a1 + a2 (+ a3 when not converged): the shared prefix of both launch shapes.
// Returns true when the pre-BP converged (cbits then hold its decision).
template <bool LW, bool WIDE, int UG>
__device__ bool window_prefix(const DecodeArgs& A, const WinDev& W, char* sm, long long shot, int* t_run_out,
                              Stager& stg) {
  const KParams& P = A.P;
  const Layout& L = A.L;
  const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = NT >> 5;
  const int nr = W.n_rows, nc = W.n_cols, rw = L.rw, ncp = 32 * L.cw, nrp = 32 * rw;
  uint32_t* sbits = (uint32_t*)(sm + L.sbits);
  uint32_t* cbits = (uint32_t*)(sm + L.cbits);
  char* U = prebp_base<UG>(A, sm);
  float* post = (float*)(U + L.p_post);
  float* key = (float*)(U + L.p_key);
  CNState* cns = (CNState*)(U + L.p_cns);
  uint32_t* parb = (uint32_t*)(U + L.p_par);
  uint32_t* spre = parb + rw;  // the window syndrome by check label

  // ---- a1: window syndrome ----
  const uint32_t* dp = A.det + (size_t)shot * A.det_words;
#pragma unroll 1
  for (int x = tid; x < rw; x += NT) {
    const int b0 = W.row0 + 32 * x;
    const uint32_t lo = dp[b0 >> 5];
    const uint32_t hi = ((b0 >> 5) + 1 < A.det_words) ? dp[(b0 >> 5) + 1] : 0u;
    const int sh = b0 & 31;
    uint32_t v = sh ? ((lo >> sh) | (hi << (32 - sh))) : lo;
    const int rem = nr - 32 * x;
    if (rem < 32) v &= (1u << rem) - 1u;
    sbits[x] = v;
  }
#pragma unroll 1
  for (int x = tid; x < L.cw; x += NT) cbits[x] = 0;
  __syncthreads();

  // the window graph in shared memory for the pre-BP loop when there is room
  PreBp X{post, key, cns, spre, W.s_rent, W.s_cent, W.s_roff, W.s_coff, W.s_llr};
  if (L.pre_stage) {  // (an array that is not staged has no bytes)
    const unsigned sg = L.pre_stage;
    const StagePiece pc[5] = {{U + L.q_rent, W.s_rent, sg & kStageRent ? 256u * W.row_quads : 0u},
                              {U + L.q_cent, W.s_cent, sg & kStageCent ? 128u * W.col_cells : 0u},
                              {U + L.q_roff, W.s_roff, sg & kStageOff ? al16(2u * (rw + 1)) : 0u},
                              {U + L.q_coff, W.s_coff, sg & kStageOff ? al16(2u * (L.cw + 1)) : 0u},
                              {U + L.q_sllr, W.s_llr, sg & kStageLlr ? 4u * ncp : 0u}};
    stage_pieces(stg, pc);
    if (sg & kStageRent) X.rent = (const uint16_t*)(U + L.q_rent);
    if (sg & kStageCent) X.cent = (const uint32_t*)(U + L.q_cent);
    if (sg & kStageLlr) X.llr = (const float*)(U + L.q_sllr);
    if (sg & kStageOff) {
      X.roff = (const uint16_t*)(U + L.q_roff);
      X.coff = (const uint16_t*)(U + L.q_coff);
    }
  }
#pragma unroll 1
  for (int s = warp; s < rw; s += nw) {
    const int j = 32 * s + lane;
    const unsigned m = __ballot_sync(FULL, j < nr && bit_of(sbits, W.s_row[j]));
    if (lane == 0) spre[s] = m;
  }
  if (tid == 0) {
    post[ncp] = dead_post();                    // the dummy column
    cns[nrp] = CNState{0.0f, 0.0f, 0u, 0u};     // the dummy check: message +0
  }

  // ---- a2: pre-BP on the full window ----
  bool conv = false;
  int t = 0;
  const int tk0 = P.n_pre - 3 > 1 ? P.n_pre - 3 : 1;
  if (P.n_pre == 0) {
#pragma unroll 1
    for (int l = tid; l < nc; l += NT) {
      const float li = X.llr[l];
      post[l] = li;
      key[l] = __fadd_rn(__fadd_rn(__fadd_rn(li, li), li), li);
    }
    __syncthreads();
  } else {
    // the first VN->CN messages of the pre-BP: the prior, or (message reuse)
    // what the previous window's output path kept for the same DEM column
    const float* kept = (A.keep && A.prev) ? A.keep + (size_t)shot * A.keep_ld : nullptr;
#pragma unroll 1
    for (int l = tid; l < nc; l += NT) {
      float v = X.llr[l];
      if (kept) {
        const int pc = A.prev[W.s_col[l]];
        if (pc >= 0) {
          const float x = kept[pc];
          if (x == x) v = x;
        }
      }
      post[l] = v;
    }
    __syncthreads();
  }
  int t_conv = 0;
  if (WIDE && UG != 1 && UG != 2 && P.n_pre > 0 && cl_size() > 1 && nr >= 2 * (int)cl_size() && nc >= 2 * (int)cl_size()) {
    t = prebp_cluster<LW>(A, W, X, sm, conv, t_conv);
  } else {
#pragma unroll 1
    for (t = 1; t <= P.n_pre; ++t) {
      // check nodes; each check also takes the parity of the hard decisions it
      // reads, so for t >= 2 the pass is the convergence test of iteration t-1
      LwOrdered lw{nullptr};
      if (LW && t > 1) lw.w = weight_row(W.w_row, W.wT, 128 * W.row_quads, t - 1);
      uint32_t unsat = 0u;
#pragma unroll 1
      for (int s = warp; s < rw; s += nw) {
        const int r0 = X.roff[s], nq = (int)X.roff[s + 1] - r0;
        unsat |= check_lane<LW>((const uint2*)X.rent + r0 * 32 + lane, nq, (const char*)post, cns + 32 * s + lane,
                                (spre[s] >> lane) & 1u, P.alpha, P.clip, lw, (r0 * 32 + lane) * 4, t == 1);
      }
      if (!__syncthreads_or(unsat != 0u) && t >= 2) {  // iteration t-1 satisfies H e = s
        conv = true;
        t_conv = t - 1;
        break;
      }
      auto put = [&](int s, float p) {
        const int l = 32 * s + lane;
        post[l] = p;
        if (t >= tk0) key[l] = prebp_key(P, X, l, t, tk0, p);
      };
      prebp_columns<LW>(W, X, t, warp, nw, lane, put);
      __syncthreads();
    }
  }
  if (!conv) {  // the convergence test of the last iteration (or of the priors)
    bool unsat = false;
#pragma unroll 1
    for (int s = warp; s < rw; s += nw) {
      const uint32_t hp = (((spre[s] >> lane) & 1u) << 31) ^
                          check_parity((const uint2*)X.rent + (int)X.roff[s] * 32 + lane,
                                       (int)X.roff[s + 1] - (int)X.roff[s], (const char*)post);
      unsat |= (hp >> 31) != 0u;
    }
    if (!__syncthreads_or(unsat)) {
      conv = true;
      t_conv = P.n_pre;
    }
  }
  *t_run_out = conv ? t_conv : P.n_pre;
  if (conv) {
#pragma unroll 1
    for (int l = tid; l < nc; l += NT)
      if (post[l] <= 0.0f) {
        const int c = W.s_col[l];
        atomicOr(&cbits[c >> 5], 1u << (c & 31));
      }
    __syncthreads();
    return true;
  }

  // ---- a3: rank by the four-iteration sum, keep the first n_short ----
  const int n_short = W.n_short, nsp = 32 * L.sw;
  unsigned long long* sortb = (unsigned long long*)(U + L.p_sort);
  auto sort_key = [&](int l, uint32_t k) {  // ties by window column
    return ((unsigned long long)k << 32) | ((unsigned)W.s_col[l] << 16) | (unsigned)l;
  };
  if (L.sortn >= nc) {
#pragma unroll 1
    for (int l = tid; l < L.sortn; l += NT) sortb[l] = l < nc ? sort_key(l, ordkey(key[l])) : ~0ull;
  } else {
    // select before sorting: bisection for the n_short-th smallest key, then
    // (equal keys) for the column up to which its equals are taken.  Sorting all
    // 4096 places was a tenth of a window of the paper preset (3000 shots of
    // [[144,12,12]] 44.5 ms; 42.4 with the 512 selected ones).
    uint32_t* uk = (uint32_t*)key;
    // (the sort buffer follows the keys, over the dead check records; the
    // posteriors before them are dead too)
    const CtaGrp cta{tid, NT, (char*)post};
    auto count = [&](auto&& in) {
      int n = 0;
#pragma unroll 4
      for (int l = tid; l < nc; l += NT) n += in(l) ? 1 : 0;
      return cta.sum_i(n);
    };
#pragma unroll 1
    for (int l = tid; l < nc; l += NT) uk[l] = ordkey(key[l]);
    uint32_t lo = 0u, hi = 0xFFFFFFFFu;
    int most = nc;  // keys <= hi
#pragma unroll 1
    while (lo < hi) {
      const uint32_t mid = lo + (hi - lo) / 2;
      const int n = count([&](int l) { return uk[l] <= mid; });
      if (n >= n_short) {
        hi = mid;
        most = n;
      } else {
        lo = mid + 1;
      }
    }
    int c_lo = 0, c_hi = most == n_short ? 0x7fff : nc - 1;
    if (most > n_short) {
#pragma unroll 1
      while (c_lo < c_hi) {
        const int mid = (c_lo + c_hi) / 2;
        const int n = count([&](int l) { return uk[l] < hi || (uk[l] == hi && (int)W.s_col[l] <= mid); });
        if (n >= n_short) c_hi = mid;
        else c_lo = mid + 1;
      }
    }
    int* next = (int*)(sm + L.misc) + 5;
    if (tid == 0) *next = 0;
#pragma unroll 1
    for (int l = n_short + tid; l < L.sortn; l += NT) sortb[l] = ~0ull;
    __syncthreads();
#pragma unroll 1
    for (int l = tid; l < nc; l += NT)
      if (uk[l] < hi || (uk[l] == hi && (int)W.s_col[l] <= c_hi)) sortb[atomicAdd(next, 1)] = sort_key(l, uk[l]);
  }
  __syncthreads();
  block_sort_u64(sortb, L.sortn);
  // (from here on the pre-BP's arrays are dead: the shortened graph takes their place)
  uint16_t* sel = (uint16_t*)(sm + L.sel);
  uint16_t* roff = (uint16_t*)(sm + L.s_roff);
  uint16_t* coff = (uint16_t*)(sm + L.s_coff);
  float* sllr = (float*)(sm + L.s_llr);
  uint8_t* svd = (uint8_t*)(sm + L.s_vdeg);
  uint16_t* cperm = (uint16_t*)(sm + L.s_cperm);
  uint16_t* vperm = (uint16_t*)(sm + L.s_vperm);
#pragma unroll 1
  for (int k = tid; k < n_short; k += NT) sel[k] = (uint16_t)(sortb[k] >> 16);
  __syncthreads();
  // sort keys of the labels, (degree, lowest index first), by rank and by row;
  // zero in the padding
  unsigned* ckey = (unsigned*)(U + L.p_scr);
  unsigned* rkey = ckey + nsp;
  int* rc = (int*)(rkey + nrp);  // degree by window row, later entries placed by label
#pragma unroll 1
  for (int j = tid; j < nrp; j += NT) rc[j] = 0;
  __syncthreads();
  // ---- shortened matrix in shared memory, numbered in processing order ----
  // Columns and checks get labels by descending degree (ties by rank / row),
  // so the lanes of a round loop alike; vperm and cperm map a label back to
  // the ranked column and the window row, which decide every tie.  A column's
  // checks stay in ascending window row (the order of the sum of Eq. (2)).
#pragma unroll 1
  for (int k = tid; k < nsp; k += NT) {
    unsigned d = 0;
    if (k < n_short) {
      const int c = sel[k], e0 = W.col_ptr[c];
      d = W.col_ptr[c + 1] - e0;
#pragma unroll 1
      for (unsigned u = 0; u < d; ++u) atomicAdd(&rc[W.col_rows[e0 + u]], 1);  // rows of the shortened matrix
    }
    ckey[k] = k < n_short ? (d << 16) | (0xFFFFu - (unsigned)k) : 0u;
  }
  __syncthreads();
#pragma unroll 1
  for (int j = tid; j < nrp; j += NT) rkey[j] = j < nr ? ((unsigned)rc[j] << 16) | (0xFFFFu - (unsigned)j) : 0u;
  // a label is the number of larger keys; no sort needed at these sizes
  auto above = [](const unsigned* key, int n, unsigned k) {
    int r = 0;
#pragma unroll 2
    for (int i = 0; i < n; i += 4) {
      const uint4 x = *(const uint4*)(key + i);
      r += (x.x > k) + (x.y > k) + (x.z > k) + (x.w > k);
    }
    return r;
  };
#pragma unroll 1
  for (int k = tid; k < n_short; k += NT) {
    const unsigned key_k = ckey[k];
    const int r = above(ckey, nsp, key_k);
    vperm[r] = (uint16_t)k;
    svd[r] = (uint8_t)(key_k >> 16);
  }
  __syncthreads();
#pragma unroll 1
  for (int j = tid; j < nr; j += NT) cperm[above(rkey, nrp, rkey[j])] = (uint16_t)j;
  __syncthreads();
  int* cinv = (int*)rkey;  // window row -> label, once the keys have been read
  // slice starts (a slice is as wide as its first node), one warp each
  if (warp == 0) {
    int run = 0;
#pragma unroll 1
    for (int b = 0; b < rw; b += 32) {
      const int s = b + lane;
      int v = s < rw ? (rc[cperm[32 * s]] + 3) >> 2 : 0;
      v = warp_incl_scan(v, lane);
      if (s < rw) roff[s + 1] = (uint16_t)(run + v);
      run += __shfl_sync(FULL, v, 31);
    }
    if (lane == 0) roff[0] = 0;
  }
  if (warp == (nw > 1 ? 1 : 0)) {
    // (a check past 32 entries is rare in a shortened graph: one flag for all)
    const uint16_t flag = rc[cperm[0]] > 32 ? kWideSlice : (uint16_t)0;
    int run = 0;
#pragma unroll 1
    for (int b = 0; b < L.sw; b += 32) {
      const int s = b + lane;
      int v = s < L.sw ? (int)svd[32 * s] : 0;
      v = warp_incl_scan(v, lane);
      if (s < L.sw) coff[s + 1] = (uint16_t)((run + v) | flag);
      run += __shfl_sync(FULL, v, 31);
    }
    if (lane == 0) coff[0] = flag;
    if (lane < 4) {  // slices at least 4 - lane wide
      int n = 0;
#pragma unroll 1
      while (n < L.sw && svd[32 * n] >= 4 - lane) ++n;
      ((int*)(sm + L.s_cls))[lane] = n;
    }
  }
  __syncthreads();
  // the shot's own layout
  SlotPlan S;
  {
    int rwz = 0;
#pragma unroll 1
    while (rwz < rw && roff[rwz + 1] > roff[rwz]) ++rwz;
    S = slot_plan(L, roff[rw], coff[L.sw] & (kWideSlice - 1), rwz, ((const int*)(sm + L.s_cls))[1],
                  UG == 1 || UG == 2 ? (unsigned)A.ubytes : L.total, UG == 1 || UG == 2, nw);
    if (tid == 0) *(SlotPlan*)(sm + L.plan) = S;
  }
  char* ents = graph_base<UG>(A, sm);
  uint32_t* rent = (uint32_t*)(ents + S.rent);
  uint32_t* cent = (uint32_t*)(ents + S.cent);
  uint16_t* sref = (uint16_t*)(ids_base<UG>(A, sm) + S.ref);
  uint16_t* scef = (uint16_t*)(ids_base<UG>(A, sm) + S.cef);
  // every place a dummy, then the edges
  {
    const int nq = roff[rw], ncell = coff[L.sw] & (kWideSlice - 1);
#pragma unroll 1
    for (int x = tid; x < 128 * nq; x += NT) rent[x] = 4u * (unsigned)nsp;
#pragma unroll 1
    for (int x = tid; x < 32 * ncell; x += NT) cent[x] = (unsigned)(32 * S.rwz) << 16;
    if (LW) {
#pragma unroll 1
      for (int x = tid; x < 128 * nq; x += NT) sref[x] = 0;
#pragma unroll 1
      for (int x = tid; x < 32 * ncell; x += NT) scef[x] = kNoEdge;
    }
#pragma unroll 1
    for (int l = tid; l < nr; l += NT) cinv[cperm[l]] = l;
#pragma unroll 1
    for (int k = n_short + tid; k < nsp; k += NT) sllr[k] = 0.0f;
  }
  __syncthreads();
#pragma unroll 1
  for (int j = tid; j < nrp; j += NT) rc[j] = 0;
  __syncthreads();
#pragma unroll 1
  for (int k = tid; k < n_short; k += NT) {
    const int c = sel[vperm[k]], e0 = W.col_ptr[c], d = svd[k];
    sllr[k] = W.llr[c];
    const int ci = (coff[k >> 5] & (kWideSlice - 1)) * 32 + (k & 31);
#pragma unroll 1
    for (int u = 0; u < d; ++u) {
      const int r = cinv[W.col_rows[e0 + u]];
      const int pos = atomicAdd(&rc[r], 1);
      const int ri = (roff[r >> 5] + (pos >> 2)) * 128 + 4 * (r & 31) + (pos & 3);
      rent[ri] = 4u * (unsigned)k;
      cent[ci + 32 * u] = ((unsigned)r << 16) | (unsigned)pos;
      if (LW) {  // the shortened edge keeps its full-window edge's weights
        sref[ri] = (uint16_t)(e0 + u);
        scef[ci + 32 * u] = (uint16_t)(e0 + u);
      }
    }
  }
  __syncthreads();
  return false;
}

template <int UG>
__device__ __forceinline__ ShortG short_graph(const DecodeArgs& A, char* sm, const Layout& L, const SlotPlan& S,
                                              const WinDev& W, int ns) {
  const char *ents = graph_base<UG>(A, sm), *ids = ids_base<UG>(A, sm);
  return ShortG{W.n_rows, ns, L.rw, L.sw, S.rwz,
                (const uint32_t*)(ents + S.rent), (const uint32_t*)(ents + S.cent),
                (const uint16_t*)(sm + L.s_roff), (const uint16_t*)(sm + L.s_coff),
                (const float*)(sm + L.s_llr),     (const uint8_t*)(sm + L.s_vdeg),
                (const uint32_t*)(sm + L.sbits),  (const uint16_t*)(ids + S.ref),   (const uint16_t*)(ids + S.cef),
                (const ColClasses*)(sm + L.s_cls), W.wts, W.wT, W.n_edges, W.rows_per_block,
                (const uint16_t*)(sm + L.sel),
                (const uint16_t*)(sm + L.s_cperm), (const uint16_t*)(sm + L.s_vperm), W.n_commit_rows};
}

__device__ __forceinline__ PathOut trace_out(const DecodeArgs& A, char* tr, int id, long long shot) {
  PathOut o{};
  if (tr) {
    o.btr = (BranchTrace*)(tr + trace_off_br()) + id;
    o.st = (StepTrace*)(tr + trace_off_st(A.P.nb)) + (size_t)id * A.dmx;
    o.fstat = (int8_t*)(tr + trace_off_fs(A.P.nb, A.dmx)) + (size_t)id * A.ns_max;
  }
  o.visits = &A.counters[1];
  o.exec = A.exec;
  o.shot = shot;
  return o;
}

// The output path of a window in which no path converged: path 0, or under a
// fallback rule the least fallback key (stored in the path-metric slot of an
// unconverged path), ties to the lowest id.
__device__ __forceinline__ int fallback_path(const KParams& P, const double* pm) {
  int fb = 0;
  if (P.fallback)
#pragma unroll 1
    for (int id = 1; id < P.nb; ++id)
      if (pm[id] < pm[fb]) fb = id;
  return fb;
}

__device__ void write_outputs(const DecodeArgs& A, char* sm, long long shot, bool conv, int winner,
                              int n_short, int t_run, char* tr) {
  const Layout& L = A.L;
  const int tid = threadIdx.x, NT = blockDim.x;
  const uint32_t* cbits = (const uint32_t*)(sm + L.cbits);
  uint32_t* co = A.corr + (size_t)shot * A.corr_words;
#pragma unroll 1
  for (int x = tid; x < A.corr_words; x += NT) co[x] = x < L.cw ? cbits[x] : 0u;
  if (tr && !conv)
#pragma unroll 1
    for (int k = tid; k < n_short; k += NT)
      ((uint16_t*)(tr + trace_off_sel(A.P.nb, A.dmx, A.ns_max)))[k] = ((const uint16_t*)(sm + L.sel))[k];
  if (tid == 0) {
    if (A.status_out) A.status_out[shot] = conv ? -1 : (winner >= 0 ? winner : -2);
    if (tr) {
      int32_t* h = (int32_t*)tr;
      h[0] = conv ? 1 : 0;
      h[1] = conv ? -1 : winner;
      h[2] = conv ? 0 : n_short;
      h[3] = t_run;
    }
    atomicAdd((unsigned long long*)&A.counters[0], (unsigned long long)t_run * A.W.n_edges);
    atomicAdd((unsigned long long*)&A.counters[conv ? 2 : 3], 1ull);
  }
}

// Message reuse: the values this window leaves the next one, per window
// column (all threads of the CTA).  kp = the output path's values by label;
// kp = nullptr: the pre-BP converged, and its posterior `post` (still in the
// union region's pre-BP scratch) is kept for every column.
__device__ void keep_for_next(const DecodeArgs& A, char* sm, long long shot, const float* kp, int n_short,
                              const float* post = nullptr) {
  const int tid = threadIdx.x, NT = blockDim.x, nc = A.W.n_cols;
  float* out = A.keep + (size_t)shot * A.keep_ld;
  if (!kp) {
#pragma unroll 1
    for (int l = tid; l < nc; l += NT) out[A.W.s_col[l]] = post[l];
    return;
  }
  const uint16_t* sel = (const uint16_t*)(sm + A.L.sel);
  const uint16_t* vperm = (const uint16_t*)(sm + A.L.s_vperm);
#pragma unroll 1
  for (int c = tid; c < nc; c += NT) out[c] = CUDART_NAN_F;
  __syncthreads();
#pragma unroll 1
  for (int k = tid; k < n_short; k += NT) out[sel[vperm[k]]] = __ldcg(kp + k);
}

// ---- shot mode: persistent CTAs of up to 12 warps, one warp per decision path ----
// One shot of one window by the whole CTA (every thread calls).  misc[2], the
// decision-path queue, must be 0 on entry.
template <bool LW, int UG>
__device__ void shot_body(const DecodeArgs& A, long long shot, char* sm, Stager& stg) {
  const Layout& L = A.L;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int* misc = (int*)(sm + L.misc);
  int* res_status = (int*)(sm + L.res_status);
  double* res_pm = (double*)(sm + L.res_pm);
  uint32_t* res_e = (uint32_t*)(sm + L.res_ebits);
  uint32_t* cbits = (uint32_t*)(sm + L.cbits);
  const uint16_t* sel = (const uint16_t*)(sm + L.sel);
  char* tr = A.trace ? A.trace + (size_t)shot * A.tr_bytes : nullptr;
  int t_run = 0;
  const bool conv = window_prefix<LW, false, UG>(A, A.W, sm, shot, &t_run, stg);
  int winner = -1;
  const int n_short = conv ? 0 : A.W.n_short;
  if (!conv) {
    // warps beyond the shot's path slots sit out the paths
    const SlotPlan& S = *(const SlotPlan*)(sm + L.plan);
    if (warp < S.nslots) {
      const ShortG G = short_graph<UG>(A, sm, L, S, A.W, n_short);
      char* slot = union_base<UG>(A, sm, S) + (size_t)warp * S.b_size;
      const Slot B = make_slot(slot, S);
      const WarpGrp g{lane};
      // shared prefixes and preemption, when planned and this CTA has a pool
      const bool fork = A.F.pool && (int)blockIdx.x < A.F.pool_ctas;
      const int nb = A.P.nb;
      ForkCtx F{};
      F.flags = (int*)(sm + L.red);
      F.pool = fork ? A.F.pool + (size_t)blockIdx.x * A.F.cta_bytes : nullptr;
      F.stride = kSnapHeader + L.b_size;
      F.slot = slot;
      F.slot_bytes = S.b_size;
      F.st0 = tr ? (const StepTrace*)(tr + trace_off_st(nb)) : nullptr;
      F.sched = (fork && A.F.sched) ? (unsigned*)(sm + L.red) + kMaxForkNodes : nullptr;
      F.fnode = A.F.fnode;
      F.fdep = A.F.fdep;
      F.n_nodes = A.F.n_nodes;
      int next = -1;  // the path taken at a preemption point
      unsigned next_w = 0;
#pragma unroll 1
      while (true) {
        int id = -1;
        unsigned w0 = PS_QUEUED;  // the taken path's state word: queued or parked after step D
        if (next >= 0) {
          id = next;
          w0 = next_w;
          next = -1;
        } else {
#pragma unroll 1
          while (true) {  // the next queued path that no preemption took
            int pos = 0;
            if (lane == 0) pos = atomicAdd(&misc[2], 1);
            pos = __shfl_sync(FULL, pos, 0);
            if (pos >= nb) break;
            const int cand = fork ? (int)A.F.order[pos] : path_at(A.P, pos);
            int ok = 1;
            if (F.sched && lane == 0) ok = atomicCAS(&F.sched[cand], (unsigned)PS_QUEUED, (unsigned)PS_RUNNING) == PS_QUEUED;
            if (__shfl_sync(FULL, ok, 0)) {
              id = cand;
              break;
            }
          }
          if (id < 0 && F.sched) {  // a waiting path, the one with the most steps left
#pragma unroll 1
            for (int tries = 0; tries < 4 * nb; ++tries) {
              unsigned cw = 0;
              const int c = longest_waiting(A.P, F, lane, 0, cw);
              if (c < 0) break;
              int ok = 0;
              if (lane == 0) ok = atomicCAS(&F.sched[c], cw, (unsigned)PS_RUNNING) == cw;
              if (__shfl_sync(FULL, ok, 0)) {
                id = c;
                w0 = cw;
                break;
              }
            }
          }
          if (id < 0) break;
        }
        PathOut o = trace_out(A, tr, id, shot);
        o.status = &res_status[id];
        o.pm = &res_pm[id];
        o.ebits = res_e + (size_t)id * L.sw;
        if (A.keep) o.keep = A.kpath + ((size_t)blockIdx.x * nb + id) * A.ns_max;
        F.chain = (fork && F.n_nodes > 0) ? A.F.chain + (size_t)id * A.dmx : nullptr;
        F.src = nullptr;
        if ((w0 & 3u) == PS_PARKED) {  // its own parking snapshot
          __threadfence();
          F.src = F.pool + (size_t)(F.n_nodes + id) * F.stride;
        } else if (F.chain) {  // the deepest ready snapshot on this path's chain
          int node = -1;
          const int dm = path_dmax(A.P, id, path_split(A.P, id));
#pragma unroll 1
          for (int b = (dm - 1) & ~31; b >= 0 && node < 0; b -= 32) {  // a lane per depth
            const int n = b + lane < dm ? F.chain[b + lane] : -1;
            const unsigned m = __ballot_sync(FULL, n >= 0 && *(volatile int*)&F.flags[n >= 0 ? n : 0] == 2);
            if (m) node = __shfl_sync(FULL, n, 31 - __clz(m));
          }
          if (node >= 0) {
            __threadfence();  // the snapshot's contents after its flag
            F.src = F.pool + (size_t)node * F.stride;
          }
        }
        next = run_path<LW>(A.P, G, B, id, g, o, A.dmx, F, &next_w);
      }
    }
    __syncthreads();
    // ---- a8: least path metric, ties to the lowest id ----
    if (tid == 0) {
      int best = -1;
      double bp = CUDART_INF;
#pragma unroll 1
      for (int id = 0; id < A.P.nb; ++id)
        if (res_status[id] == BR_CONVERGED && res_pm[id] < bp) {
          bp = res_pm[id];
          best = id;
        }
      misc[1] = best;
      misc[4] = best >= 0 ? best : fallback_path(A.P, res_pm);
    }
    __syncthreads();
    winner = misc[1];
    const int outp = misc[4];
    const uint32_t* eb = res_e + (size_t)outp * L.sw;
#pragma unroll 1
    for (int k = tid; k < n_short; k += blockDim.x)
      if ((eb[k >> 5] >> (k & 31)) & 1u) atomicOr(&cbits[sel[k] >> 5], 1u << (sel[k] & 31));
    if (A.keep) {
      const float* kp = A.kpath + ((size_t)blockIdx.x * A.P.nb + outp) * A.ns_max;
      keep_for_next(A, sm, shot, kp, n_short);
    }
    __syncthreads();
  } else if (A.keep) {
    keep_for_next(A, sm, shot, nullptr, 0, (const float*)(prebp_base<UG>(A, sm) + L.p_post));
  }
  write_outputs(A, sm, shot, conv, winner, n_short, t_run, tr);
}

// CTAS: CTAs per SM (register budget), see configure_layouts.  What bounds it with
// three: instruction issue (73 % of the cycles), the ALU pipe (65 % of its peak)
// and shared-memory wavefronts (69 %, 29 % of them bank conflicts), at 22.6 warps
// per SM; HBM is idle.  One warp per path keeps every barrier of a path a warp's;
// 5000 shots of [[144,12,12]], all windows, took 450 ms with two CTAs per SM and
// the graph in CSR, 231 ms so; 9001 of the paper preset 200 and 104 ms.
template <bool LW, int UG, int CTAS>
__global__ void __launch_bounds__(CTAS == 1 ? 384 : 256, CTAS) decode_shot_kernel(DecodeArgs A) {
  extern __shared__ __align__(16) char sm[];
  int* misc = (int*)(sm + A.L.misc);
  Stager stg = stager_init((char*)(misc + 8), &A.counters[4]);
#pragma unroll 1
  while (true) {
    __syncthreads();
    if (threadIdx.x == 0) {
      misc[0] = atomicAdd(A.work, 1);
      misc[2] = 0;  // decision-path queue, path 0 first
    }
    // no snapshot yet, every path queued
    if (threadIdx.x < 2 * kMaxForkNodes) ((int*)(sm + A.L.red))[threadIdx.x] = 0;
    __syncthreads();
    const long long shot = misc[0];
    if (shot >= A.n_shots) break;
    shot_body<LW, UG>(A, shot, sm, stg);
  }
}

// ---- batched shot mode: one persistent launch over the same window step of
// several decoders (codes and window sizes of different shapes).  Shots are
// numbered across the members in table order; a CTA takes the next one and
// runs it with that member's graph, layout and buffers.  A member's layout
// has as many path slots as fit in the launch's shared memory (at most one
// per warp): small windows use every warp, large ones fewer. ----
template <bool LW>
__global__ void __launch_bounds__(256, 2) decode_batch_kernel(const __grid_constant__ BatchArgs B) {
  extern __shared__ __align__(16) char sm[];
  int* q = (int*)(sm + B.q_off);
  Stager stg = stager_init((char*)(q + 4), &B.seg[0].counters[4]);
#pragma unroll 1
  while (true) {
    __syncthreads();
    if (threadIdx.x == 0) q[0] = atomicAdd(B.work, 1);
    __syncthreads();
    const long long g = q[0];
    if (g >= B.seg_end[B.n_seg - 1]) break;
    int m = 0;
#pragma unroll 1
    while (g >= B.seg_end[m]) ++m;
    const DecodeArgs& A = B.seg[m];
    const long long shot = g - (m ? B.seg_end[m - 1] : 0);
    if (threadIdx.x == 0) ((int*)(sm + A.L.misc))[2] = 0;
    if (A.F.pool)  // no snapshot yet, every path queued (a CTA may have fewer threads than there are words)
#pragma unroll 1
      for (int x = threadIdx.x; x < 2 * kMaxForkNodes; x += blockDim.x) ((int*)(sm + A.L.red))[x] = 0;
    __syncthreads();
    // (members without learned weights may share the launch with others)
    if (LW && A.W.wts) shot_body<true, 0>(A, shot, sm, stg);
    else shot_body<false, 0>(A, shot, sm, stg);
  }
}

// ---- path mode: one CTA per (shot, path); the last CTA of a shot decides ----
// What bounds it: one path's serial chain (250 iterations of two passes with a
// barrier each) after the cluster's pre-BP; 16 CTAs of 512 threads for one
// [[144,12,12]] shot issue in 34 % of the cycles, half of the stalls are barriers.
// One shot, all windows decoded and committed: 8.2 ms with eight lanes per check,
// remote reads in the pre-BP and the graph in CSR, 5.9 ms so.  The threads per CTA
// follow the batch (path_shape).
template <bool LW, int UG>
__global__ void __launch_bounds__(512, 1) decode_path_kernel(DecodeArgs A) {
  extern __shared__ __align__(16) char sm[];
  const Layout& L = A.L;
  const int tid = threadIdx.x;
  const int nb = A.P.nb;
  const long long shot = blockIdx.x / A.cps;
  const int id = blockIdx.x % A.cps;
  int* misc = (int*)(sm + L.misc);
  char* tr = A.trace ? A.trace + (size_t)shot * A.tr_bytes : nullptr;
  Stager stg = stager_init((char*)(misc + 8), &A.counters[4]);
  int t_run = 0;
  const bool conv = window_prefix<LW, true, UG>(A, A.W, sm, shot, &t_run, stg);
  if (id >= nb) return;  // a CTA that only shared the pre-BP of its cluster
  if (conv) {
    if (id == 0) {
      write_outputs(A, sm, shot, true, -1, 0, t_run, tr);
      if (A.keep) keep_for_next(A, sm, shot, nullptr, 0, (const float*)(prebp_base<UG>(A, sm) + L.p_post));
    }
    return;
  }
  const int n_short = A.W.n_short;
  const SlotPlan& S = *(const SlotPlan*)(sm + L.plan);
  const ShortG G = short_graph<UG>(A, sm, L, S, A.W, n_short);
  const Slot B = make_slot(union_base<UG>(A, sm, S), S);
  const CtaGrp g{tid, (int)blockDim.x, sm + L.red};
  const size_t rb = path_result_bytes(A.sw_max);
  char* mine = A.path_res + ((size_t)shot * nb + id) * rb;
  PathOut o = trace_out(A, tr, id, shot);
  o.status = (int*)mine;
  o.pm = (double*)(mine + 8);
  o.ebits = (uint32_t*)(mine + 16);
  if (A.keep) o.keep = A.kpath + ((size_t)shot * nb + id) * A.ns_max;
  run_path<LW>(A.P, G, B, id, g, o, A.dmx, ForkCtx{});
  // publish, then count arrivals; the last CTA of the shot reduces
  __threadfence();
  __syncthreads();
  if (tid == 0) misc[3] = (atomicAdd(&A.arrive[shot], 1) == nb - 1);
  __syncthreads();
  if (!misc[3]) return;
  __threadfence();
  if (tid == 0) {
    int best = -1, fb = 0;
    double bp = CUDART_INF, bk = CUDART_INF;
#pragma unroll 1
    for (int q = 0; q < nb; ++q) {
      const char* r = A.path_res + ((size_t)shot * nb + q) * rb;
      const int st = __ldcg((const int*)r);
      const double pm = __ldcg((const double*)(r + 8));
      if (st == BR_CONVERGED && pm < bp) {
        bp = pm;
        best = q;
      }
      if (A.P.fallback && st != BR_CONVERGED && pm < bk) {  // the fallback key (see fallback_path)
        bk = pm;
        fb = q;
      }
    }
    misc[1] = best;
    misc[4] = best >= 0 ? best : fb;
    A.arrive[shot] = 0;  // ready for the next launch
  }
  __syncthreads();
  const int winner = misc[1];
  const int outp = misc[4];
  const uint32_t* eb = (const uint32_t*)(A.path_res + ((size_t)shot * nb + outp) * rb + 16);
  uint32_t* cbits = (uint32_t*)(sm + L.cbits);
  const uint16_t* sel = (const uint16_t*)(sm + L.sel);
#pragma unroll 1
  for (int k = tid; k < n_short; k += blockDim.x)
    if ((__ldcg(&eb[k >> 5]) >> (k & 31)) & 1u) atomicOr(&cbits[sel[k] >> 5], 1u << (sel[k] & 31));
  if (A.keep) keep_for_next(A, sm, shot, A.kpath + ((size_t)shot * nb + outp) * A.ns_max, n_short);
  __syncthreads();
  write_outputs(A, sm, shot, false, winner, n_short, t_run, tr);
}

// Learned weights of a window in the order in which the pre-BP's passes walk its
// edges, [T][check entries] and [T][column entries], so that they load them
// side by side instead of through edge ids.  Runs before every decode of the
// window (the caller may change the weights in between): 1.4 MB for
// [[144,12,12]] (3,1) windows and T = 25, a few microseconds at L2 rates.  2000
// shots took 181 ms with gathers through edge ids, 147 ms so.
__global__ void __launch_bounds__(256) order_weights_kernel(const float* __restrict__ w, const uint16_t* __restrict__ ref,
                                                            const uint16_t* __restrict__ cef, int T, int ne, int nrow,
                                                            int ncol, float* __restrict__ w_row,
                                                            float* __restrict__ w_col) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, t = blockIdx.y;
  if (i >= nrow + ncol) return;
  const uint32_t e = i < nrow ? ref[i] : cef[i - nrow];
  const float x = e == kNoEdge ? 0.0f : w[(size_t)t * ne + e];
  if (i < nrow) w_row[(size_t)t * nrow + i] = x;
  else w_col[(size_t)t * ncol + (i - nrow)] = x;
}

// ---- Philox4x32-10 (Salmon et al., SC'11) ----
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    k.x += 0x9E3779B9u;
    k.y += 0xBB67AE85u;
  }
  return c;
}

// One warp per shot, four columns per lane and trip.  Fired columns (some 25 of
// 8784 at p = 0.003) go to a list in shared memory that the warp works off one
// column per lane, so that the loads of a column's detectors wait for one
// another once per list and not once per fault.  What bounds it: the integer
// instructions of Philox (ten rounds, two wide multiplications and two
// three-way xors each; the multiplier is what warps wait for).  100000 shots of
// [[144,12,12]], 12 rounds, took 1061 us with scalar threshold loads and every
// fault worked off on the spot, 726 us so.
constexpr int kFireList = 160;  // at most 31 waiting and 128 new ones a trip
__global__ void __launch_bounds__(256) sample_kernel(int n_cols, const uint4* __restrict__ thr,
                                                     const int* __restrict__ cptr, const int* __restrict__ cdet,
                                                     const uint32_t* __restrict__ cobs, int det_words,
                                                     unsigned long long seed, unsigned long long off, long long n,
                                                     uint32_t* __restrict__ det, uint32_t* __restrict__ obs) {
  extern __shared__ uint32_t srow[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  const long long s = (long long)blockIdx.x * wpb + wib;
  if (s >= n) return;  // the whole warp
  uint32_t* row = srow + (size_t)wib * det_words;
  int* list = (int*)(srow + (size_t)wpb * det_words) + wib * kFireList;
  for (int x = lane; x < det_words; x += 32) row[x] = 0;
  __syncwarp();
  uint32_t ob = 0;
  int cnt = 0;
  auto flush = [&]() {
    __syncwarp();
    for (int i = lane; i < cnt; i += 32) {
      const int c = list[i];
      const int e0 = cptr[c], e1 = cptr[c + 1];
      ob ^= cobs[c];
      for (int e = e0; e < e1; ++e) {
        const int d = cdet[e];
        atomicXor(&row[d >> 5], 1u << (d & 31));
      }
    }
    cnt = 0;
    __syncwarp();
  };
  const unsigned long long shot = off + (unsigned long long)s;
  const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
  const int ng = (n_cols + 3) >> 2, full = ng & ~63;
  auto fired = [&](int g, const uint4& u, const uint4& t) {  // columns 4 g .. 4 g + 3, every lane calling
    const bool f[4] = {u.x < t.x, u.y < t.y, u.z < t.z, u.w < t.w};
    if (!__any_sync(FULL, f[0] | f[1] | f[2] | f[3])) return;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const unsigned m = __ballot_sync(FULL, f[r]);
      if (f[r]) list[cnt + __popc(m & ((1u << lane) - 1u))] = 4 * g + r;
      cnt += __popc(m);
    }
    if (cnt >= 32) flush();
  };
  auto draw = [&](int g) {
    return philox4x32_10(make_uint4((uint32_t)g, (uint32_t)shot, (uint32_t)(shot >> 32), 0u), key);
  };
#pragma unroll 1
  for (int g = lane; g < full; g += 64) {  // two independent draws
    const uint4 t0 = thr[g], t1 = thr[g + 32];
    const uint4 u0 = draw(g), u1 = draw(g + 32);
    fired(g, u0, t0);
    fired(g + 32, u1, t1);
  }
#pragma unroll 1
  for (int b = full; b < ng; b += 32) {  // (thresholds past the last column are 0: they never fire)
    const int g = b + lane;
    const uint4 t = g < ng ? thr[g] : make_uint4(0u, 0u, 0u, 0u);
    fired(g, draw(g), t);
  }
  flush();
  ob = __reduce_xor_sync(FULL, ob);
  for (int x = lane; x < det_words; x += 32) det[(size_t)s * det_words + x] = row[x];
  if (lane == 0) obs[s] = ob;
}

// Commit (Eq. (10)) + residue test (Eq. (11)) of shot s.
__device__ void commit_one(const CommitArgs& C, long long s) {
  const uint32_t* c = C.corr + (size_t)s * C.corr_words;
  uint32_t* d = C.det + (size_t)s * C.det_words;
  uint32_t ob = 0;
  const int nw = (C.n_commit + 31) >> 5;
#pragma unroll 1
  for (int x = 0; x < nw; ++x) {
    uint32_t m = c[x];
    const int rem = C.n_commit - 32 * x;
    if (rem < 32) m &= (1u << rem) - 1u;
#pragma unroll 1
    while (m) {
      const int b = __ffs(m) - 1;
      m &= m - 1;
      const int col = 32 * x + b;
#pragma unroll 1
      for (int e = C.cptr[col]; e < C.cptr[col + 1]; ++e) {
        const int q = C.cdet[e];
        d[q >> 5] ^= 1u << (q & 31);
      }
      ob ^= C.cobs[col];
    }
  }
  C.obs_pred[s] ^= ob;
  uint32_t bad = 0;
#pragma unroll 1
  for (int q = C.b0; q < C.b1;) {
    const int wq = q >> 5, lo = q & 31;
    const int hiq = min(C.b1, (wq + 1) * 32);
    uint32_t m = d[wq] >> lo;
    const int nb = hiq - q;
    if (nb < 32) m &= (1u << nb) - 1u;
    bad |= m;
    q = hiq;
  }
  if (bad) C.resid[s] |= 1u;
}

// one thread per shot
__global__ void commit_kernel(const CommitArgs C) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s < C.n) commit_one(C, s);
}

// one thread per shot over several decoders' shots
__global__ void commit_batch_kernel(const __grid_constant__ CommitBatch B) {
  const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= B.seg_end[B.n_seg - 1]) return;
  int m = 0;
#pragma unroll 1
  while (g >= B.seg_end[m]) ++m;
  commit_one(B.seg[m], g - (m ? B.seg_end[m - 1] : 0));
}

__global__ void evaluate_kernel(const uint32_t* __restrict__ pred, const uint32_t* __restrict__ obs,
                                const uint32_t* __restrict__ resid, long long n, uint32_t* __restrict__ fail,
                                long long* __restrict__ n_fail) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t f = 0;
  if (s < n) {
    f = (resid[s] & 1u) | ((pred[s] != obs[s]) ? 2u : 0u);
    if (fail) fail[s] = f;
  }
  const unsigned m = __ballot_sync(FULL, f != 0);
  if (n_fail && (threadIdx.x & 31) == 0 && m) atomicAdd((unsigned long long*)n_fail, (unsigned long long)__popc(m));
}

}  // namespace dev

// ---------------------------------------------------------------------------
// Host-side launch wrappers (declared in qdec_internal.h).

size_t trace_bytes_per_shot(int nb, int dmx, int ns_max) { return dev::trace_bytes(nb, dmx, ns_max); }

cudaError_t set_decode_smem(size_t bytes) {
  const void* f[] = {(const void*)dev::decode_shot_kernel<false, 0, 2>, (const void*)dev::decode_shot_kernel<true, 0, 2>,
                     (const void*)dev::decode_shot_kernel<false, 1, 2>,  (const void*)dev::decode_shot_kernel<true, 1, 2>,
                     (const void*)dev::decode_shot_kernel<false, 2, 2>, (const void*)dev::decode_shot_kernel<true, 2, 2>,
                     (const void*)dev::decode_shot_kernel<false, 0, 1>, (const void*)dev::decode_shot_kernel<true, 0, 1>,
                     (const void*)dev::decode_shot_kernel<false, 0, 3>, (const void*)dev::decode_path_kernel<false, 0>,
                     (const void*)dev::decode_path_kernel<true, 0>,         (const void*)dev::decode_path_kernel<true, 3>,
                     (const void*)dev::decode_batch_kernel<false>,
                     (const void*)dev::decode_batch_kernel<true>};
  for (const void* k : f)
    if (cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes)) return e;
  return cudaSuccess;
}

cudaError_t batch_occupancy(int threads, size_t smem, int* blocks) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, dev::decode_batch_kernel<false>, threads, smem);
}

cudaError_t launch_decode_batch(cudaStream_t st, int grid, int threads, size_t smem, unsigned q_off, int* work,
                                const BatchMember* m, int n) {
  if (n <= 0 || n > kMaxBatch) return n <= 0 ? cudaSuccess : cudaErrorInvalidValue;
  dev::BatchArgs B{};
  B.n_seg = n;
  B.q_off = q_off;
  B.work = work;
  bool lw = false;
  long long end = 0;
  for (int i = 0; i < n; ++i) {
    const BatchMember& x = m[i];
    end += x.n;
    B.seg_end[i] = end;
    B.seg[i] = dev::DecodeArgs{*x.P,   *x.W,   *x.L,     x.det,      x.det_words, x.n,      x.corr,
                               x.corr_words, nullptr, nullptr, 0,     x.dmx,    x.ns_max, nullptr,
                               x.counters, nullptr, nullptr, x.sw_max, nullptr, 0, 1,
                               x.counters ? x.counters + 5 : nullptr, x.fork ? *x.fork : ForkDev{}};
    lw = lw || x.W->wts != nullptr;
  }
  if (lw) dev::decode_batch_kernel<true><<<grid, threads, smem, st>>>(B);
  else dev::decode_batch_kernel<false><<<grid, threads, smem, st>>>(B);
  return cudaGetLastError();
}

cudaError_t launch_commit_batch(cudaStream_t st, const BatchMember* m, int n) {
  if (n <= 0 || n > kMaxBatch) return n <= 0 ? cudaSuccess : cudaErrorInvalidValue;
  dev::CommitBatch B{};
  B.n_seg = n;
  long long end = 0;
  for (int i = 0; i < n; ++i) {
    const BatchMember& x = m[i];
    end += x.n;
    B.seg_end[i] = end;
    B.seg[i] = dev::CommitArgs{x.n_commit, x.cptr, x.cdet, x.cobs, x.corr_words, x.corr, x.n,
                               (uint32_t*)x.det, x.det_words, x.obs_pred, x.resid, x.b0, x.b1};
  }
  if (end == 0) return cudaSuccess;
  const int tpb = 128;
  dev::commit_batch_kernel<<<(unsigned)((end + tpb - 1) / tpb), tpb, 0, st>>>(B);
  return cudaGetLastError();
}

cudaError_t decode_occupancy(int mode, int ctas, int threads, size_t smem, int* blocks) {
  if (mode == 1)
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, dev::decode_path_kernel<false, 0>, threads, smem);
  if (mode == 4)  // shot mode with the shortened graph's entries in global memory as well
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, dev::decode_shot_kernel<false, 2, 2>, threads, smem);
  if (mode == 3)  // shot mode with the union region in global memory
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, dev::decode_shot_kernel<false, 1, 2>, threads, smem);
  if (ctas == 1)
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, dev::decode_shot_kernel<false, 0, 1>, threads, smem);
  if (ctas >= 3)
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, dev::decode_shot_kernel<false, 0, 3>, threads, smem);
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, dev::decode_shot_kernel<false, 0, 2>, threads, smem);
}

cudaError_t path_cluster_occupancy(int threads, size_t smem, int cluster, int* clusters) {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at[1];
  cfg.gridDim = dim3((unsigned)cluster);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cluster;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaOccupancyMaxActiveClusters(clusters, dev::decode_path_kernel<false, 0>, &cfg);
}

cudaError_t launch_decode(int mode, int ctas, int grid, int threads, size_t smem, cudaStream_t st, const KParams& P,
                          const WinDev& W, const Layout& L, const uint32_t* det, int det_words, long long n,
                          uint32_t* corr, int corr_words, int32_t* status, char* trace, size_t tr_bytes, int dmx,
                          int ns_max, int* work, long long* counters, char* path_res, int* arrive, int sw_max,
                          char* uglob, size_t ubytes, int cps, int cluster, const ForkDev* fork,
                          const ReuseDev* reuse) {
  // counters[5]: the GDG edge visits the launch executed (counters[1] adds
  // the resumed prefixes every path counts as its own)
  const dev::DecodeArgs A{P,     W,        L,     det,      det_words, n,     corr,     corr_words, status,
                          trace, tr_bytes, dmx,   ns_max,   work,      counters, path_res, arrive,     sw_max,
                          uglob, ubytes,   cps,   counters ? counters + 5 : nullptr, fork ? *fork : ForkDev{},
                          reuse ? reuse->keep : nullptr, reuse ? reuse->keep_ld : 0, reuse ? reuse->prev : nullptr,
                          reuse ? reuse->kpath : nullptr};
  const bool lw = W.wts != nullptr;
  if (mode == 1) {  // one cluster of `cluster` CTAs shares each shot's pre-BP
    // every path needs its CTA, and a cluster never spans two shots
    if (cluster < 1 || cps < P.nb || cps % cluster || grid % cps) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cluster;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (lw && L.gg == kIdsGlobal) {
      if (!uglob) return cudaErrorInvalidValue;
      return cudaLaunchKernelEx(&cfg, dev::decode_path_kernel<true, 3>, A);
    }
    if (lw) return cudaLaunchKernelEx(&cfg, dev::decode_path_kernel<true, 0>, A);
    return cudaLaunchKernelEx(&cfg, dev::decode_path_kernel<false, 0>, A);
  } else {
    if (uglob && L.gg == kGraphGlobal) {
      if (lw) dev::decode_shot_kernel<true, 2, 2><<<grid, threads, smem, st>>>(A);
      else dev::decode_shot_kernel<false, 2, 2><<<grid, threads, smem, st>>>(A);
    } else if (uglob) {
      if (lw) dev::decode_shot_kernel<true, 1, 2><<<grid, threads, smem, st>>>(A);
      else dev::decode_shot_kernel<false, 1, 2><<<grid, threads, smem, st>>>(A);
    } else if (ctas == 1) {
      if (lw) dev::decode_shot_kernel<true, 0, 1><<<grid, threads, smem, st>>>(A);
      else dev::decode_shot_kernel<false, 0, 1><<<grid, threads, smem, st>>>(A);
    } else if (ctas >= 3 && !lw) {
      dev::decode_shot_kernel<false, 0, 3><<<grid, threads, smem, st>>>(A);
    } else {
      if (lw) dev::decode_shot_kernel<true, 0, 2><<<grid, threads, smem, st>>>(A);
      else dev::decode_shot_kernel<false, 0, 2><<<grid, threads, smem, st>>>(A);
    }
  }
  return cudaGetLastError();
}

cudaError_t launch_order_weights(cudaStream_t st, const WinDev& W) {
  const int nrow = 128 * W.row_quads, ncol = 32 * W.col_cells;
  for (int t0 = 0; t0 < W.w_rows; t0 += 65535) {  // (the grid's y limit)
    const int T = W.w_rows - t0 < 65535 ? W.w_rows - t0 : 65535;
    dev::order_weights_kernel<<<dim3((unsigned)((nrow + ncol + 255) / 256), (unsigned)T), 256, 0, st>>>(
        W.wts + (size_t)t0 * W.n_edges, W.s_ref, W.s_cef, T, W.n_edges, nrow, ncol, W.w_row + (size_t)t0 * nrow,
        W.w_col + (size_t)t0 * ncol);
  }
  return cudaGetLastError();
}

cudaError_t launch_sample(cudaStream_t st, int n_cols, const uint32_t* thr, const int* cptr, const int* cdet,
                          const uint32_t* cobs, int det_words, unsigned long long seed, unsigned long long off,
                          long long n, uint32_t* det, uint32_t* obs) {
  if (n <= 0) return cudaSuccess;
  // eight warps per CTA, fewer where their rows and fire lists would not fit the
  // shared memory that any kernel may have (more than 1376 detector words)
  int wpb = 8;
  while (wpb > 1 && sizeof(uint32_t) * wpb * (det_words + dev::kFireList) > (48u << 10)) wpb >>= 1;
  const long long blocks = (n + wpb - 1) / wpb;
  dev::sample_kernel<<<(unsigned)blocks, 32 * wpb, sizeof(uint32_t) * wpb * (det_words + dev::kFireList), st>>>(
      n_cols, (const uint4*)thr, cptr, cdet, cobs, det_words, seed, off, n, det, obs);
  return cudaGetLastError();
}

cudaError_t launch_commit(cudaStream_t st, int n_commit, const int* cptr, const int* cdet, const uint32_t* cobs,
                          int corr_words, const uint32_t* corr, long long n, uint32_t* det, int det_words,
                          uint32_t* obs_pred, uint32_t* resid, int b0, int b1) {
  if (n <= 0) return cudaSuccess;
  const int tpb = 128;
  const dev::CommitArgs C{n_commit, cptr, cdet, cobs, corr_words, corr, n, det, det_words, obs_pred, resid, b0, b1};
  dev::commit_kernel<<<(unsigned)((n + tpb - 1) / tpb), tpb, 0, st>>>(C);
  return cudaGetLastError();
}

cudaError_t launch_evaluate(cudaStream_t st, const uint32_t* pred, const uint32_t* obs, const uint32_t* resid,
                            long long n, uint32_t* fail, long long* n_fail) {
  if (n <= 0) return cudaSuccess;
  const int tpb = 256;
  dev::evaluate_kernel<<<(unsigned)((n + tpb - 1) / tpb), tpb, 0, st>>>(pred, obs, resid, n, fail, n_fail);
  return cudaGetLastError();
}

}  // namespace qd
