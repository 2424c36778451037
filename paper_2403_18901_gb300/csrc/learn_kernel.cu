// learn_kernel.cu -- training kernels of the learned weighted min-sum.
//
// There is no counterpart in the paper: the fixed normalisation alpha of
// Eq. (1) becomes a weight w[t][e] per edge and iteration, trained by
// gradient descent on window samples.
//
// Forward (one sample = one window syndrome), T unrolled flooding iterations
// on the full window with explicit per-edge messages, t = 1..T:
//   c2v[e]  = (-1)^{s_j} * w[t][e] * min_{e' != e} |v2c[e']| * prod_{e' != e} sign(v2c[e'])
//   post[i] = Lambda_i + sum_{e in M(i)} c2v[e]          (ascending check order)
//   v2c[e]  = clip(post[i] - c2v[e], +-clip)
// starting from v2c = Lambda.  Loss: soft-syndrome BCE at t = T,
//   P(check j odd) = (1 - prod_{i in N(j)} tanh(post_i / 2)) / 2,
//   loss = mean_j BCE(P_j, s_j),
// since 1 - 2 sigma(-x) = tanh(x / 2).
// Backward: the adjoint of the unrolled iterations.  A min-sum check sends each
// edge the magnitude of one other edge (the smallest, or the second smallest
// for the edge holding the smallest), so its gradient flows to at most two
// inputs; derivatives of sign() and of a saturated clip are zero.  Everything
// the adjoint of iteration t needs of the forward pass is in the checks'
// records of iterations t and t + 1: the two smallest magnitudes and their
// positions and the messages' signs; an input is within the clip exactly when
// its magnitude is below it.  So the forward pass keeps 16 bytes per check and
// iteration in global scratch and nothing is computed twice -- or, where that
// would take too much memory (kWmsKeepBytes), every `ckpt`-th iteration's, and
// the backward pass computes the records of one segment at a time again from
// the one before it (a record and its iteration's weights give every message,
// so what it computes is what the forward pass computed).  The gradient
// into the inputs of an iteration is non-zero at two edges per check only:
// their cells are written, the columns sum theirs in ascending order (float
// atomics on the columns would be quicker by a tenth, but make a sample's
// gradient vary between runs), and an edge whose column got nothing has no
// weight gradient (but in the last iteration, where every column has one).
// FP32 throughout (the loss is summed in FP64); tanhf / logf are CUDA's.
//
// What bounds it: issue and latency of the checks' serial passes over their 35
// inputs; 40 KB of shared memory a CTA for [[144,12,12]] (3,1) windows keeps
// four CTAs of 8 warps on an SM.  With the messages of both directions and
// their gradients in shared memory (123 KB, one CTA per SM), checkpoints and
// two recomputations, 1024 samples of 25 iterations took 10.0 ms; so, 1.06 ms
// (five CTAs per SM spill: 1.37 ms).
#include <cuda_runtime.h>
#include <math_constants.h>

#include <cstdint>
#include <type_traits>

#include "gdg_kernel.cuh"

namespace qd {

namespace lrn {

constexpr unsigned FULL = 0xffffffffu;
__device__ __forceinline__ float clipf(float x, float c) { return x > c ? c : (x < -c ? -c : x); }

// A check's record of one iteration: its two smallest |v2c|; sg, pw: the signs
// of the messages it sends, position p at bit 31 - p of sg (p < 32) or bit
// 63 - p of pw; pw also holds (bit 12) whether the inputs' own signs are those
// inverted, and the positions of the two smallest inputs (bits 11..6 the
// second, 5..0 the first).
struct __align__(16) WRec {
  float m1, m2;
  uint32_t sg, pw;
};
__device__ __forceinline__ uint32_t rec_sign(const WRec& r, int p) {  // of position p's message, at bit 31
  return ((p < 32 ? r.sg : r.pw) << (p & 31)) & 0x80000000u;
}
__device__ __forceinline__ float with_sign(float x, uint32_t s) {
  return __uint_as_float(__float_as_uint(x) ^ s);
}

// Check pass of one check by one lane: the record of its inputs v2c.
__device__ __forceinline__ WRec check_forward(const uint16_t* cell, int n, const float* v2c, uint32_t sj) {
  float m1 = CUDART_INF_F, m2 = CUDART_INF_F;
  uint32_t p1 = 0u, p2 = 0u, sg[2] = {0u, 0u};
#pragma unroll
  for (int h = 0; h < 2; ++h) {  // 32 positions to a word
    const int u0 = 32 * h, u1 = min(n, u0 + 32);
    uint32_t s = 0u;
#pragma unroll 4
    for (int u = u0; u < u1; ++u) {
      const float x = v2c[cell[32 * u]];  // (a dummy is +inf)
      const float a = fabsf(x);
      const bool l1 = a < m1, l2 = a < m2;  // the first of equal magnitudes stays
      p2 = l1 ? p1 : (l2 ? (uint32_t)u : p2);
      p1 = l1 ? (uint32_t)u : p1;
      m2 = l1 ? m1 : (l2 ? a : m2);  // (a NaN, inf - inf, is neither)
      m1 = fminf(m1, a);
      s = s + s + (x < 0.0f ? 1u : 0u);
    }
    if (u1 > u0) sg[h] = s << ((32 - (u1 - u0)) & 31);
  }
  const uint32_t par = (__popc(sg[0]) + __popc(sg[1]) + sj) & 1u;
  const uint32_t all = 0u - par;  // message sign = parity xor s_j xor the own sign
  return WRec{m1, m2, sg[0] ^ all, ((sg[1] ^ all) & 0xFFFFE000u) | (par << 12) | (p2 << 6) | p1};
}

// The weight of a column entry; a dummy has no edge, and its message has to be
// +0 (an infinite weight would make it NaN).
__device__ __forceinline__ float entry_weight(const float* wt, uint32_t id) { return id == kNoEdge ? 0.0f : wt[id]; }

// Message of Eq. (1) with weight w for the edge at position p.
__device__ __forceinline__ float message(const WRec& r, uint32_t p, float w) {
  const float m = (r.pw & 63u) == p ? r.m2 : r.m1;
  return with_sign(__fmul_rn(w, m), rec_sign(r, (int)p));
}

// The records of iterations t0 + 1 .. t1 into out, from that of t0 (unused for
// t0 = 0), by the whole CTA with the forward pass's operations; v2c is zero
// before and after.  Apart from the kernel, whose registers it would take.
__device__ __noinline__ void recompute_records(const WmsSlices& G, const float* w, const uint32_t* sb, float* v2c,
                                               const WRec* from, int t0, int t1, WRec* out) {
  const int NT = blockDim.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = NT >> 5, nrp = 32 * G.nrs;
  auto columns = [&](const WRec* rec, const float* wt) {  // the inputs of the iteration after rec's
    for (int s = warp; s < G.ncs; s += nw) {
      const int c0 = 32 * G.coff[s] + lane, c1 = 32 * G.coff[s + 1];
      auto input = [&](int c) {
        const uint32_t e = G.cent[c], l = e >> 16;
        if ((int)l >= nrp) return 0.0f;  // the dummy check's message
        return message(rec[l], e & 0xFFFFu, entry_weight(wt, G.ceid[c]));
      };
      float p = G.llr[32 * s + lane];
      for (int c = c0; c < c1; c += 32) p = __fadd_rn(p, input(c));  // ascending check order
      for (int c = c0; c < c1; c += 32) v2c[c] = clipf(__fsub_rn(p, input(c)), G.clip);
    }
  };
  __syncthreads();
  if (t0 > 0) {
    columns(from, w + (size_t)(t0 - 1) * G.ne);
  } else {
    for (int s = warp; s < G.ncs; s += nw)
      for (int c = 32 * G.coff[s] + lane; c < 32 * G.coff[s + 1]; c += 32) v2c[c] = G.llr[32 * s + lane];
  }
  __syncthreads();
  for (int t = t0 + 1; t <= t1; ++t) {
    WRec* o = out + (size_t)(t - t0 - 1) * nrp;
    for (int s = warp; s < G.nrs; s += nw) {
      const int r0 = G.roff[s], l = 32 * s + lane, j = G.row[l];
      o[l] = check_forward(G.rcell + 32 * r0 + lane, G.roff[s + 1] - r0, v2c, (sb[j >> 5] >> (j & 31)) & 1u);
    }
    __syncthreads();
    if (t < t1) columns(o, w + (size_t)(t - 1) * G.ne);
    __syncthreads();
  }
  for (int c = threadIdx.x; c < 32 * G.col_cells; c += NT) v2c[c] = 0.0f;
  __syncthreads();
}

// SEG: G.seg > 0 (a template, so that the kernel that keeps every record has no
// bookkeeping for the others: 1 % of its time).
template <bool SEG>
__global__ void __launch_bounds__(256, 4) wms_kernel(const __grid_constant__ WmsSlices G, const float* __restrict__ w,
                                                     const uint32_t* __restrict__ synd, long long n, int backward,
                                                     float grad_scale, float* __restrict__ grad_w,
                                                     float* __restrict__ loss_out, float* __restrict__ post_out,
                                                     WRec* __restrict__ scratch, int* __restrict__ work) {
  extern __shared__ __align__(16) char smem[];
  const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = NT >> 5;
  const int nrp = 32 * G.nrs, ncp = 32 * G.ncs, cells = 32 * G.col_cells;
  float* v2c = (float*)smem;                       // by column cell; [cells] = +inf
  float* post = v2c + cells + 32;                  // by column label
  WRec* rec = (WRec*)(post + ncp + 32);                 // this iteration's, [nrp] = zero (the dummy check)
  uint32_t* sb = (uint32_t*)(rec + nrp + 1);       // window syndrome by row
  double* red = (double*)(sb + ((G.rw + 3) & ~3));  // [32]
  int* sh_sample = (int*)(red + 32);
  WRec* hist = scratch + (size_t)blockIdx.x * (SEG ? G.records() : G.T) * nrp;  // records by iteration (slot_forward)
  while (true) {
    __syncthreads();
    if (tid == 0) *sh_sample = atomicAdd(work, 1);
    __syncthreads();
    const long long smp = *sh_sample;
    if (smp >= n) break;
    for (int x = tid; x < G.rw; x += NT) sb[x] = synd[(size_t)smp * G.rw + x];
    for (int s = warp; s < G.ncs; s += nw) {  // t = 0: v2c = Lambda
      const float l = G.llr[32 * s + lane];
      for (int c = G.coff[s]; c < G.coff[s + 1]; ++c) v2c[32 * c + lane] = l;
    }
    if (tid == 0) {
      v2c[cells] = CUDART_INF_F;
      rec[nrp] = WRec{0.0f, 0.0f, 0u, 0u};
    }
    __syncthreads();
    // ---- forward ----
    for (int t = 1; t <= G.T; ++t) {
      const int slot = !backward ? -1 : (SEG ? G.slot_forward(t) : t - 1);
      for (int s = warp; s < G.nrs; s += nw) {
        const int r0 = G.roff[s], l = 32 * s + lane;
        const int j = G.row[l];  // window row (0 for the padding, whose inputs are dummies)
        const WRec r = check_forward(G.rcell + 32 * r0 + lane, G.roff[s + 1] - r0, v2c, (sb[j >> 5] >> (j & 31)) & 1u);
        rec[l] = r;
        if (SEG ? slot >= 0 : backward != 0) hist[(size_t)slot * nrp + l] = r;
      }
      __syncthreads();
      const float* wt = w + (size_t)(t - 1) * G.ne;
      for (int s = warp; s < G.ncs; s += nw) {
        const int c0 = G.coff[s], d = G.coff[s + 1] - c0;
        float p = G.llr[32 * s + lane];
        auto column = [&](auto cnt) {  // the messages stay in registers
          constexpr int N = decltype(cnt)::value;
          float m[N];
#pragma unroll
          for (int u = 0; u < N; ++u) {
            const int c = 32 * (c0 + u) + lane;
            const uint32_t e = G.cent[c];
            m[u] = message(rec[e >> 16], e & 0xFFFFu, entry_weight(wt, G.ceid[c]));
          }
#pragma unroll
          for (int u = 0; u < N; ++u) p = __fadd_rn(p, m[u]);  // ascending check order
#pragma unroll
          for (int u = 0; u < N; ++u) v2c[32 * (c0 + u) + lane] = clipf(__fsub_rn(p, m[u]), G.clip);
        };
        switch (d) {
          case 1: column(std::integral_constant<int, 1>{}); break;
          case 2: column(std::integral_constant<int, 2>{}); break;
          case 3: column(std::integral_constant<int, 3>{}); break;
          case 4: column(std::integral_constant<int, 4>{}); break;
          case 5: column(std::integral_constant<int, 5>{}); break;
          case 6: column(std::integral_constant<int, 6>{}); break;
          default:
            for (int pass = 0; pass < 2; ++pass)
              for (int u = 0; u < d; ++u) {
                const int c = 32 * (c0 + u) + lane;
                const uint32_t e = G.cent[c];
                const float m = message(rec[e >> 16], e & 0xFFFFu, entry_weight(wt, G.ceid[c]));
                if (pass == 0) p = __fadd_rn(p, m);
                else v2c[c] = clipf(__fsub_rn(p, m), G.clip);
              }
        }
        if (t == G.T) post[32 * s + lane] = p;
      }
      __syncthreads();
    }
    if (post_out)
      for (int l = tid; l < G.nc; l += NT) post_out[(size_t)smp * G.nc + G.col[l]] = post[l];
    // ---- soft-syndrome BCE; dLoss/dpost by edge in v2c's place ----
    __syncthreads();
    for (int l = tid; l < ncp; l += NT) post[l] = tanhf(0.5f * post[l]);
    __syncthreads();
    double lsum = 0.0;
    for (int s = warp; s < G.nrs; s += nw) {
      const int r0 = G.roff[s], d = G.roff[s + 1] - r0, l = 32 * s + lane;
      if (l >= G.nr) continue;
      const uint16_t *cell = G.rcell + 32 * r0 + lane, *col = G.rcol + 32 * r0 + lane;
      float prod = 1.0f;
      for (int u = 0; u < d; ++u) {
        if (col[32 * u] >= G.nc) break;  // (dummies come last)
        v2c[cell[32 * u]] = prod;        // prefix product (exclusive)
        prod *= post[col[32 * u]];
      }
      const int j = G.row[l];
      const uint32_t sj = (sb[j >> 5] >> (j & 31)) & 1u;
      float P = 0.5f * (1.0f - prod);
      const float eps = 1e-7f;
      const bool clamped = P < eps || P > 1.0f - eps;
      P = fminf(fmaxf(P, eps), 1.0f - eps);
      lsum += (double)(sj ? -logf(P) : -logf(1.0f - P));
      if (backward) {
        // dL/dprod = dL/dP * dP/dprod, with dP/dprod = -1/2
        const float dP = clamped ? 0.0f : (sj ? -1.0f / P : 1.0f / (1.0f - P)) / (float)G.nr;
        const float dprod = -0.5f * dP;
        float suf = 1.0f;
        for (int u = d - 1; u >= 0; --u) {
          if (col[32 * u] >= G.nc) continue;
          const float th = post[col[32 * u]];
          const int c = cell[32 * u];
          v2c[c] = dprod * v2c[c] * suf * 0.5f * (1.0f - th * th);  // contribution to dL/dpost_i
          suf *= th;
        }
      }
    }
#pragma unroll
    for (int off = 16; off; off >>= 1) lsum += __shfl_xor_sync(FULL, lsum, off);
    if (lane == 0) red[warp] = lsum;
    __syncthreads();
    if (tid == 0 && loss_out) {
      double tot = 0.0;
      for (int x = 0; x < nw; ++x) tot += red[x];
      loss_out[smp] = (float)(tot / (double)G.nr);
    }
    if (!backward) continue;
    for (int s = warp; s < G.ncs; s += nw) {  // dL/dpost (its contributions sit in v2c's place)
      float g = 0.0f;
      for (int c = G.coff[s]; c < G.coff[s + 1]; ++c)
        if ((int)(G.cent[32 * c + lane] >> 16) < nrp) g += v2c[32 * c + lane];
      post[32 * s + lane] = g;
    }
    __syncthreads();
    for (int c = tid; c < cells; c += NT) v2c[c] = 0.0f;
    if (tid == 0) post[ncp] = 0.0f;  // the dummy column's
    // ---- adjoint: post holds the gradient into iteration t's posteriors, v2c
    // that into its inputs, and a check's record the two input gradients it
    // sends: gA, gB; their cells; the positions and whether the clip passes ----
    for (int t = G.T; t >= 1; --t) {
      if (t < G.T) {
        if (SEG && t % G.seg == 0)  // the last iteration of a segment gone through next
          recompute_records(G, w, sb, v2c, hist + (size_t)max(t / G.seg - 2, 0) * nrp, t - G.seg, t,
                            hist + (size_t)(G.segs() - 1) * nrp);
        __syncthreads();
        for (int s = warp; s < G.nrs; s += nw) {
          const WRec a = rec[32 * s + lane];
          if (a.pw & 0x1000u) v2c[a.sg & 0xFFFFu] = a.m1;
          if (a.pw & 0x2000u) v2c[a.sg >> 16] = a.m2;
        }
        __syncthreads();
        for (int s = warp; s < G.ncs; s += nw) {
          float g = 0.0f;
          for (int c = 32 * G.coff[s] + lane; c < 32 * G.coff[s + 1]; c += 32) {
            const float x = v2c[c];
            if (x != 0.0f) {
              g += x;
              v2c[c] = 0.0f;
            }
          }
          post[32 * s + lane] = g;
        }
      }
      __syncthreads();
      const float* wt = w + (size_t)(t - 1) * G.ne;
      float* gw = grad_w + (size_t)(t - 1) * G.ne;
      for (int s = warp; s < G.nrs; s += nw) {
        const int r0 = G.roff[s], d = G.roff[s + 1] - r0, l = 32 * s + lane;
        const uint16_t *col = G.rcol + 32 * r0 + lane, *eid = G.reid + 32 * r0 + lane, *cell = G.rcell + 32 * r0 + lane;
        const WRec r = hist[(size_t)(SEG ? G.slot_backward(t) : t - 1) * nrp + l];
        WRec a{0.0f, 0.0f, 0u, 0u};
        if (t < G.T) a = rec[l];
        const int q1 = a.pw & 0x1000u ? (int)(a.pw & 63u) : -1, q2 = a.pw & 0x2000u ? (int)((a.pw >> 6) & 63u) : -1;
        const int p1 = (int)(r.pw & 63u), p2 = (int)((r.pw >> 6) & 63u);
        float g1 = 0.0f, g2 = 0.0f;  // into |v2c| at p1 and p2
#pragma unroll 4
        for (int u = 0; u < d; ++u) {
          float gc = post[col[32 * u]];  // dL/dc2v: the column's less the edge's own
          if (u == q1) gc -= a.m1;
          if (u == q2) gc -= a.m2;
          if (gc != 0.0f) {
            const int e = eid[32 * u];
            const uint32_t sg = rec_sign(r, u);
            atomicAdd(&gw[e], with_sign(grad_scale * gc, sg) * (u == p1 ? r.m2 : r.m1));
            const float gm = with_sign(gc, sg) * wt[e];
            if (u == p1) g2 += gm;
            else g1 += gm;
          }
        }
        // gradient into the inputs at p1 and p2: times their own signs
        const uint32_t par = (r.pw << 19) & 0x80000000u;
        a.m1 = with_sign(g1, rec_sign(r, p1) ^ par);
        a.m2 = with_sign(g2, rec_sign(r, p2) ^ par);
        a.sg = d > 0 ? (uint32_t)cell[32 * min(p1, d - 1)] | ((uint32_t)cell[32 * min(p2, d - 1)] << 16) : 0u;
        a.pw = (r.pw & 0xFFFu) | (r.m1 < G.clip ? 0x1000u : 0u) | (r.m2 < G.clip ? 0x2000u : 0u);
        rec[l] = a;
      }
    }
  }
}

// window-local shots: every window column fires with its prior; the syndrome
// is H_win e over the window's rows (Philox counter word 3 = 1 + window)
__device__ __forceinline__ uint4 philox(uint4 c, uint2 k) {
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

// Window-local samples: every window column fires with its prior (Philox
// word 3 = domain).  Outputs (each optional): the window syndrome [n][rw];
// the same bits placed at rows row0.. of a whole-shot detector vector
// [n][det_words] (zeros elsewhere); the fired columns [n][cw].
__global__ void wms_sample_kernel(WmsGraph G, const uint32_t* __restrict__ thr, unsigned long long seed,
                                  unsigned long long off, long long n, uint32_t domain,
                                  uint32_t* __restrict__ synd, uint32_t* __restrict__ det, int det_words,
                                  int row0, uint32_t* __restrict__ fault, int cw) {
  extern __shared__ uint32_t srow[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const long long s = (long long)blockIdx.x * (blockDim.x >> 5) + wib;
  uint32_t* row = srow + (size_t)wib * G.rw;
  for (int x = lane; x < G.rw; x += 32) row[x] = 0;
  __syncwarp();
  if (s < n) {
    const unsigned long long shot = off + (unsigned long long)s;
    const uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
    for (int g = lane; g < (G.nc + 3) / 4; g += 32) {
      const uint4 u = philox(make_uint4((uint32_t)g, (uint32_t)shot, (uint32_t)(shot >> 32), domain), key);
      const uint32_t uu[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int c = 4 * g + r;
        if (c < G.nc && uu[r] < thr[c]) {
          for (int e = G.col_ptr[c]; e < G.col_ptr[c + 1]; ++e) {
            const int j = G.col_rows[e];
            atomicXor(&row[j >> 5], 1u << (j & 31));
          }
          if (fault) atomicOr(&fault[(size_t)s * cw + (c >> 5)], 1u << (c & 31));
        }
      }
    }
  }
  __syncwarp();
  if (s < n) {
    if (synd)
      for (int x = lane; x < G.rw; x += 32) synd[(size_t)s * G.rw + x] = row[x];
    if (det)
      for (int x = lane; x < det_words; x += 32) {
        // detector bits 32x .. 32x + 31 = window rows 32x - row0 ..
        const int b = 32 * x - row0;
        uint32_t v = 0;
        if (b > -32 && b < G.nr) {
          const int wq = b >= 0 ? (b >> 5) : -1, sh = b & 31;
          const uint32_t lo = (wq >= 0 && wq < G.rw) ? row[wq] : 0u;
          const uint32_t hi = (wq + 1 >= 0 && wq + 1 < G.rw) ? row[wq + 1] : 0u;
          v = sh ? ((lo >> sh) | (hi << (32 - sh))) : lo;
        }
        det[(size_t)s * det_words + x] = v;
      }
  }
}

__global__ void adam_kernel(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, long long n, float lr, float b1, float b2, float eps,
                            float c1, float c2) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.0f - b1) * gi;
  const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

}  // namespace lrn

size_t wms_window_bytes(int ne, int nc, int rw) { return sizeof(float) * (4 * (size_t)ne + 2 * (size_t)nc) + 4 * (size_t)rw; }

size_t wms_smem_bytes(const WmsSlices& G) {
  return sizeof(float) * (32 * (size_t)G.col_cells + 32 + 32 * G.ncs + 32) +
         sizeof(lrn::WRec) * (32 * (size_t)G.nrs + 1) + 4 * (size_t)((G.rw + 3) & ~3) + 32 * sizeof(double) + 16;
}

size_t wms_scratch_per_cta(const WmsSlices& G) { return sizeof(lrn::WRec) * 32 * (size_t)G.nrs * G.records(); }

cudaError_t wms_set_smem(size_t bytes) {
  const cudaError_t e =
      cudaFuncSetAttribute(lrn::wms_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(lrn::wms_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

cudaError_t wms_occupancy(size_t smem, int* blocks) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, lrn::wms_kernel<false>, 256, smem);
}

cudaError_t launch_wms(cudaStream_t st, int grid, size_t smem, const WmsSlices& G, const float* w, const uint32_t* synd,
                       long long n, int backward, float grad_scale, float* grad_w, float* loss, float* post,
                       char* scratch, int* work) {
  const auto kernel = G.seg ? lrn::wms_kernel<true> : lrn::wms_kernel<false>;
  kernel<<<grid, 256, smem, st>>>(G, w, synd, n, backward, grad_scale, grad_w, loss, post, (lrn::WRec*)scratch, work);
  return cudaGetLastError();
}

cudaError_t launch_wms_sample(cudaStream_t st, const WmsGraph& G, const uint32_t* thr, unsigned long long seed,
                              unsigned long long off, long long n, unsigned domain, uint32_t* synd, uint32_t* det,
                              int det_words, int row0, uint32_t* fault, int cw) {
  if (n <= 0) return cudaSuccess;
  if (fault) {
    const cudaError_t e = cudaMemsetAsync(fault, 0, sizeof(uint32_t) * (size_t)n * cw, st);
    if (e != cudaSuccess) return e;
  }
  const int wpb = 8;
  lrn::wms_sample_kernel<<<(unsigned)((n + wpb - 1) / wpb), 32 * wpb, sizeof(uint32_t) * wpb * G.rw, st>>>(
      G, thr, seed, off, n, domain, synd, det, det_words, row0, fault, cw);
  return cudaGetLastError();
}

cudaError_t launch_adam(cudaStream_t st, float* w, const float* g, float* m, float* v, long long n, float lr,
                        float b1, float b2, float eps, int step) {
  if (n <= 0) return cudaSuccess;
  const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
  lrn::adam_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(w, g, m, v, n, lr, b1, b2, eps, c1, c2);
  return cudaGetLastError();
}

}  // namespace qd
