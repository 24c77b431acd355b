// solve32.cu -- FP32 messages + FP64 iterative refinement, and the convergence fix.
//
// The precision messages do not depend on b (eq_prec, eq_prec_message: P_ij =
// -A_ij^2 / P_{i\j}), so they are iterated once per matrix, then frozen.  With
// P frozen, the information-form mean message is linear in the cavity:
//   h_ij = c_ij (h~_i - h_ji),   c_ij = -A_ij / (P~_i - P_ji)       (Algorithm 2),
// and x_i = h~_i / P~_i.  These iterations run in FP32; the only FP64 steps are
// the outer residual r = b - A x and the update x <- x + d, where d is the FP32
// GaBP solution of A d = r.  With a diagonal loading Gamma the inner solves run
// on A + Gamma and the same outer loop is the paper's convergence fix
//   x^(t+1) = x^(t) + (A + Gamma)^{-1} (b - A x^(t)) = (A + Gamma)^{-1}(b + Gamma x^(t))
// (Chapter "Fixing convergence of GaBP", eq:iterative_method).
//
// Recompute form.  Slot e of row i (sender k) keeps its own in-message in one of
// two chains (even / odd rounds).  Round t needs the reverse message i -> k of
// round t-1, which row i itself can recompute from what it held at round t-2:
//   h_{i->k}^{(t-1)} = c_out (h~_i^{(t-2)} - h_{k->i}^{(t-2)}),
//   h_{k->i}^{(t)}   = c_in  (h~_k^{(t-1)} - h_{i->k}^{(t-1)}),
// with c_in = c_ki and c_out = c_ik stored side by side in slot e.  The same
// holds for the precision messages.  Every edge array is then read and written
// in place, coalesced, with no gather or scatter through rev[]; only the node
// values h~_k^{(t-1)} are gathered (they stay in L2).  In exact arithmetic this
// is the synchronous schedule of Algorithm 2; in FP32 it rounds the same way as
// computing h_{i->k}^{(t-1)} once and storing it.
//
// Large graphs of short rows run these rounds on a sliced layout (ks32_*, ensure_sell32), dense matrices on
// arrays of their own (k32_dense), the rest and pinned shapes with L lanes a row (k32_*).
#include "gabp_internal.cuh"
#include "devutil.cuh"
#include "sell64.cuh"

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

namespace gabp {

constexpr int kPrecMaxRounds = 300;  // cap of the FP32 precision phase
constexpr int kUnroll32 = 4;         // default slots per lane whose loads are issued together

// Round-kernel shapes the autotuner chooses from: (lanes per row L, slots per
// lane whose loads are issued together U), packed as L | U << 8.
constexpr int shape_code(int L, int U) { return L | (U << 8); }
constexpr int kShapes[] = {shape_code(1, 4), shape_code(2, 4), shape_code(4, 4), shape_code(8, 4),
                           shape_code(1, 8), shape_code(2, 8), shape_code(4, 8),
                           shape_code(2, 2), shape_code(4, 2), shape_code(8, 2),
                           shape_code(16, 1), shape_code(16, 2)};
template <int V> using IC = std::integral_constant<int, V>;

// The shape a pinned (options.lanes, options.unroll) pair selects, or 0 if the
// library has no such kernel.
int pinned_shape32(int lanes, int unroll) {
  const int L = lanes > 16 ? 16 : lanes;
  const int U = unroll ? unroll : (L >= 16 ? 1 : kUnroll32);
  for (int sc : kShapes)
    if (sc == shape_code(L, U)) return sc;
  return 0;
}

// f(IC<L>, IC<U>) for a shape code (unknown codes map to (4, 4)).
template <typename F>
void with_shape(int code, F &&f) {
  switch (code) {
    case shape_code(1, 4): f(IC<1>{}, IC<4>{}); break;
    case shape_code(2, 4): f(IC<2>{}, IC<4>{}); break;
    case shape_code(8, 4): f(IC<8>{}, IC<4>{}); break;
    case shape_code(1, 8): f(IC<1>{}, IC<8>{}); break;
    case shape_code(2, 8): f(IC<2>{}, IC<8>{}); break;
    case shape_code(4, 8): f(IC<4>{}, IC<8>{}); break;
    case shape_code(2, 2): f(IC<2>{}, IC<2>{}); break;
    case shape_code(4, 2): f(IC<4>{}, IC<2>{}); break;
    case shape_code(8, 2): f(IC<8>{}, IC<2>{}); break;
    case shape_code(16, 1): f(IC<16>{}, IC<1>{}); break;
    case shape_code(16, 2): f(IC<16>{}, IC<2>{}); break;
    default: f(IC<4>{}, IC<4>{}); break;
  }
}

struct Args32 {
  int n;
  int dense;  // complete pattern (a dense matrix): k32_mean derives the sender from the slot
  int ld;     // row length of the dense mean rounds' arrays (0: k32_mean runs the mean rounds)
  float *Cin, *Cout, *Hd;  // [n][ld] coefficients c_in, c_out and stored messages of those rounds
  float *Sp;               // [gridDim][ld] partial column sums
  const int *__restrict__ rp;
  const int *__restrict__ ci;
  const float *__restrict__ av;
  const float *__restrict__ ad;   // diagonal of the matrix the inner solves run on (A + Gamma)
  float *MP0, *MP1;               // precision chains
  float *NP0, *NP1, *NP2;         // P~ ring
  float2 *CF;                     // {c_in, c_out}
  float *invP;
  float *H0, *H1;                 // mean chains
  float *NH0, *NH1, *NH2;         // h~ ring
  const float *rhs;               // FP32 right-hand side of the inner solve
  float2 *NQ0, *NQ1, *NQ2;        // {P~, h~} ring of the joint rounds
  DevCtl *ctl;
  double *partials;
  int ns;                           // slices of the sliced layout (0: row kernels); node arrays by position then
  const int *sp;                    // [ns + 1] first slot of each slice
  cudaGraphConditionalHandle cond;  // while-node condition cleared when the run is decided
  int use_cond;                     // (only inside the device-loop graph)
};

__host__ __device__ __forceinline__ float *ring3(float *a, float *b, float *c, int t) {
  int m = t % 3;
  return m == 0 ? a : (m == 1 ? b : c);
}
__device__ __forceinline__ float2 *ring3(float2 *a, float2 *b, float2 *c, int t) {
  int m = t % 3;
  return m == 0 ? a : (m == 1 ? b : c);
}

// ---------------------------------------------------------------------------- precision phase
// Round t of the precision-only iteration (eq_prec + eq_prec_message, Algorithm 2),
// recompute form.  The run stops once every message has |P^(t) - P^(t-1)| <=
// 2^-s |P^(t)| (s = options.prec_stop_log2, default 16; kept in ctl->tol2bb)
// in two consecutive rounds, on a zero cavity, or at max_iter; a non-finite
// message after round 1 stops it as diverged.  The reciprocals use the fast
// FP32 division (__fdividef, about 2 ulp): the FP32 precision state only has to
// be FP32-accurate, the FP64 refinement absorbs what the frozen coefficients are
// off by (|divisor| >= 2^126 would give 0; such precisions are outside FP32's use).
// FP32 rounding keeps some messages moving by a few ulp forever, so an exact
// stationary point is not waited for: the outer FP64 refinement absorbs what
// the frozen coefficients are off by.
template <int L, int U>
__global__ void __launch_bounds__(kBlock) k32_prec(Args32 a) {
  DevCtl *ctl = a.ctl;
  if (ctl->done) return;
  const int t = ctl->round + 1;
  float *__restrict__ Mc = (t & 1) ? a.MP1 : a.MP0;        // holds t-2, becomes t
  const float *__restrict__ Mo = (t & 1) ? a.MP0 : a.MP1;  // holds t-1
  const float *__restrict__ Pm1 = ring3(a.NP0, a.NP1, a.NP2, t + 2);
  const float *__restrict__ Pm2 = ring3(a.NP0, a.NP1, a.NP2, t + 1);
  float *__restrict__ Pt = ring3(a.NP0, a.NP1, a.NP2, t);
  constexpr int RPW = 32 / L;
  const int lane = threadIdx.x & 31, sl = lane & (L - 1), sw = lane / L;
  const int warp = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * kBlock) >> 5;
  const float thr = (float)ctl->tol2bb;  // 2^-prec_stop_log2
  int bad = 0, moving = 0, nonfinite = 0;
  for (int base = warp * RPW; base < a.n; base += nwarps * RPW) {
    const int i = base + sw;
    float acc = 0.f;
    if (i < a.n) {
      const float Pi2 = t >= 2 ? Pm2[i] : 0.f;
      const int e1 = a.rp[i + 1];
      for (int eb = a.rp[i] + sl; eb < e1; eb += L * U) {
        // all loads of U slots first (memory-level parallelism), then the gathers
        int k[U];
        float A[U], Ps[U], Pp[U], Pk[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int e = eb + u * L;
          if (e < e1) { k[u] = __ldcs(a.ci + e); A[u] = __ldcs(a.av + e); Ps[u] = __ldcs(Mc + e); Pp[u] = __ldcs(Mo + e); }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (eb + u * L < e1) Pk[u] = Pm1[k[u]];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int e = eb + u * L;
          if (e < e1) {
            const float A2 = A[u] * A[u];
            float Pout = 0.f;
            if (t >= 2) {
              const float d1 = Pi2 - Ps[u];
              bad |= (d1 == 0.f);
              Pout = -A2 * __fdividef(1.f, d1);
            }
            const float d2 = Pk[u] - Pout;
            bad |= (d2 == 0.f);
            const float Pn = -A2 * __fdividef(1.f, d2);
            __stcs(Mc + e, Pn);
            acc += Pn;
            moving |= !(fabsf(Pn - Pp[u]) <= thr * fabsf(Pn));  // a NaN counts as moving
            nonfinite |= !isfinite(Pn);
          }
        }
      }
    }
    acc = sub_sum<L>(acc);
    if (i < a.n && sl == 0) {
      const float P = a.ad[i] + acc;
      bad |= (P == 0.f);
      Pt[i] = P;
    }
  }
  double v[3] = {(double)bad, (double)moving, (double)nonfinite}, tot[3];
  block_sum<3>(v);
  if (last_block_reduce<3>(v, a.partials, &ctl->arrive, tot) && threadIdx.x == 0) {
    ctl->round = t;
    ctl->maxrel = tot[1];                      // messages that moved by more than 2^-s
    ctl->stable = tot[1] == 0.0 ? ctl->stable + 1 : 0;
    if (ctl->no_stop) {
      // autotuning run: no decision
    } else if (tot[0] > 0.0) {
      ctl->status = GABP_BREAKDOWN; ctl->iters = t; ctl->result_round = t; ctl->done = 1;
    } else if (tot[2] > 0.0 && t > 1) {
      ctl->status = GABP_DIVERGED; ctl->iters = t; ctl->result_round = t; ctl->done = 1;
    } else if (ctl->stable >= 2) {
      ctl->status = GABP_OK; ctl->iters = t; ctl->result_round = t; ctl->done = 1;
    } else if (t >= ctl->max_iter) {
      ctl->status = GABP_NOT_CONVERGED; ctl->iters = t; ctl->result_round = t; ctl->done = 1;
    }
    ctl->arrive = 0;
    __threadfence();
  }
}

// ---------------------------------------------------------------------------- joint rounds
// Round t of the full FP32 iteration (Algorithm 2: eq_prec_message and
// eq_mean_message for every directed edge, in information form), recompute form
// for both messages.  Slot e = (i, k) keeps the in-messages P_ki, h_ki; the
// reverse messages of round t-1 are recomputed from row i's own round t-2 state:
//   P_ik = -A^2 / (P~_i - P_ki),  h_ik = -A (h~_i - h_ki) / (P~_i - P_ki),
// then  P_ki^t = -A^2 / (P~_k - P_ik),  h_ki^t = -A (h~_k - h_ik) / (P~_k - P_ik)
// with the sender's round t-1 aggregates {P~_k, h~_k} fetched as ONE 8-byte
// gather.  The node aggregates go to the {P~, h~} ring and to the P~ and h~ rings
// the precision-only and frozen-coefficient kernels read, so the run can freeze
// the coefficients at any round T and continue with k32_mean from round T + 1.
// Stop rule: the precision phase's (relative change <= 2^-s in two consecutive
// rounds, zero cavity, max_iter).
__device__ __forceinline__ void joint_decide(const Args32 &a, DevCtl *ctl, int t, const double (&tot)[3]) {
  ctl->round = t;
  ctl->maxrel = tot[1];                      // messages that moved by more than 2^-s
  ctl->stable = tot[1] == 0.0 ? ctl->stable + 1 : 0;
  if (ctl->no_stop) {
    // autotuning run: no decision
  } else if (tot[0] > 0.0) {
    ctl->status = GABP_BREAKDOWN; ctl->iters = t; ctl->result_round = t; ctl->done = 1;
  } else if (tot[2] > 0.0 && t > 1) {
    ctl->status = GABP_DIVERGED; ctl->iters = t; ctl->result_round = t; ctl->done = 1;
  } else if (ctl->stable >= 2) {
    ctl->status = GABP_OK; ctl->iters = t; ctl->result_round = t; ctl->done = 1;
  } else if (t >= ctl->max_iter) {
    ctl->status = GABP_NOT_CONVERGED; ctl->iters = t; ctl->result_round = t; ctl->done = 1;
  }
  if (a.use_cond && ctl->done) cudaGraphSetConditional(a.cond, 0);
  ctl->arrive = 0;
  __threadfence();
}

template <int L, int U>
__global__ void __launch_bounds__(kBlock, 4) k32_joint(Args32 a) {
  DevCtl *ctl = a.ctl;
  if (ctl->done) return;
  const int t = ctl->round + 1;
  float *__restrict__ Mc = (t & 1) ? a.MP1 : a.MP0;        // P chain: holds t-2, becomes t
  const float *__restrict__ Mo = (t & 1) ? a.MP0 : a.MP1;  // P at t-1
  float *__restrict__ Hc = (t & 1) ? a.H1 : a.H0;          // h chain: holds t-2, becomes t
  const float2 *__restrict__ Qm1 = ring3(a.NQ0, a.NQ1, a.NQ2, t + 2);
  const float2 *__restrict__ Qm2 = ring3(a.NQ0, a.NQ1, a.NQ2, t + 1);
  float2 *__restrict__ Qt = ring3(a.NQ0, a.NQ1, a.NQ2, t);
  float *__restrict__ Pt = ring3(a.NP0, a.NP1, a.NP2, t);
  float *__restrict__ Ht = ring3(a.NH0, a.NH1, a.NH2, t);
  constexpr int RPW = 32 / L;
  const int lane = threadIdx.x & 31, sl = lane & (L - 1), sw = lane / L;
  const int warp = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * kBlock) >> 5;
  const float thr = (float)ctl->tol2bb;  // 2^-prec_stop_log2
  int bad = 0, moving = 0, nonfinite = 0;
  for (int base = warp * RPW; base < a.n; base += nwarps * RPW) {
    const int i = base + sw;
    float accP = 0.f, accH = 0.f, ad_i = 0.f, rhs_i = 0.f;
    if (i < a.n) {
      const float2 q2 = t >= 2 ? Qm2[i] : make_float2(0.f, 0.f);
      ad_i = a.ad[i];  // requested before the slots (latency overlap)
      rhs_i = a.rhs[i];
      const int e1 = a.rp[i + 1];
      for (int eb = a.rp[i] + sl; eb < e1; eb += L * U) {
        int k[U];
        float A[U], Ps[U], Pp[U], hs[U];
        float2 qk[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int e = eb + u * L;
          if (e < e1) {
            k[u] = __ldcs(a.ci + e); A[u] = __ldcs(a.av + e);
            Ps[u] = __ldcs(Mc + e); Pp[u] = __ldcs(Mo + e); hs[u] = __ldcs(Hc + e);
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (eb + u * L < e1) qk[u] = __ldcg(Qm1 + k[u]);  // random gather, L2 only
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int e = eb + u * L;
          if (e < e1) {
            float Pout = 0.f, hout = 0.f;
            if (t >= 2) {  // message i -> k of round t-1
              const float d1 = q2.x - Ps[u];
              bad |= (d1 == 0.f);
              const float r1 = __fdividef(1.f, d1);
              Pout = -A[u] * A[u] * r1;
              hout = -A[u] * (q2.y - hs[u]) * r1;
            }
            const float d2 = qk[u].x - Pout;  // message k -> i of round t
            bad |= (d2 == 0.f);
            const float r2 = __fdividef(1.f, d2);
            const float Pn = -A[u] * A[u] * r2;
            const float hn = -A[u] * (qk[u].y - hout) * r2;
            __stcs(Mc + e, Pn);
            __stcs(Hc + e, hn);
            accP += Pn;
            accH += hn;
            moving |= !(fabsf(Pn - Pp[u]) <= thr * fabsf(Pn));  // a NaN counts as moving
            nonfinite |= !isfinite(Pn);
          }
        }
      }
    }
    accP = sub_sum<L>(accP);
    accH = sub_sum<L>(accH);
    if (i < a.n && sl == 0) {
      const float P = ad_i + accP, hh = rhs_i + accH;
      bad |= (P == 0.f);
      Qt[i] = make_float2(P, hh);
      Pt[i] = P;
      Ht[i] = hh;
    }
  }
  double v[3] = {(double)bad, (double)moving, (double)nonfinite}, tot[3];
  block_sum<3>(v);
  if (last_block_reduce<3>(v, a.partials, &ctl->arrive, tot) && threadIdx.x == 0) joint_decide(a, ctl, t, tot);
}

// The same on the sliced layout (ensure_sell32): lane by row.  The sums are those of the row kernel with 4 lanes a
// row, bit for bit: systems whose FP32 rounds go one way or the other by their rounding (indefinite augmented ones of
// least squares) go the same way on both.  U slots a lane in flight and the registers for them
// (whole 2^20-row solves in us): U 4 at 3 blocks 2396, 3 at 4 2382, 2 at 5 2430, 4 at 4 (spills) 2535, 1 at 8 2786.
// 130 us a round at 16.8 M slots, 157 with the row kernel (the streams and gathers alone, without rows: 101).
__global__ void __launch_bounds__(kBlock, 3) ks32_joint(Args32 a) {
  constexpr int U = 4;  // slots a lane in flight
  DevCtl *ctl = a.ctl;
  if (ctl->done) return;
  const int t = ctl->round + 1;
  float *Mc = (t & 1) ? a.MP1 : a.MP0;        // P chain: holds t-2, becomes t
  const float *Mo = (t & 1) ? a.MP0 : a.MP1;  // P at t-1
  float *Hc = (t & 1) ? a.H1 : a.H0;          // h chain: holds t-2, becomes t
  const float2 *__restrict__ Qm1 = ring3(a.NQ0, a.NQ1, a.NQ2, t + 2);
  const float2 *__restrict__ Qm2 = ring3(a.NQ0, a.NQ1, a.NQ2, t + 1);
  float2 *__restrict__ Qt = ring3(a.NQ0, a.NQ1, a.NQ2, t);
  float *__restrict__ Pt = ring3(a.NP0, a.NP1, a.NP2, t);
  float *__restrict__ Ht = ring3(a.NH0, a.NH1, a.NH2, t);
  const WarpPos w = warp_pos();
  const float thr = (float)ctl->tol2bb;  // 2^-prec_stop_log2
  int bad = 0, moving = 0, nonfinite = 0;
  for (int m = 0; m * (int64_t)w.nwarps < a.ns; ++m) {
    const int s = pass_slice(w, m);
    if (s >= a.ns) continue;
    const int p = 32 * s + w.lane, q1 = a.sp[s + 1];
    const float2 q2 = t >= 2 ? Qm2[p] : make_float2(0.f, 0.f);
    const float ad = a.ad[p], rhs = a.rhs[p];
    float aP[4] = {}, aH[4] = {};  // as by 4 lanes a row
    for (int qb = a.sp[s] + w.lane; qb < q1; qb += 32 * U) {
      int k[U];
      float A[U], Ps[U], Pp[U], hs[U];
      float2 qk[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int q = qb + 32 * u;
        k[u] = -1;
        if (q < q1) {
          k[u] = __ldcs(a.ci + q); A[u] = __ldcs(a.av + q);
          Ps[u] = __ldcs(Mc + q); Pp[u] = __ldcs(Mo + q); hs[u] = __ldcs(Hc + q);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (k[u] >= 0) qk[u] = __ldcg(Qm1 + k[u]);  // random gather, L2 only
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (k[u] >= 0) {
          float Pout = 0.f, hout = 0.f;
          if (t >= 2) {  // message i -> k of round t-1
            const float d1 = q2.x - Ps[u];
            bad |= (d1 == 0.f);
            const float r1 = __fdividef(1.f, d1);
            Pout = -A[u] * A[u] * r1;
            hout = -A[u] * (q2.y - hs[u]) * r1;
          }
          const float d2 = qk[u].x - Pout;  // message k -> i of round t
          bad |= (d2 == 0.f);
          const float r2 = __fdividef(1.f, d2);
          const float Pn = -A[u] * A[u] * r2;
          const float hn = -A[u] * (qk[u].y - hout) * r2;
          __stcs(Mc + qb + 32 * u, Pn);
          __stcs(Hc + qb + 32 * u, hn);
          aP[u] += Pn;
          aH[u] += hn;
          moving |= !(fabsf(Pn - Pp[u]) <= thr * fabsf(Pn));  // a NaN counts as moving
          nonfinite |= !isfinite(Pn);
        }
    }
    const float P = ad + ((aP[0] + aP[2]) + (aP[1] + aP[3])), hh = rhs + ((aH[0] + aH[2]) + (aH[1] + aH[3]));
    bad |= (P == 0.f);
    Qt[p] = make_float2(P, hh);
    Pt[p] = P;
    Ht[p] = hh;
  }
  double v[3] = {(double)bad, (double)moving, (double)nonfinite}, tot[3];
  block_sum<3>(v);
  if (last_block_reduce<3>(v, a.partials, &ctl->arrive, tot) && threadIdx.x == 0) joint_decide(a, ctl, t, tot);
}

// round-0 state of the joint rounds: zero messages, {P~, h~} = {A_ii (+ Gamma_ii), r}
__global__ void k32_joint_init(int n, const float *__restrict__ ad, const float *__restrict__ rhs, float2 *nq0,
                               float *np0) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    nq0[i] = make_float2(ad[i], rhs[i]);
    np0[i] = ad[i];
  }
}

// Freeze: c_out = c_ik = -A / (P~_i - P_ki), P_ik = c_out A, c_in = c_ki = -A / (P~_k - P_ik),
// 1/P~_i.  Uses round T's precision state.
template <int L>
__global__ void __launch_bounds__(kBlock) k32_coef(Args32 a, int T) {
  const float *__restrict__ Ms = (T & 1) ? a.MP1 : a.MP0;
  const float *__restrict__ PT = ring3(a.NP0, a.NP1, a.NP2, T);
  constexpr int RPW = 32 / L;
  const int lane = threadIdx.x & 31, sl = lane & (L - 1), sw = lane / L;
  const int warp = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * kBlock) >> 5;
  for (int base = warp * RPW; base < a.n; base += nwarps * RPW) {
    const int i = base + sw;
    if (i >= a.n) continue;
    const float Pi = PT[i];
    for (int e = a.rp[i] + sl; e < a.rp[i + 1]; e += L) {
      const int k = a.ci[e];
      const float A = a.av[e];
      const float cout = -A / (Pi - Ms[e]);
      const float Pout = cout * A;
      const float cin = -A / (PT[k] - Pout);
      a.CF[e] = make_float2(cin, cout);
    }
    if (sl == 0) a.invP[i] = 1.f / Pi;
  }
}

// The decision after mean round t, from the squared norms tot of its update and iterate.
__device__ __forceinline__ void mean_decide(const Args32 &a, DevCtl *ctl, int t, const double (&tot)[2]) {
  ctl->round = t;
  ctl->rr = tot[0];
  ctl->xx = tot[1];
  if (ctl->no_stop) {
    // autotuning run: no decision
  } else if (!isfinite(tot[0]) || !isfinite(tot[1])) {
    ctl->status = GABP_DIVERGED; ctl->iters = t; ctl->result_round = t; ctl->done = 1;
  } else if (t >= 2 && tot[0] <= ctl->tol2bb * tot[1]) {
    ctl->status = GABP_OK; ctl->iters = t; ctl->result_round = t; ctl->done = 1;
  } else if (t >= ctl->max_iter) {
    ctl->status = GABP_NOT_CONVERGED; ctl->iters = t; ctl->result_round = t; ctl->done = 1;
  }
  if (a.use_cond && ctl->done) cudaGraphSetConditional(a.cond, 0);
  ctl->arrive = 0;
  __threadfence();
}

// ---------------------------------------------------------------------------- mean phase, one RHS
// Round t of the frozen-precision mean iteration (recompute form).  The inner
// solve stops when ||x^(t) - x^(t-1)|| <= inner_tol ||x^(t)|| (node-local
// quantities, no extra edge traffic) or at max_iter.
template <int L, int U, bool DENSE = false>
__global__ void __launch_bounds__(kBlock) k32_mean(Args32 a) {
  DevCtl *ctl = a.ctl;
  if (ctl->done) return;
  const int t = ctl->round + 1;
  float *__restrict__ Hc = (t & 1) ? a.H1 : a.H0;  // holds t-2, becomes t
  const float *__restrict__ Hm1 = ring3(a.NH0, a.NH1, a.NH2, t + 2);
  const float *__restrict__ Hm2 = ring3(a.NH0, a.NH1, a.NH2, t + 1);
  float *__restrict__ Ht = ring3(a.NH0, a.NH1, a.NH2, t);
  constexpr int RPW = 32 / L;
  const int lane = threadIdx.x & 31, sl = lane & (L - 1), sw = lane / L;
  const int warp = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * kBlock) >> 5;
  float dxx = 0.f, xx = 0.f;  // per-thread partial sums stay in FP32 (the FP64 pipe is narrow)
  for (int base = warp * RPW; base < a.n; base += nwarps * RPW) {
    const int i = base + sw;
    float acc = 0.f, rhs_i = 0.f, ip = 0.f, hprev = 0.f;
    if (i < a.n) {
      // the row's own values are requested before its slots, so that their latency overlaps the slot loads
      const float hi2 = t >= 2 ? Hm2[i] : 0.f;
      rhs_i = a.rhs[i];
      ip = a.invP[i];
      hprev = Hm1[i];
      const int e0 = a.rp[i], e1 = a.rp[i + 1];
      for (int eb = e0 + sl; eb < e1; eb += L * U) {
        int k[U];
        float2 cf[U];
        float hs[U], hk[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int e = eb + u * L;
          if (e < e1) {
            // a complete pattern: slot p of row i holds column p + (p >= i), no column stream
            k[u] = DENSE ? (e - e0) + (e - e0 >= i) : __ldcs(a.ci + e);
            cf[u] = __ldcs(a.CF + e);
            hs[u] = __ldcs(Hc + e);
          }
        }
        // random gathers bypass L1 (no reuse there), which keeps L1 for the slot streams' sectors; a
        // complete pattern reads the aggregates in column order, the same vector in every row: L1
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (eb + u * L < e1) hk[u] = DENSE ? __ldg(Hm1 + k[u]) : __ldcg(Hm1 + k[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int e = eb + u * L;
          if (e < e1) {
            const float hout = t >= 2 ? cf[u].y * (hi2 - hs[u]) : 0.f;  // message i -> k at t-1
            const float hn = cf[u].x * (hk[u] - hout);                  // message k -> i at t
            __stcs(Hc + e, hn);
            acc += hn;
          }
        }
      }
    }
    acc = sub_sum<L>(acc);
    if (i < a.n && sl == 0) {
      const float hnew = rhs_i + acc;
      Ht[i] = hnew;
      const float x = hnew * ip, dx = (hnew - hprev) * ip;
      dxx = fmaf(dx, dx, dxx);
      xx = fmaf(x, x, xx);
    }
  }
  double v[2] = {(double)dxx, (double)xx}, tot[2];
  block_sum<2>(v);
  if (last_block_reduce<2>(v, a.partials, &ctl->arrive, tot) && threadIdx.x == 0) {
    mean_decide(a, ctl, t, tot);
  }
}

// The same on the sliced layout (ensure_sell32): lane by row.  95 us a round at 16.8 M slots, 117 with the row
// kernel (the streams and gathers alone, without rows: 86).
__global__ void __launch_bounds__(kBlock, 4) ks32_mean(Args32 a) {
  constexpr int U = 4;  // slots a lane in flight
  DevCtl *ctl = a.ctl;
  if (ctl->done) return;
  const int t = ctl->round + 1;
  float *Hc = (t & 1) ? a.H1 : a.H0;  // holds t-2, becomes t
  const float *__restrict__ Hm1 = ring3(a.NH0, a.NH1, a.NH2, t + 2);
  const float *__restrict__ Hm2 = ring3(a.NH0, a.NH1, a.NH2, t + 1);
  float *__restrict__ Ht = ring3(a.NH0, a.NH1, a.NH2, t);
  const WarpPos w = warp_pos();
  float dxx = 0.f, xx = 0.f;
  for (int m = 0; m * (int64_t)w.nwarps < a.ns; ++m) {
    const int s = pass_slice(w, m);
    if (s >= a.ns) continue;
    const int p = 32 * s + w.lane, q1 = a.sp[s + 1];
    const float hi2 = t >= 2 ? Hm2[p] : 0.f, rhs = a.rhs[p], ip = a.invP[p], hprev = Hm1[p];
    float acc[4] = {};  // as by 4 lanes a row
    for (int qb = a.sp[s] + w.lane; qb < q1; qb += 32 * U) {
      int k[U];
      float2 cf[U];
      float hs[U], hk[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int q = qb + 32 * u;
        k[u] = -1;
        if (q < q1) { k[u] = __ldcs(a.ci + q); cf[u] = __ldcs(a.CF + q); hs[u] = __ldcs(Hc + q); }
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (k[u] >= 0) hk[u] = __ldcg(Hm1 + k[u]);  // random gather, L2 only
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (k[u] >= 0) {
          const float hout = t >= 2 ? cf[u].y * (hi2 - hs[u]) : 0.f;  // message i -> k at t-1
          const float hn = cf[u].x * (hk[u] - hout);                  // message k -> i at t
          __stcs(Hc + qb + 32 * u, hn);
          acc[u] += hn;
        }
    }
    const float hnew = rhs + ((acc[0] + acc[2]) + (acc[1] + acc[3]));
    Ht[p] = hnew;
    const float x = hnew * ip, dx = (hnew - hprev) * ip;
    dxx = fmaf(dx, dx, dxx);
    xx = fmaf(x, x, xx);
  }
  double v[2] = {(double)dxx, (double)xx}, tot[2];
  block_sum<2>(v);
  if (last_block_reduce<2>(v, a.partials, &ctl->arrive, tot) && threadIdx.x == 0) mean_decide(a, ctl, t, tot);
}

// ---------------------------------------------------------------------------- mean phase, dense matrix
// Mean rounds of a complete pattern on full n x ld arrays (column k of row i at i ld + k; the diagonal
// and the padding columns hold zeros, which make zero messages).  With every slot (i, k) come c_in =
// c_ki and c_out = c_ik, so that what a column of the matrix sends needs no transposed access:
//   write rounds     as k32_mean (recompute form): message k -> i of round t into slot (i, k); on the
//                    way column k collects S_k = sum_i c_ik h_{k->i}^{(t)}, the messages' part of what
//                    node k will receive next;
//   product rounds   node i receives sum_k c_ki (h~_k^{(t)} - h_{i->k}^{(t)}) = sum_k c_ki h~_k^{(t)} - S_i:
//                    a matrix-vector product with c_in alone, no message read or written.
// The two alternate, so a pair of rounds moves 20 bytes a slot where k32_mean moves 32 (both
// coefficients, message read and write, in every round).  HBM bounds both: 8192 points, 162 us a write
// round (158 at the measured copy rate) and 50 us a product round (39), against 237 us with k32_mean.
// A CTA owns a range of rows, 4 at a time; thread x owns columns 4 x, 4 x + 4 kBlock, ..., whose sums S
// it keeps in shared memory; the CTAs' sums go to Sp and are added in CTA order.
constexpr int kDenseRows = 4;  // rows whose loads are issued together
// Smallest dense matrix of these rounds; below, the launches bound either.  Whole solves, k32_mean / these:
// 300 points 3.0 / 2.6 ms, 800 4.4 / 3.0, 2000 9.4 / 4.5, 4096 24.5 / 9.7, 8192 54.3 / 27.9.
constexpr int kDenseMin = 256;

__device__ __forceinline__ int dense_group0(int n, int b, int nb) {  // first row group of CTA b
  return (int)((int64_t)((n + kDenseRows - 1) / kDenseRows) * b / nb);
}

// c_in, c_out and, for an inner solve that starts from the joint rounds' state, the messages of its start
// round from the row-CSR arrays; zeros on the diagonal and in the padding.
__global__ void __launch_bounds__(kBlock) k32_dense_pack(Args32 a, int with_h) {
  constexpr int U = 4;  // columns a thread whose loads are issued together
  const float *__restrict__ Hs = (a.ctl->start & 1) ? a.H1 : a.H0;
  for (int i = blockIdx.x; i < a.n; i += gridDim.x) {
    const int64_t e0 = (int64_t)i * (a.n - 1), o = (int64_t)i * a.ld;
    for (int k0 = threadIdx.x; k0 < a.ld; k0 += U * kBlock) {
      float2 cf[U];
      float hs[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int k = k0 + u * kBlock;
        const bool in = k < a.n && k != i;
        const int64_t e = e0 + k - (k > i);
        cf[u] = in ? __ldcs(a.CF + e) : make_float2(0.f, 0.f);
        hs[u] = in && with_h ? __ldcs(Hs + e) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int k = k0 + u * kBlock;
        if (k >= a.ld) break;
        __stcs(a.Cin + o + k, cf[u].x);
        __stcs(a.Cout + o + k, cf[u].y);
        if (with_h) __stcs(a.Hd + o + k, hs[u]);
      }
    }
  }
}

// The 4 rows from i0 of a write round: row sums into acc, column sums into cs (shared).  ZERO: the stored
// messages are the zero ones a run starts from (not read).
template <bool ZERO>
__device__ __forceinline__ void dense_write_rows(const Args32 &a, int i0, const float *__restrict__ Hm1,
                                                 const float *__restrict__ Hm2, float *cs, float (&acc)[kDenseRows]) {
  float h2[kDenseRows];
#pragma unroll
  for (int r = 0; r < kDenseRows; ++r) h2[r] = Hm2[min(i0 + r, a.n - 1)];
  for (int c = 4 * threadIdx.x; c < a.ld; c += 4 * kBlock) {
    float4 ci[kDenseRows], co[kDenseRows], hs[kDenseRows];
#pragma unroll
    for (int r = 0; r < kDenseRows; ++r) {
      const int64_t o = (int64_t)min(i0 + r, a.n - 1) * a.ld + c;
      ci[r] = __ldcs(reinterpret_cast<const float4 *>(a.Cin + o));
      co[r] = __ldcs(reinterpret_cast<const float4 *>(a.Cout + o));
      hs[r] = ZERO ? make_float4(0.f, 0.f, 0.f, 0.f) : __ldcs(reinterpret_cast<const float4 *>(a.Hd + o));
    }
    const float4 hk = *reinterpret_cast<const float4 *>(Hm1 + c);
    float4 s = *reinterpret_cast<const float4 *>(cs + c);
#pragma unroll
    for (int r = 0; r < kDenseRows; ++r) {
      if (i0 + r >= a.n) break;
      float4 hn;
      hn.x = ci[r].x * (hk.x - co[r].x * (h2[r] - hs[r].x));
      hn.y = ci[r].y * (hk.y - co[r].y * (h2[r] - hs[r].y));
      hn.z = ci[r].z * (hk.z - co[r].z * (h2[r] - hs[r].z));
      hn.w = ci[r].w * (hk.w - co[r].w * (h2[r] - hs[r].w));
      __stcs(reinterpret_cast<float4 *>(a.Hd + (int64_t)(i0 + r) * a.ld + c), hn);
      acc[r] += (hn.x + hn.y) + (hn.z + hn.w);
      s.x = fmaf(co[r].x, hn.x, s.x);
      s.y = fmaf(co[r].y, hn.y, s.y);
      s.z = fmaf(co[r].z, hn.z, s.z);
      s.w = fmaf(co[r].w, hn.w, s.w);
    }
    *reinterpret_cast<float4 *>(cs + c) = s;
  }
}

// The 4 rows from i0 of a product round.
__device__ __forceinline__ void dense_product_rows(const Args32 &a, int i0, const float *__restrict__ Hm1,
                                                   float (&acc)[kDenseRows]) {
  for (int c = 4 * threadIdx.x; c < a.ld; c += 4 * kBlock) {
    float4 ci[kDenseRows];
#pragma unroll
    for (int r = 0; r < kDenseRows; ++r)
      ci[r] = __ldcs(reinterpret_cast<const float4 *>(a.Cin + (int64_t)min(i0 + r, a.n - 1) * a.ld + c));
    const float4 hk = *reinterpret_cast<const float4 *>(Hm1 + c);
#pragma unroll
    for (int r = 0; r < kDenseRows; ++r)
      acc[r] += fmaf(ci[r].x, hk.x, ci[r].y * hk.y) + fmaf(ci[r].z, hk.z, ci[r].w * hk.w);
  }
}

__global__ void __launch_bounds__(kBlock, 2) k32_dense(Args32 a) {
  DevCtl *ctl = a.ctl;
  if (ctl->done) return;
  extern __shared__ __align__(16) float cs[];  // [ld] column sums of this CTA's rows
  __shared__ float red[kDenseRows][kBlock / 32];
  __shared__ float sfrom[kBlock / 32][32];
  const int t = ctl->round + 1, start = ctl->start;
  const bool write = ((t ^ start) & 1) == 0;
  const float *__restrict__ Hm1 = ring3(a.NH0, a.NH1, a.NH2, t + 2);
  const float *__restrict__ Hm2 = ring3(a.NH0, a.NH1, a.NH2, t + 1);
  float *__restrict__ Ht = ring3(a.NH0, a.NH1, a.NH2, t);
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int g0 = dense_group0(a.n, blockIdx.x, gridDim.x), g1 = dense_group0(a.n, blockIdx.x + 1, gridDim.x);
  if (write)
    for (int c = threadIdx.x; c < a.ld; c += kBlock) cs[c] = 0.f;  // each thread clears others' columns too
  __syncthreads();
  float dxx = 0.f, xx = 0.f;
  for (int g = g0; g < g1; ++g) {
    const int i0 = g * kDenseRows;
    float acc[kDenseRows] = {};
    if (!write) {
      dense_product_rows(a, i0, Hm1, acc);
      // S of every eighth group of 32 rows: lane = row, the warps share the CTAs' sums
      if (t > 1 && ((g - g0) & 7) == 0) {
        float sv = 0.f;
        if (i0 + lane < a.ld)
          for (int b = wib; b < (int)gridDim.x; b += kBlock / 32) sv += __ldcg(a.Sp + (int64_t)b * a.ld + i0 + lane);
        __syncthreads();
        sfrom[wib][lane] = sv;
      }
    } else if (t == 2 && start == 0) {
      dense_write_rows<true>(a, i0, Hm1, Hm2, cs, acc);
    } else {
      dense_write_rows<false>(a, i0, Hm1, Hm2, cs, acc);
    }
#pragma unroll
    for (int r = 0; r < kDenseRows; ++r) {
      const float v = warp_sum(acc[r]);
      if (lane == 0) red[r][wib] = v;
    }
    __syncthreads();
    if (threadIdx.x < kDenseRows && i0 + (int)threadIdx.x < a.n) {
      const int i = i0 + threadIdx.x;
      float v = 0.f;
#pragma unroll
      for (int q = 0; q < kBlock / 32; ++q) v += red[threadIdx.x][q];
      if (!write && t > 1) {
        float sv = 0.f;
#pragma unroll
        for (int q = 0; q < kBlock / 32; ++q) sv += sfrom[q][kDenseRows * ((g - g0) & 7) + threadIdx.x];
        v -= sv;
      }
      const float hnew = a.rhs[i] + v, ip = a.invP[i];
      Ht[i] = hnew;
      const float x = hnew * ip, dx = (hnew - Hm1[i]) * ip;
      dxx = fmaf(dx, dx, dxx);
      xx = fmaf(x, x, xx);
    }
    __syncthreads();
  }
  if (write)
    for (int c = 4 * threadIdx.x; c < a.ld; c += 4 * kBlock)
      *reinterpret_cast<float4 *>(a.Sp + (int64_t)blockIdx.x * a.ld + c) = *reinterpret_cast<const float4 *>(cs + c);
  double v[2] = {(double)dxx, (double)xx}, tot[2];
  block_sum<2>(v);
  if (last_block_reduce<2>(v, a.partials, &ctl->arrive, tot) && threadIdx.x == 0) mean_decide(a, ctl, t, tot);
}

// ---------------------------------------------------------------------------- coefficient freeze
// The first frozen-coefficient mean round after the joint rounds, fused with the
// freeze: from round T's precision state ({P~, h~} ring and P chain) it writes
//   c_out = c_ik = -A / (P~_i - P_ki),  c_in = c_ki = -A / (P~_k - c_out A),  1/P~_i
// and uses them at once for mean round T + 1, the sender's {P~_k, h~_k} coming
// from ONE 8-byte gather (the separate freeze pass would re-read every slot and
// gather P~_k).  Same arithmetic as k32_coef followed by k32_mean.  If the mean
// solve is already decided (T reached the inner cap) only the coefficients and
// 1/P~ are written.
template <int L, int U>
__global__ void __launch_bounds__(kBlock) k32_freeze(Args32 a) {
  DevCtl *ctl = a.ctl;
  const bool coef_only = ctl->done;
  const int T = ctl->round, t = T + 1;
  const float *__restrict__ Ms = (T & 1) ? a.MP1 : a.MP0;  // P_ki of round T
  const float2 *__restrict__ QT = ring3(a.NQ0, a.NQ1, a.NQ2, T);
  float *__restrict__ Hc = (t & 1) ? a.H1 : a.H0;  // holds t-2, becomes t
  const float *__restrict__ Hm2 = ring3(a.NH0, a.NH1, a.NH2, t + 1);
  float *__restrict__ Ht = ring3(a.NH0, a.NH1, a.NH2, t);
  constexpr int RPW = 32 / L;
  const int lane = threadIdx.x & 31, sl = lane & (L - 1), sw = lane / L;
  const int warp = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * kBlock) >> 5;
  float dxx = 0.f, xx = 0.f;
  for (int base = warp * RPW; base < a.n; base += nwarps * RPW) {
    const int i = base + sw;
    float acc = 0.f;
    float2 qi = make_float2(1.f, 0.f);
    float rhs_i = 0.f;
    if (i < a.n) {
      qi = QT[i];
      const float hi2 = t >= 2 ? Hm2[i] : 0.f;
      rhs_i = a.rhs[i];  // requested before the slots (latency overlap)
      const int e1 = a.rp[i + 1];
      for (int eb = a.rp[i] + sl; eb < e1; eb += L * U) {
        int k[U];
        float A[U], Ps[U], hs[U];
        float2 qk[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int e = eb + u * L;
          if (e < e1) { k[u] = __ldcs(a.ci + e); A[u] = __ldcs(a.av + e); Ps[u] = __ldcs(Ms + e); hs[u] = __ldcs(Hc + e); }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (eb + u * L < e1) qk[u] = __ldcg(QT + k[u]);  // random gather, L2 only
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int e = eb + u * L;
          if (e < e1) {
            const float cout = -A[u] / (qi.x - Ps[u]);
            const float Pout = cout * A[u];
            const float cin = -A[u] / (qk[u].x - Pout);
            a.CF[e] = make_float2(cin, cout);
            if (!coef_only) {
              const float hout = t >= 2 ? cout * (hi2 - hs[u]) : 0.f;  // message i -> k at t-1
              const float hn = cin * (qk[u].y - hout);                 // message k -> i at t
              __stcs(Hc + e, hn);
              acc += hn;
            }
          }
        }
      }
    }
    acc = sub_sum<L>(acc);
    if (i < a.n && sl == 0) {
      const float ip = 1.f / qi.x;
      a.invP[i] = ip;
      if (!coef_only) {
        const float hnew = rhs_i + acc;
        Ht[i] = hnew;
        const float x = hnew * ip, dx = (hnew - qi.y) * ip;
        dxx = fmaf(dx, dx, dxx);
        xx = fmaf(x, x, xx);
      }
    }
  }
  if (coef_only) return;
  double v[2] = {(double)dxx, (double)xx}, tot[2];
  block_sum<2>(v);
  if (last_block_reduce<2>(v, a.partials, &ctl->arrive, tot) && threadIdx.x == 0) mean_decide(a, ctl, t, tot);
}

// The same on the sliced layout (118 us at 16.8 M slots, 158 with the row kernel).
__global__ void __launch_bounds__(kBlock, 4) ks32_freeze(Args32 a) {
  constexpr int U = 4;  // slots a lane in flight
  DevCtl *ctl = a.ctl;
  const bool coef_only = ctl->done;
  const int T = ctl->round, t = T + 1;
  const float *__restrict__ Ms = (T & 1) ? a.MP1 : a.MP0;  // P_ki of round T
  const float2 *__restrict__ QT = ring3(a.NQ0, a.NQ1, a.NQ2, T);
  float *Hc = (t & 1) ? a.H1 : a.H0;  // holds t-2, becomes t
  const float *__restrict__ Hm2 = ring3(a.NH0, a.NH1, a.NH2, t + 1);
  float *__restrict__ Ht = ring3(a.NH0, a.NH1, a.NH2, t);
  const WarpPos w = warp_pos();
  float dxx = 0.f, xx = 0.f;
  for (int m = 0; m * (int64_t)w.nwarps < a.ns; ++m) {
    const int s = pass_slice(w, m);
    if (s >= a.ns) continue;
    const int p = 32 * s + w.lane, q1 = a.sp[s + 1];
    const float2 qi = QT[p];
    const float hi2 = t >= 2 ? Hm2[p] : 0.f, rhs = a.rhs[p];
    float acc[4] = {};  // as by 4 lanes a row
    for (int qb = a.sp[s] + w.lane; qb < q1; qb += 32 * U) {
      int k[U];
      float A[U], Ps[U], hs[U];
      float2 qk[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int q = qb + 32 * u;
        k[u] = -1;
        if (q < q1) { k[u] = __ldcs(a.ci + q); A[u] = __ldcs(a.av + q); Ps[u] = __ldcs(Ms + q); hs[u] = __ldcs(Hc + q); }
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (k[u] >= 0) qk[u] = __ldcg(QT + k[u]);  // random gather, L2 only
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (k[u] >= 0) {
          const float cout = -A[u] / (qi.x - Ps[u]);
          const float Pout = cout * A[u];
          const float cin = -A[u] / (qk[u].x - Pout);
          a.CF[qb + 32 * u] = make_float2(cin, cout);
          if (!coef_only) {
            const float hout = t >= 2 ? cout * (hi2 - hs[u]) : 0.f;  // message i -> k at t-1
            const float hn = cin * (qk[u].y - hout);                 // message k -> i at t
            __stcs(Hc + qb + 32 * u, hn);
            acc[u] += hn;
          }
        }
    }
    const float ip = 1.f / qi.x;
    a.invP[p] = ip;
    if (!coef_only) {
      const float hnew = rhs + ((acc[0] + acc[2]) + (acc[1] + acc[3]));
      Ht[p] = hnew;
      const float x = hnew * ip, dx = (hnew - qi.y) * ip;
      dxx = fmaf(dx, dx, dxx);
      xx = fmaf(x, x, xx);
    }
  }
  if (coef_only) return;
  double v[2] = {(double)dxx, (double)xx}, tot[2];
  block_sum<2>(v);
  if (last_block_reduce<2>(v, a.partials, &ctl->arrive, tot) && threadIdx.x == 0) mean_decide(a, ctl, t, tot);
}

// ---------------------------------------------------------------------------- FP64 outer steps
// r = b - A x over the full CSR (diagonal included), in FP64; the FP32 copy of r
// seeds the next inner solve (its round-0 aggregate h~^(0) = r and its RHS).
template <int L>
__global__ void __launch_bounds__(kBlock) k64_residual(int n, const int *__restrict__ rowptr,
                                                       const int *__restrict__ col, const double *__restrict__ val,
                                                       const double *__restrict__ b, const double *__restrict__ x,
                                                       float *__restrict__ rhs32, float *__restrict__ nh0,
                                                       DevCtl *ctl, double *partials, int set_bb,
                                                       const int *__restrict__ pos, const int *skip = nullptr,
                                                       int x_zero = 0) {
  if (skip && *skip) return;  // device-loop graph: the loop already stopped
  constexpr int RPW = 32 / L;
  const int lane = threadIdx.x & 31, sl = lane & (L - 1), sw = lane / L;
  const int warp = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * kBlock) >> 5;
  constexpr int U = 4;  // entries per lane whose loads are issued together
  double rr = 0.0;
  for (int base = warp * RPW; base < n; base += nwarps * RPW) {
    const int i = base + sw;
    double ax = 0.0, bi = 0.0;
    if (i < n) {
      bi = b[i];  // requested before the row's entries (latency overlap)
      if (!x_zero) {  // x = 0 (the first residual): r = b exactly, no product needed
        const int p1 = rowptr[i + 1];
        for (int pb = rowptr[i] + sl; pb < p1; pb += L * U) {
          int c[U];
          double v[U], xc[U];
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (pb + u * L < p1) { c[u] = __ldcs(col + pb + u * L); v[u] = __ldcs(val + pb + u * L); }
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (pb + u * L < p1) xc[u] = __ldcg(x + c[u]);  // random gather, L2 only
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (pb + u * L < p1) ax = fma(v[u], xc[u], ax);
        }
      }
    }
    ax = sub_sum<L>(ax);
    if (i < n && sl == 0) {
      const double r = bi - ax;
      rr = fma(r, r, rr);
      const float rf = (float)r;
      const int at = pos ? pos[i] : i;  // position in the sliced layout
      rhs32[at] = rf;
      nh0[at] = rf;
    }
  }
  double v[1] = {rr}, tot[1];
  block_sum<1>(v);
  if (last_block_reduce<1>(v, partials, &ctl->arrive, tot) && threadIdx.x == 0) {
    ctl->rr = tot[0];
    if (set_bb) {
      ctl->bb = tot[0];
    }
    ctl->arrive = 0;
    __threadfence();
  }
}

// x <- x + d, d_i = h~_i / P~_i of the inner solve's final round (FP64 accumulate).
__global__ void k64_update(int n, double *__restrict__ x, const float *__restrict__ hT,
                           const float *__restrict__ invP, const int *__restrict__ pos) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int at = pos ? pos[i] : i;
  x[i] += (double)(hT[at] * invP[at]);
}

__global__ void k_to_f32(int64_t m, const double *__restrict__ s, float *__restrict__ d) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < m) d[i] = (float)s[i];
}

__global__ void k_diag32(int n, const double *__restrict__ ad, const double *__restrict__ gam,
                         float *__restrict__ d32) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) d32[i] = (float)(ad[i] + (gam ? gam[i] : 0.0));
}

__global__ void k_ctl_reset(DevCtl *c, int max_iter, double tol2, int round0 = 0) {
  c->round = round0;
  c->start = round0;
  c->done = round0 > 0 && round0 >= max_iter;
  c->status = GABP_NOT_CONVERGED;
  c->iters = round0;
  c->result_round = round0;
  c->max_iter = max_iter;
  c->check_from = 1;
  c->stable = 0;
  c->tol2bb = tol2;
  c->rr = 0.0;
  c->xx = 0.0;
  c->maxrel = 0.0;
  c->arrive = 0;
  c->edge_bad = 0;
  c->no_stop = 0;
}

// Diagonal loading of the convergence fix.  mode 1: Gamma_i = gamma A_ii (the
// unit-diagonal model I - R loaded by gamma I, in A's scaling; walk-summable for
// gamma > rho(|R|) - 1).  mode 2: Gamma_i = max(0, sum_j |A_ij| - A_ii) + gamma A_ii,
// which makes A + Gamma diagonally dominant for gamma > 0.
__global__ void k_gamma(int n, int mode, double gamma, const int *__restrict__ rp, const double *__restrict__ av,
                        const double *__restrict__ ad, double *__restrict__ out) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double d = ad[i];
  if (mode == 1) {
    out[i] = gamma * d;
  } else {
    double s = 0.0;
    for (int e = rp[i]; e < rp[i + 1]; ++e) s += fabs(av[e]);
    out[i] = fmax(0.0, s - d) + gamma * d;
  }
}

__global__ void k32_marginals(int n, const float *__restrict__ P, const int *__restrict__ pos, double *__restrict__ Pi) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) Pi[i] = (double)P[pos ? pos[i] : i];
}

// ---------------------------------------------------------------------------- sliced layout
// Rows sorted by degree (descending, stable) in windows of kSellWindow, one window a block: srow, its inverse
// pos, and the width of each slice at sp[slice + 1].
constexpr int kMaxKeyDegree = 0xfffff;
__global__ void __launch_bounds__(1024) k_sort32(int n, int npos, const int *__restrict__ rp, int *__restrict__ srow,
                                                 int *__restrict__ pos, int *__restrict__ sp) {
  __shared__ unsigned key[kSellWindow];
  const int w0 = blockIdx.x * kSellWindow;
  for (int j = threadIdx.x; j < kSellWindow; j += 1024) {
    const int d = w0 + j < n ? rp[w0 + j + 1] - rp[w0 + j] : 0;
    key[j] = ((unsigned)(kMaxKeyDegree - min(d, kMaxKeyDegree)) << 12) | (unsigned)j;
  }
  for (int k = 2; k <= kSellWindow; k <<= 1)
    for (int d = k >> 1; d > 0; d >>= 1) {
      __syncthreads();
      for (int x = threadIdx.x; x < kSellWindow / 2; x += 1024) {
        const int lo = 2 * x - (x & (d - 1)), hi = lo + d;
        const unsigned u = key[lo], v = key[hi];
        if ((u > v) == ((lo & k) == 0)) {
          key[lo] = v;
          key[hi] = u;
        }
      }
    }
  __syncthreads();
  for (int j = threadIdx.x; j < kSellWindow; j += 1024) {
    const int p = w0 + j, i = w0 + (int)(key[j] & (kSellWindow - 1));
    if (p >= npos) continue;
    srow[p] = i < n ? i : -1;
    if (i < n) pos[i] = p;
    if ((p & 31) == 0) sp[p / 32 + 1] = kMaxKeyDegree - (int)(key[j] >> 12);
  }
}

// Widths at sp[1 ..] to first slots; out: slots in all, the widest slice.  One block.
__global__ void __launch_bounds__(1024) k_scan32(int ns, int *__restrict__ sp, long long *__restrict__ out) {
  __shared__ long long sum[1024];
  __shared__ int top[1024];
  const int c = (ns + 1023) / 1024, s0 = min(ns, (int)threadIdx.x * c), s1 = min(ns, s0 + c);
  long long v = 0;
  int wmax = 0;
  for (int s = s0; s < s1; ++s) {
    v += 32LL * sp[s + 1];
    wmax = max(wmax, sp[s + 1]);
  }
  sum[threadIdx.x] = v;
  top[threadIdx.x] = wmax;
  for (int d = 1; d < 1024; d <<= 1) {
    __syncthreads();
    const long long u = threadIdx.x >= d ? sum[threadIdx.x - d] : 0;
    const int x = threadIdx.x >= d ? top[threadIdx.x - d] : 0;
    __syncthreads();
    sum[threadIdx.x] += u;
    top[threadIdx.x] = max(top[threadIdx.x], x);
  }
  __syncthreads();
  long long at = sum[threadIdx.x] - v;
  for (int s = s0; s < s1; ++s) {
    at += 32LL * sp[s + 1];
    sp[s + 1] = (int)at;
  }
  if (threadIdx.x == 0) sp[0] = 0;
  if (threadIdx.x == 1023) {
    out[0] = sum[1023];
    out[1] = top[1023];
  }
}

// f(position, slot of the CSR or -1) for every position of the slices, a warp a slice; g(p, i) for its rows.
template <typename F, typename G>
__device__ __forceinline__ void for_slices(int ns, const int *__restrict__ srow, const int *__restrict__ sp,
                                           const int *__restrict__ rp, F &&f, G &&g) {
  const WarpPos w = warp_pos();
  for (int s = w.warp; s < ns; s += w.nwarps) {
    const int p = 32 * s + w.lane, i = srow[p], q1 = sp[s + 1];
    const int e0 = i < 0 ? 0 : rp[i], e1 = i < 0 ? 0 : rp[i + 1];
    g(p, i);
    int e = e0;
    for (int q = sp[s] + w.lane; q < q1; q += 32, ++e) f(q, e < e1 ? e : -1);
  }
}
__global__ void __launch_bounds__(kBlock) k_fill32(Sell32 S, const int *__restrict__ rp, const int *__restrict__ ci,
                                                   const double *__restrict__ av, int columns) {
  for_slices(S.ns, S.srow, S.sp, rp,
             [&](int q, int e) {
               if (columns) S.sci[q] = e < 0 ? -1 : S.pos[ci[e]];
               S.sav[q] = e < 0 ? 0.f : (float)av[e];
             },
             [](int, int) {});
}
// Frozen coefficients from the CSR order to the sliced one, and back.
__global__ void __launch_bounds__(kBlock) k_coef_slice(Sell32 S, const int *__restrict__ rp, const float2 *__restrict__ CF,
                                                       const float *__restrict__ invP) {
  for_slices(S.ns, S.srow, S.sp, rp, [&](int q, int e) { if (e >= 0) S.CF[q] = CF[e]; },
             [&](int p, int i) { S.invP[p] = i < 0 ? 1.f : invP[i]; });
}
__global__ void __launch_bounds__(kBlock) k_coef_unslice(Sell32 S, const int *__restrict__ rp, float2 *__restrict__ CF,
                                                         float *__restrict__ invP) {
  for_slices(S.ns, S.srow, S.sp, rp, [&](int q, int e) { if (e >= 0) CF[e] = S.CF[q]; },
             [&](int p, int i) { if (i >= 0) invP[i] = S.invP[p]; });
}
// Diagonal (+ loading) by position, 1 where there is no row.
__global__ void k_diag32_sliced(int npos, const int *__restrict__ srow, const double *__restrict__ ad,
                                const double *__restrict__ gam, float *__restrict__ d32) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= npos) return;
  const int i = srow[p];
  d32[p] = i < 0 ? 1.f : (float)(ad[i] + (gam ? gam[i] : 0.0));
}

// ---------------------------------------------------------------------------- host side
gabp_status make_gamma(gabp_handle h, double *out) {
  Graph &g = h->g;
  k_gamma<<<(g.n + kBlock - 1) / kBlock, kBlock, 0, h->stream>>>(g.n, h->opt.gamma_mode, h->opt.gamma, g.rp, g.av,
                                                                   g.ad, out);
  GABP_CUDA(cudaGetLastError());
  return GABP_OK;
}

gabp_status marginals32(gabp_handle h, double *Pi) {
  Work32 &w = h->w32;
  if (!w.MP[0] || w.prec_round < 0) return GABP_ERR_INVALID;
  Graph &g = h->g;
  const float *P = w.prec_sliced ? w.sl.NP[w.prec_round % 3] : w.NP[w.prec_round % 3];
  k32_marginals<<<(g.n + kBlock - 1) / kBlock, kBlock, 0, h->stream>>>(g.n, P, w.prec_sliced ? w.sl.pos : nullptr, Pi);
  GABP_CUDA(cudaGetLastError());
  GABP_CUDA(cudaStreamSynchronize(h->stream));
  return GABP_OK;
}

// Graphs whose FP32 rounds may run on the sliced layout (ensure_sell32).
constexpr double kSellRowsSlot = 12000.0;
static bool sell32_size(const Graph &g) { return g.E > 0 && g.n >= kSellRowsSlot * g.avg_deg; }

gabp_status ensure_w32(gabp_handle h, int R) {
  Work32 &w = h->w32;
  Graph &g = h->g;
  size_t E = (size_t)(g.E > 0 ? g.E : 1), n = (size_t)g.n;
  // the chains serve the sliced layout, too: 3 % for its padding where it may be built
  const size_t Es = sell32_size(g) ? E + E / 32 + 4096 : E;
  w.chain = Es;
  if (!w.MP[0]) {
    GABP_CUDA(cudaMalloc(&w.MP[0], sizeof(float) * Es));
    GABP_CUDA(cudaMalloc(&w.MP[1], sizeof(float) * Es));
    for (int j = 0; j < 3; ++j) GABP_CUDA(cudaMalloc(&w.NP[j], sizeof(float) * n));
    GABP_CUDA(cudaMalloc(&w.CF, sizeof(float2) * E));
    GABP_CUDA(cudaMalloc(&w.invP, sizeof(float) * n));
    GABP_CUDA(cudaMalloc(&g.av32, sizeof(float) * E));
    w.av32_ok = false;
    GABP_CUDA(cudaMalloc(&g.ad32, sizeof(float) * n));
    GABP_CUDA(cudaMalloc(&w.ctlR, sizeof(DevCtl)));
    GABP_CUDA(cudaMemsetAsync(w.ctlR, 0, sizeof(DevCtl), h->stream));
    for (int j = 0; j < 3; ++j) GABP_CUDA(cudaMalloc(&w.NQ[j], sizeof(float2) * n));
  }
  if (w.R < R) {
    cudaFree(w.H[0]); cudaFree(w.H[1]);
    for (int j = 0; j < 3; ++j) cudaFree(w.NH[j]);
    cudaFree(w.rhs32); cudaFree(w.X); cudaFree(w.Rs); cudaFree(w.Bt);
    w.H[0] = w.H[1] = nullptr;
    w.NH[0] = w.NH[1] = w.NH[2] = nullptr;
    w.rhs32 = nullptr; w.X = w.Rs = w.Bt = nullptr;
    w.R = 0;
    GABP_CUDA(cudaMalloc(&w.H[0], sizeof(float) * Es * R));
    GABP_CUDA(cudaMalloc(&w.H[1], sizeof(float) * Es * R));
    for (int j = 0; j < 3; ++j) {  // room for the dense rounds' padding columns, finite values there
      const size_t rows = (n + 31) / 32 * 32;
      GABP_CUDA(cudaMalloc(&w.NH[j], sizeof(float) * rows * R));
      GABP_CUDA(cudaMemsetAsync(w.NH[j], 0, sizeof(float) * rows * R, h->stream));
    }
    GABP_CUDA(cudaMalloc(&w.rhs32, sizeof(float) * n * R));
    GABP_CUDA(cudaMalloc(&w.X, sizeof(double) * n * R));
    w.R = R;
    if (h->gH32) cudaGraphExecDestroy(h->gH32);
    h->gH32 = nullptr;
    h->gH32_R = -1;
    if (h->gRef) cudaGraphExecDestroy(h->gRef);  // holds the old buffers
    if (h->gRefG) cudaGraphDestroy(h->gRefG);
    h->gRef = nullptr;
    h->gRefG = nullptr;
    h->gRef_key = -1;
  }
  return GABP_OK;
}

// The FP32 values of the row CSR (the sliced layout has its own).
gabp_status csr_values32(gabp_handle h) {
  Graph &g = h->g;
  if (h->w32.av32_ok) return GABP_OK;
  if (g.E > 0) k_to_f32<<<(int)(((int64_t)g.E + kBlock - 1) / kBlock), kBlock, 0, h->stream>>>((int64_t)g.E, g.av, g.av32);
  GABP_CUDA(cudaGetLastError());
  h->w32.av32_ok = true;
  return GABP_OK;
}

static void free_sell32(Sell32 &S) {
  cudaFree(S.srow); cudaFree(S.pos); cudaFree(S.sp); cudaFree(S.sci); cudaFree(S.sav); cudaFree(S.CF);
  cudaFree(S.nodes);
  S = Sell32{};
}

void free_w32(gabp_handle h) {
  Work32 &w = h->w32;
  cudaFree(w.MP[0]); cudaFree(w.MP[1]);
  for (int j = 0; j < 3; ++j) { cudaFree(w.NP[j]); cudaFree(w.NH[j]); cudaFree(w.NQ[j]); }
  cudaFree(w.CF); cudaFree(w.invP); cudaFree(w.H[0]); cudaFree(w.H[1]);
  cudaFree(w.rhs32); cudaFree(w.X); cudaFree(w.Rs); cudaFree(w.Bt); cudaFree(w.colnorm);
  cudaFree(w.ctlR); cudaFree(w.rhs_active); cudaFree(w.rc); cudaFree(w.Bd);
  cudaFree(w.dCin); cudaFree(w.dCout); cudaFree(w.dH); cudaFree(w.dSp);
  free_sell32(w.sl);
  if (w.rc_host) cudaFreeHost(w.rc_host);
  w = Work32{};
}

static Args32 args32(gabp_handle h) {
  Args32 a;
  Graph &g = h->g;
  Work32 &w = h->w32;
  a.n = g.n; a.rp = g.rp; a.ci = g.ci; a.av = g.av32; a.ad = g.ad32;
  a.dense = g.n > 1 && (int64_t)g.E == (int64_t)g.n * (g.n - 1);  // every off-diagonal entry stored
  a.ld = w.dense_ld; a.Cin = w.dCin; a.Cout = w.dCout; a.Hd = w.dH; a.Sp = w.dSp;
  a.MP0 = w.MP[0]; a.MP1 = w.MP[1];
  a.NP0 = w.NP[0]; a.NP1 = w.NP[1]; a.NP2 = w.NP[2];
  a.CF = w.CF; a.invP = w.invP;
  a.H0 = w.H[0]; a.H1 = w.H[1];
  a.NH0 = w.NH[0]; a.NH1 = w.NH[1]; a.NH2 = w.NH[2];
  a.rhs = w.rhs32;
  a.NQ0 = w.NQ[0]; a.NQ1 = w.NQ[1]; a.NQ2 = w.NQ[2];
  a.ns = 0;
  a.sp = nullptr;
  a.cond = 0;
  a.use_cond = 0;
  a.ctl = h->ctl;
  a.partials = h->partials;
  return a;
}

// The arguments of the joint, freeze and mean rounds: the sliced layout's arrays where it is in use.
static Args32 round_args32(gabp_handle h) {
  Args32 a = args32(h);
  Work32 &w = h->w32;
  if (!w.sl_on) return a;
  const Sell32 &S = w.sl;
  a.n = 32 * S.ns; a.ns = S.ns; a.sp = S.sp; a.ci = S.sci; a.av = S.sav; a.ad = S.ad;
  a.NP0 = S.NP[0]; a.NP1 = S.NP[1]; a.NP2 = S.NP[2];
  a.CF = S.CF; a.invP = S.invP; a.rhs = S.rhs;
  a.NH0 = S.NH[0]; a.NH1 = S.NH[1]; a.NH2 = S.NH[2];
  a.NQ0 = S.NQ[0]; a.NQ1 = S.NQ[1]; a.NQ2 = S.NQ[2];
  return a;
}

// The sliced layout of the FP32 rounds (sets w.sl_on when they run on it): 32 rows a slice, lane by row, so that a
// warp's load of a stream is one line.  The row kernels' loads are cut at the rows (16 slots a row, 8 lanes: 4 to 8
// lines a load), and the L1, which takes a line a cycle, bounds them: the gathers alone need 65 us of it for 16.8 M
// slots.  Whole solves, row kernels / sliced: 2^20 rows of 16 slots 2907 / 2396 us, 1.6 M rows of 10 (least squares)
// 7548 / 5844, 2^22 rows of 6 with new values, forward and adjoint 13597 / 10459; the first solve of a 400 K-row
// graph 13.8 / 2.5 ms (no shapes to tune).
// Not where there are too few rows for a lane each: the row kernels give a row up to 16.  6 slots a row: 20 K rows
// 448 / 472 us, 40 K 507 / 499, 80 K 556 / 523; 16 slots: 80 K 521 / 544, 160 K 710 / 723, 400 K 1316 / 1194: from
// kSellRowsSlot rows a slot of the average row on.  Not where a lane's row would be long, where the padding exceeds the
// chains' room, or where there is no memory for it.
constexpr int kSellWidth32 = 96;
static gabp_status ensure_sell32(gabp_handle h) {
  Work32 &w = h->w32;
  Sell32 &S = w.sl;
  const Graph &g = h->g;
  w.sl_on = false;
  if (h->opt.lanes || w.dense_ld || !sell32_size(g)) return GABP_OK;
  if (!S.tried) {
    S.tried = true;
    const int ns = (g.n - 1) / 32 + 1, npos = 32 * ns;
    long long out[2] = {0, 0};
    bool room = cudaMalloc(&S.srow, sizeof(int) * npos) == cudaSuccess &&
                cudaMalloc(&S.pos, sizeof(int) * (size_t)g.n) == cudaSuccess &&
                cudaMalloc(&S.sp, sizeof(int) * ((size_t)ns + 1)) == cudaSuccess;
    if (room) {
      k_sort32<<<(g.n - 1) / kSellWindow + 1, 1024, 0, h->stream>>>(g.n, npos, g.rp, S.srow, S.pos, S.sp);
      long long *dout = reinterpret_cast<long long *>(h->partials);  // idle between runs
      k_scan32<<<1, 1024, 0, h->stream>>>(ns, S.sp, dout);
      GABP_CUDA(cudaGetLastError());
      GABP_CUDA(cudaMemcpyAsync(out, dout, sizeof(out), cudaMemcpyDeviceToHost, h->stream));
      GABP_CUDA(cudaStreamSynchronize(h->stream));
      room = out[1] <= kSellWidth32 && out[0] < INT32_MAX - 4096 && (size_t)out[0] <= w.chain;
    }
    if (room) {
      const size_t Es = (size_t)out[0], nodes = sizeof(float) * 15 * (size_t)npos;
      room = cudaMalloc(&S.sci, sizeof(int) * Es) == cudaSuccess && cudaMalloc(&S.sav, sizeof(float) * Es) == cudaSuccess &&
             cudaMalloc(&S.CF, sizeof(float2) * Es) == cudaSuccess && cudaMalloc(&S.nodes, nodes) == cudaSuccess;
      if (room) {
        GABP_CUDA(cudaMemsetAsync(S.nodes, 0, nodes, h->stream));  // zeros where there is no row
        float *at = S.nodes;
        for (int j = 0; j < 3; ++j, at += 2 * (size_t)npos) S.NQ[j] = reinterpret_cast<float2 *>(at);
        for (int j = 0; j < 3; ++j, at += npos) S.NP[j] = at;
        for (int j = 0; j < 3; ++j, at += npos) S.NH[j] = at;
        S.invP = at; S.rhs = at + npos; S.ad = at + 2 * (size_t)npos;
        S.ns = ns;
        S.Es = (int)Es;
        k_fill32<<<blocks_for(ns, kBlock / 32, h->max_blocks), kBlock, 0, h->stream>>>(S, g.rp, g.ci, g.av, 1);
        GABP_CUDA(cudaGetLastError());
        S.vals_ok = true;
      }
    }
    if (!room) {
      cudaGetLastError();
      free_sell32(S);
      S.tried = true;
    }
  }
  if (!S.ns) return GABP_OK;
  if (!S.vals_ok) {
    k_fill32<<<blocks_for(S.ns, kBlock / 32, h->max_blocks), kBlock, 0, h->stream>>>(S, g.rp, g.ci, g.av, 0);
    GABP_CUDA(cudaGetLastError());
    h->prof.launches += 1;
    S.vals_ok = true;
  }
  w.sl_on = true;
  return GABP_OK;
}

// The diagonal (+ loading) that the FP32 rounds run on.
static void diag32(gabp_handle h, const double *gamma_diag) {
  const Graph &g = h->g;
  const Sell32 &S = h->w32.sl;
  if (h->w32.sl_on)
    k_diag32_sliced<<<(32 * S.ns + kBlock - 1) / kBlock, kBlock, 0, h->stream>>>(32 * S.ns, S.srow, g.ad, gamma_diag, S.ad);
  else
    k_diag32<<<(g.n + kBlock - 1) / kBlock, kBlock, 0, h->stream>>>(g.n, g.ad, gamma_diag, g.ad32);
}

void drop_coef32(gabp_handle h) { h->w32.coef_ready = h->w32.sl.coef_ready = false; }

// Coefficients that are frozen in one order, in the other.
gabp_status csr_coef32(gabp_handle h) {
  Work32 &w = h->w32;
  if (w.coef_ready || !w.sl.coef_ready) return GABP_OK;
  k_coef_unslice<<<blocks_for(w.sl.ns, kBlock / 32, h->max_blocks), kBlock, 0, h->stream>>>(w.sl, h->g.rp, w.CF, w.invP);
  GABP_CUDA(cudaGetLastError());
  h->prof.launches += 1;
  w.coef_ready = true;
  return GABP_OK;
}
static gabp_status sliced_coef32(gabp_handle h) {
  Work32 &w = h->w32;
  if (w.sl.coef_ready || !w.coef_ready) return GABP_OK;
  k_coef_slice<<<blocks_for(w.sl.ns, kBlock / 32, h->max_blocks), kBlock, 0, h->stream>>>(w.sl, h->g.rp, w.CF, w.invP);
  GABP_CUDA(cudaGetLastError());
  h->prof.launches += 1;
  w.sl.coef_ready = true;
  return GABP_OK;
}
static gabp_status ready_coef32(gabp_handle h) { return h->w32.sl_on ? sliced_coef32(h) : csr_coef32(h); }
static void frozen32(gabp_handle h, int T) {  // the joint rounds' precisions of round T are frozen
  Work32 &w = h->w32;
  w.prec_round = T;
  w.prec_sliced = w.sl_on;
  w.coef_ready = !w.sl_on;
  w.sl.coef_ready = w.sl_on;
}

// The dense mean rounds' arrays (complete patterns of kDenseMin rows or more, unless the shape of the
// round kernels is pinned): sets w.dense_ld when they run the mean rounds.
static gabp_status ensure_dense32(gabp_handle h) {
  Work32 &w = h->w32;
  const Graph &g = h->g;
  w.dense_ld = 0;
  if (h->opt.lanes || g.n < kDenseMin || (int64_t)g.E != (int64_t)g.n * (g.n - 1)) return GABP_OK;
  const int ld = (g.n + 31) / 32 * 32;
  if (!w.dCin) {
    const int smem = (int)sizeof(float) * ld;
    int optin = 0, nb = 0;
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, h->device);
    cudaFuncAttributes fa;
    GABP_CUDA(cudaFuncGetAttributes(&fa, k32_dense));
    const int room = optin - (int)fa.sharedSizeBytes;  // beside the kernel's static shared memory
    if (smem > room) return GABP_OK;
    GABP_CUDA(cudaFuncSetAttribute(k32_dense, cudaFuncAttributeMaxDynamicSharedMemorySize, room));
    GABP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k32_dense, kBlock, smem));
    if (nb < 1) return GABP_OK;
    const int grid = blocks_for(g.n, kDenseRows, std::min(nb * h->num_sms, h->max_blocks));
    const size_t bytes = sizeof(float) * (size_t)g.n * ld;
    if (cudaMalloc(&w.dCin, bytes) != cudaSuccess || cudaMalloc(&w.dCout, bytes) != cudaSuccess ||
        cudaMalloc(&w.dH, bytes) != cudaSuccess ||
        cudaMalloc(&w.dSp, sizeof(float) * (size_t)grid * ld) != cudaSuccess) {
      cudaGetLastError();  // no room for them: k32_mean needs none
      cudaFree(w.dCin); cudaFree(w.dCout); cudaFree(w.dH); cudaFree(w.dSp);
      w.dCin = w.dCout = w.dH = w.dSp = nullptr;
      return GABP_OK;
    }
    w.dense_grid = grid;
    w.dense_packed = false;
  }
  w.dense_ld = ld;
  return GABP_OK;
}

// A mean round of shape (LL, UU) on stream st: the dense rounds or the complete-pattern
// variant when the matrix is dense.
template <int LL, int UU>
static void launch_mean(gabp_handle h, const Args32 &a, cudaStream_t st) {
  const int n = h->g.n;
  if (a.ld)
    k32_dense<<<h->w32.dense_grid, kBlock, sizeof(float) * a.ld, st>>>(a);
  else if (a.ns)
    ks32_mean<<<blocks_for(a.ns, kBlock / 32, resident_grid(h->num_sms, ks32_mean)), kBlock, 0, st>>>(a);
  else if (a.dense)
    k32_mean<LL, UU, true><<<blocks_for(n, kBlock / LL, resident_grid(h->num_sms, k32_mean<LL, UU, true>)), kBlock, 0,
                             st>>>(a);
  else
    k32_mean<LL, UU><<<blocks_for(n, kBlock / LL, resident_grid(h->num_sms, k32_mean<LL, UU>)), kBlock, 0, st>>>(a);
}

// A joint round, and the freeze fused with the first mean round, in the same forms.
template <int LL, int UU>
static void launch_joint(gabp_handle h, const Args32 &a, cudaStream_t st) {
  if (a.ns)
    ks32_joint<<<blocks_for(a.ns, kBlock / 32, resident_grid(h->num_sms, ks32_joint)), kBlock, 0, st>>>(a);
  else
    k32_joint<LL, UU><<<blocks_for(a.n, kBlock / LL, resident_grid(h->num_sms, k32_joint<LL, UU>)), kBlock, 0, st>>>(a);
}
template <int LL, int UU>
static void launch_freeze(gabp_handle h, const Args32 &a, cudaStream_t st) {
  if (a.ns)
    ks32_freeze<<<blocks_for(a.ns, kBlock / 32, resident_grid(h->num_sms, ks32_freeze)), kBlock, 0, st>>>(a);
  else
    k32_freeze<LL, UU><<<blocks_for(a.n, kBlock / LL, resident_grid(h->num_sms, k32_freeze<LL, UU>)), kBlock, 0, st>>>(a);
}

// Shape (lanes per row, unroll) of an FP32 round kernel: the option if set, else
// the autotuned one, else a heuristic (one unrolled pass of 4 slots per lane
// covers a row of average degree).
enum { K32_PREC = 0, K32_MEAN = 1, K32_JOINT = 2 };
static int &tuned32(gabp_handle h, int kind) {
  return kind == K32_MEAN ? h->tuned_Lm32 : kind == K32_JOINT ? h->tuned_Lj32 : h->tuned_Lp32;
}
static int shape32(gabp_handle h, int kind) {
  if (h->opt.lanes) return pinned_shape32(h->opt.lanes, h->opt.unroll);  // validated by the option check
  const int tuned = tuned32(h, kind);
  if (tuned) return tuned;
  double d = h->g.avg_deg;
  int L = 1;
  while (L < 8 && (2 * L) * kUnroll32 <= d + 0.5) L *= 2;
  return shape_code(L, kUnroll32);
}

// Autotuner of the FP32 round kernels' shapes: a few rounds of every candidate
// (lanes, unroll) under a scratch control block, fastest kept.
static gabp_status autotune32(gabp_handle h, int kind) {
  if (h->opt.lanes || tuned32(h, kind)) return GABP_OK;
  Graph &g = h->g;
  gabp_status s0 = tune_ctl(h, nullptr);  // allocates the scratch control block on first use
  if (s0 != GABP_OK) return s0;
  Args32 a = args32(h);
  a.ctl = h->ctl_tune;
  float best = 1e30f;
  int bestS = kShapes[0];
  gabp_status s;
  for (int sc : kShapes) {
    if ((s = tune_ctl(h, nullptr)) != GABP_OK) return s;
    float ms = 1e30f;
    with_shape(sc, [&](auto Lc, auto Uc) {
      constexpr int LL = decltype(Lc)::value, UU = decltype(Uc)::value;
      if (kind == K32_MEAN)
        ms = time_launches(h, [&] { launch_mean<LL, UU>(h, a, h->stream); }, 5);
      else if (kind == K32_JOINT)
        ms = time_launches(h, [&] {
          k32_joint<LL, UU><<<blocks_for(g.n, kBlock / LL, resident_grid(h->num_sms, k32_joint<LL, UU>)), kBlock, 0,
                              h->stream>>>(a);
        }, 5);
      else
        ms = time_launches(h, [&] {
          k32_prec<LL, UU><<<blocks_for(g.n, kBlock / LL, resident_grid(h->num_sms, k32_prec<LL, UU>)), kBlock, 0,
                             h->stream>>>(a);
        }, 5);
    });
    if (ms < best) { best = ms; bestS = sc; }
  }
  GABP_CUDA(cudaGetLastError());
  tuned32(h, kind) = bestS;
  tune_cache_store(h);
  return GABP_OK;
}

gabp_status precision_phase32(gabp_handle h, const double *gamma_diag) {
  NvtxRange nvtx_("gabp fp32 precision rounds");
  Work32 &w = h->w32;
  Graph &g = h->g;
  size_t E = (size_t)(g.E > 0 ? g.E : 1);
  gabp_status st = csr_values32(h);
  if (st != GABP_OK) return st;
  k_diag32<<<(g.n + kBlock - 1) / kBlock, kBlock, 0, h->stream>>>(g.n, g.ad, gamma_diag, g.ad32);
  // round-0 state: zero precision messages, P~ = diagonal
  auto init = [&]() -> gabp_status {
    GABP_CUDA(cudaMemsetAsync(w.MP[0], 0, sizeof(float) * E, h->stream));
    GABP_CUDA(cudaMemsetAsync(w.MP[1], 0, sizeof(float) * E, h->stream));
    GABP_CUDA(cudaMemcpyAsync(w.NP[0], g.ad32, sizeof(float) * g.n, cudaMemcpyDeviceToDevice, h->stream));
    return GABP_OK;
  };
  st = init();
  if (st != GABP_OK) return st;
  if (!h->opt.lanes && !h->tuned_Lp32) {
    if ((st = autotune32(h, K32_PREC)) != GABP_OK) return st;
    if ((st = init()) != GABP_OK) return st;
  }
  const int SH = shape32(h, K32_PREC);
  k_ctl_reset<<<1, 1, 0, h->stream>>>(h->ctl, kPrecMaxRounds, std::ldexp(1.0, -h->opt.prec_stop_log2));
  h->prof.launches += 2;
  GABP_CUDA(cudaGetLastError());
  Args32 a = args32(h);
  gabp_status s;
  with_shape(SH, [&](auto Lc, auto Uc) {
    constexpr int LL = decltype(Lc)::value, UU = decltype(Uc)::value;
    s = run_rounds(h, &h->gP32, &h->gP32_L, SH, [&] {
      const int nb = blocks_for(g.n, kBlock / LL, resident_grid(h->num_sms, k32_prec<LL, UU>));
      k32_prec<LL, UU><<<nb, kBlock, 0, h->stream>>>(a);
    }, kPrecMaxRounds, PH_PREC32);
  });
  if (s != GABP_OK) return s;
  const DevCtl c = *h->ctl_host;
  h->stats.rounds += c.round;
  if (c.status == GABP_BREAKDOWN || c.status == GABP_DIVERGED) return (gabp_status)c.status;
  const int Lc = SH & 0xff;
  GABP_DISPATCH_L(Lc, (k32_coef<LL><<<blocks_for(g.n, kBlock / LL, resident_grid(h->num_sms, k32_coef<LL>)), kBlock, 0,
                                      h->stream>>>(a, c.result_round)));
  h->prof.launches += 1;
  GABP_CUDA(cudaGetLastError());
  w.prec_round = c.result_round;
  w.prec_sliced = false;
  w.coef_ready = true;
  w.sl.coef_ready = false;
  w.dense_packed = false;
  return GABP_OK;
}

// Joint rounds (precision and mean messages together) from zero messages until
// the precisions are stationary or `cap` rounds; returns that round T, whose
// state freeze32 freezes.  The mean state of round T is the start of the first
// inner solve's frozen-coefficient rounds.  Needs rhs32 / NH[0] = r (k64_residual).
static gabp_status joint_phase32(gabp_handle h, const double *gamma_diag, int cap, int *T_out) {
  Work32 &w = h->w32;
  Graph &g = h->g;
  const Args32 a = round_args32(h);
  const size_t E = a.ns ? (size_t)w.sl.Es : (size_t)(g.E > 0 ? g.E : 1);
  diag32(h, gamma_diag);
  auto init = [&]() -> gabp_status {
    GABP_CUDA(cudaMemsetAsync(w.MP[0], 0, sizeof(float) * E, h->stream));
    GABP_CUDA(cudaMemsetAsync(w.MP[1], 0, sizeof(float) * E, h->stream));
    GABP_CUDA(cudaMemsetAsync(w.H[0], 0, sizeof(float) * E, h->stream));
    k32_joint_init<<<(a.n + kBlock - 1) / kBlock, kBlock, 0, h->stream>>>(a.n, a.ad, a.rhs, a.NQ0, a.NP0);
    GABP_CUDA(cudaGetLastError());
    return GABP_OK;
  };
  gabp_status st = init();
  if (st != GABP_OK) return st;
  if (!a.ns && !h->opt.lanes && !h->tuned_Lj32) {
    if ((st = autotune32(h, K32_JOINT)) != GABP_OK) return st;
    if ((st = init()) != GABP_OK) return st;
  }
  const int SH = shape32(h, K32_JOINT), key = a.ns ? -2 : SH;
  const int rounds = std::max(1, std::min(kPrecMaxRounds, cap));
  k_ctl_reset<<<1, 1, 0, h->stream>>>(h->ctl, rounds, std::ldexp(1.0, -h->opt.prec_stop_log2));
  h->prof.launches += 3;
  GABP_CUDA(cudaGetLastError());
  gabp_status s;
  with_shape(SH, [&](auto Lc, auto Uc) {
    constexpr int LL = decltype(Lc)::value, UU = decltype(Uc)::value;
    s = run_rounds(h, &h->gJ32, &h->gJ32_L, key, [&] {
      launch_joint<LL, UU>(h, a, h->stream);
    }, rounds, PH_PREC32);
  });
  if (s != GABP_OK) return s;
  const DevCtl c = *h->ctl_host;
  if (c.status == GABP_BREAKDOWN || c.status == GABP_DIVERGED) return (gabp_status)c.status;
  *T_out = c.result_round;
  return GABP_OK;
}

// The coefficient freeze at the joint rounds' last round T fused with mean round
// T + 1 (k32_freeze), on the control block armed for the inner solve from T.
static gabp_status freeze32(gabp_handle h, int T) {
  Graph &g = h->g;
  Work32 &w = h->w32;
  const Args32 a = round_args32(h);
  const int SH = shape32(h, K32_JOINT);
  prof_begin(h);
  with_shape(SH, [&](auto Lc, auto Uc) {
    constexpr int LL = decltype(Lc)::value, UU = decltype(Uc)::value;
    launch_freeze<LL, UU>(h, a, h->stream);
  });
  if (a.ld) k32_dense_pack<<<blocks_for(g.n, 1, h->max_blocks), kBlock, 0, h->stream>>>(a, 1);
  prof_end(h);
  GABP_CUDA(cudaGetLastError());
  prof_collect(h, PH_FREEZE32, 1);
  h->prof.launches += a.ld ? 2 : 1;
  frozen32(h, T);
  w.dense_packed = a.ld > 0;
  return GABP_OK;
}

// The packed coefficients for a solve that takes them as they are (no joint rounds).
static gabp_status dense_pack(gabp_handle h) {
  if (h->w32.dense_packed) return GABP_OK;
  k32_dense_pack<<<blocks_for(h->g.n, 1, h->max_blocks), kBlock, 0, h->stream>>>(args32(h), 0);
  GABP_CUDA(cudaGetLastError());
  h->prof.launches += 1;
  h->w32.dense_packed = true;
  return GABP_OK;
}

// ---------------------------------------------------------------------------- device-driven refinement loop
// The whole FP32 + FP64-refinement solve of one right-hand side as ONE CUDA
// graph: the stop decisions that the host loop of solve32_refine takes after
// each batch of rounds and after each residual are taken by single-thread
// kernels that set the conditions of while / if nodes (cudaGraphSetConditional),
// so the host only launches the graph and reads the result:
//
//   r = b - A x (x = 0), decide
//   while (refining) {
//     zero the inner messages
//     if (precisions not computed yet) { joint rounds while not stationary; freeze; continue at T }
//     while (inner not decided) { K frozen-coefficient mean rounds }
//     x += d; r = b - A x; decide
//   }
//
// Same arithmetic, same kernels, same decisions as the host-driven loop.
struct RefineCtl {
  // parameters of the call
  double tol, tol2, inner_tol, prec_thr;
  int max_refine, max_iter, inner_max, prec_cap;
  // loop state
  double rr, bb, it2;
  int steps, total_inner, status, skip, joint_pending, prec_round, cap;
  int joint_rounds; // rounds the joint loop ran
  int launches;     // kernels the graph launched after its first residual and decision
  int inner_start;  // round at which the current inner solve's while loop starts
};

struct RefineParams {
  double tol, inner_tol, prec_thr;
  int max_refine, max_iter, inner_max, prec_cap, joint;
};

__device__ void ctl_arm(DevCtl *c, int round0, int max_iter, double tol2) {
  c->round = round0;
  c->start = round0;
  c->done = round0 >= max_iter;
  c->status = GABP_NOT_CONVERGED;
  c->iters = round0;
  c->result_round = round0;
  c->max_iter = max_iter;
  c->check_from = 1;
  c->stable = 0;
  c->tol2bb = tol2;
  c->rr = 0.0;
  c->xx = 0.0;
  c->maxrel = 0.0;
  c->arrive = 0;
  c->edge_bad = 0;
  c->no_stop = 0;
}

__global__ void k_ref_setup(RefineCtl *rc, RefineParams p) {
  RefineCtl r = {};
  r.tol = p.tol;
  r.tol2 = p.tol * p.tol;
  r.inner_tol = p.inner_tol;
  r.prec_thr = p.prec_thr;
  r.max_refine = p.max_refine;
  r.max_iter = p.max_iter;
  r.inner_max = p.inner_max;
  r.prec_cap = p.prec_cap;
  r.status = GABP_NOT_CONVERGED;
  r.joint_pending = p.joint;
  r.prec_round = -1;
  *rc = r;
}

// After a residual: stop (converged / diverged / caps) or arm the next inner solve.
__global__ void k_ref_decide(RefineCtl *rc, const DevCtl *ctlR, DevCtl *ctl, int first,
                             cudaGraphConditionalHandle h_outer, cudaGraphConditionalHandle h_joint,
                             cudaGraphConditionalHandle h_inner) {
  int go = 0;
  if (!rc->skip) {
    if (!first) rc->steps += 1;
    const double rr = ctlR->rr, bb = ctlR->bb;
    rc->rr = rr;
    rc->bb = bb;
    if (!isfinite(rr)) rc->status = GABP_DIVERGED;
    else if (bb == 0.0 || rr <= rc->tol2 * bb) rc->status = GABP_OK;
    else if (rc->steps >= rc->max_refine || rc->total_inner >= rc->max_iter) rc->status = GABP_NOT_CONVERGED;
    else {
      go = 1;
      rc->inner_start = 0;
      rc->cap = min(rc->inner_max, max(1, rc->max_iter - rc->total_inner));
      const double it = inner_target(rc->inner_tol, rc->tol, bb, rr);
      rc->it2 = it * it;
      ctl_arm(ctl, 0, rc->cap, rc->it2);
    }
  }
  cudaGraphSetConditional(h_outer, go);
  cudaGraphSetConditional(h_joint, go && rc->joint_pending);
  cudaGraphSetConditional(h_inner, go);
}

__global__ void k_joint_prep(RefineCtl *rc, DevCtl *ctl, cudaGraphConditionalHandle h_jw) {
  ctl_arm(ctl, 0, max(1, min(rc->prec_cap, rc->cap)), rc->prec_thr);
  cudaGraphSetConditional(h_jw, 1);
}

// After the joint rounds (and the freeze at their last round T): stop on a
// breakdown, else continue the first inner solve's rounds from T.
__global__ void k_joint_after(RefineCtl *rc, DevCtl *ctl, cudaGraphConditionalHandle h_inner) {
  const int T = ctl->result_round, st = ctl->status;
  rc->joint_pending = 0;
  rc->joint_rounds = ctl->round;
  if (st == GABP_BREAKDOWN || st == GABP_DIVERGED) {
    rc->status = st;
    rc->skip = 1;
    cudaGraphSetConditional(h_inner, 0);
    return;
  }
  rc->prec_round = T;
  ctl_arm(ctl, T, rc->cap, rc->it2);
  cudaGraphSetConditional(h_inner, T < rc->cap);
}

// kLoopK round kernels per while-body iteration (later ones exit at once when decided)
constexpr int kLoopK = 2;

// The joint rounds' while loop ran ceil(rounds / kLoopK) bodies; with the prep, the
// joint-after, the freeze and this kernel: the launches of the joint block.  Marks
// the round from which the first inner solve's loop continues.
__global__ void k_joint_mark(RefineCtl *rc, const DevCtl *ctl, int pack) {
  rc->launches += 2 + 2 + 1 + pack + kLoopK * ((rc->joint_rounds + kLoopK - 1) / kLoopK);
  rc->inner_start = ctl->round;
}

__global__ void k_ref_after_inner(RefineCtl *rc, const DevCtl *ctl) {
  // this step's inner loop ran ceil(rounds / kLoopK) bodies; then this kernel, the
  // update, the residual and the decision
  const int worked = max(0, ctl->round - rc->inner_start);
  rc->launches += kLoopK * ((worked + kLoopK - 1) / kLoopK) + 4;
  rc->inner_start = ctl->round;
  if (rc->skip) return;
  rc->total_inner += ctl->result_round;
  if (ctl->status == GABP_DIVERGED) {
    rc->status = GABP_DIVERGED;
    rc->skip = 1;
  }
}

// x <- x + d with d from the inner solve's final round (read on the device)
__global__ void k64_update_ctl(int n, double *__restrict__ x, const float *NH0, const float *NH1, const float *NH2,
                               const float *__restrict__ invP, const int *__restrict__ pos, const DevCtl *ctl,
                               const int *skip) {
  if (*skip) return;
  const int m = ctl->result_round % 3;
  const float *__restrict__ hT = m == 0 ? NH0 : (m == 1 ? NH1 : NH2);
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int at = pos ? pos[i] : i;
  x[i] += (double)(hT[at] * invP[at]);
}

// A graph under construction: nodes are appended in sequence after `last`.
struct SeqGraph {
  cudaGraph_t g;
  cudaGraphNode_t last;
};

// Append the launches `f` makes on `stream`, captured, after seq.last.
template <typename F>
static cudaError_t seq_capture(SeqGraph &seq, cudaStream_t stream, F &&f) {
  cudaError_t e = cudaStreamBeginCaptureToGraph(stream, seq.g, seq.last ? &seq.last : nullptr, nullptr,
                                                seq.last ? 1 : 0, cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) return e;
  f();
  cudaStreamCaptureStatus cs;
  const cudaGraphNode_t *deps = nullptr;
  size_t nd = 0;
  e = cudaStreamGetCaptureInfo(stream, &cs, nullptr, nullptr, &deps, nullptr, &nd);
  std::vector<cudaGraphNode_t> frontier(deps, deps + (e == cudaSuccess ? nd : 0));
  cudaGraph_t out = nullptr;
  const cudaError_t e2 = cudaStreamEndCapture(stream, &out);
  if (e != cudaSuccess) return e;
  if (e2 != cudaSuccess) return e2;
  if (frontier.size() == 1) {
    seq.last = frontier[0];
  } else if (frontier.size() > 1) {
    cudaGraphNode_t join;
    cudaGraphNodeParams p = {};
    p.type = cudaGraphNodeTypeEmpty;
    e = cudaGraphAddNode(&join, seq.g, frontier.data(), nullptr, frontier.size(), &p);
    if (e != cudaSuccess) return e;
    seq.last = join;
  }
  return cudaSuccess;
}

// Append a while / if node on `handle`; returns its body as a new sequence.
static cudaError_t seq_conditional(SeqGraph &seq, cudaGraphConditionalHandle handle, cudaGraphConditionalNodeType type,
                                   SeqGraph *body) {
  cudaGraphNodeParams p = {};
  p.type = cudaGraphNodeTypeConditional;
  p.conditional.handle = handle;
  p.conditional.type = type;
  p.conditional.size = 1;
  cudaGraphNode_t node;
  cudaError_t e = cudaGraphAddNode(&node, seq.g, seq.last ? &seq.last : nullptr, nullptr, seq.last ? 1 : 0, &p);
  if (e != cudaSuccess) return e;
  seq.last = node;
  body->g = p.conditional.phGraph_out[0];
  body->last = nullptr;
  return cudaSuccess;
}

// Lanes per row of the FP64 residual: narrow (its per-row epilogue is FP64), but enough to fill the GPU
// where the rows are few and long (dense 8192 x 8192 matrix: 2 lanes 1.09 ms, 32 lanes 0.14).
static int residual_lanes(gabp_handle h) {
  if (h->opt.lanes) return h->opt.lanes;
  const Graph &g = h->g;
  int L = g.avg_deg >= 12.0 ? 2 : 1;
  while (L < 32 && (int64_t)g.n * L < (int64_t)h->num_sms * 2048 && g.avg_deg >= 16.0 * L) L *= 2;
  return L;
}

static gabp_status build_refine_graph(gabp_handle h, int SHm, int SHj, int LR) {
  Graph &g = h->g;
  Work32 &w = h->w32;
  cudaStream_t st = h->stream;
  cudaGraph_t root;
  GABP_CUDA(cudaGraphCreate(&root, 0));
  struct Guard {
    cudaGraph_t *g;
    ~Guard() { if (*g) cudaGraphDestroy(*g); }
  } guard{&root};
  cudaGraphConditionalHandle h_outer, h_joint, h_jw, h_inner;
  GABP_CUDA(cudaGraphConditionalHandleCreate(&h_outer, root, 0, cudaGraphCondAssignDefault));
  GABP_CUDA(cudaGraphConditionalHandleCreate(&h_joint, root, 0, cudaGraphCondAssignDefault));
  GABP_CUDA(cudaGraphConditionalHandleCreate(&h_jw, root, 0, cudaGraphCondAssignDefault));
  GABP_CUDA(cudaGraphConditionalHandleCreate(&h_inner, root, 0, cudaGraphCondAssignDefault));
  const Args32 a = round_args32(h);
  const size_t E = a.ns ? (size_t)w.sl.Es : (size_t)(g.E > 0 ? g.E : 1);
  const int *pos = a.ns ? w.sl.pos : nullptr;
  float *rhs32 = const_cast<float *>(a.rhs);
  int nbr = 1;
  GABP_DISPATCH_L(LR, nbr = blocks_for(g.n, kBlock / LL, resident_grid(h->num_sms, k64_residual<LL>)));
  RefineCtl *rc = w.rc;
  const int nb1 = (g.n + kBlock - 1) / kBlock;
  auto residual = [&](int first) {
    GABP_DISPATCH_L(LR, (k64_residual<LL><<<nbr, kBlock, 0, st>>>(g.n, g.rowptr, g.col, g.val, w.Bd, w.X, rhs32, a.NH0,
                                                                    w.ctlR, h->partials, first, pos, &rc->skip,
                                                                    first)));
  };
  SeqGraph top{root, nullptr};
  cudaError_t e = seq_capture(top, st, [&] {
    cudaMemsetAsync(w.X, 0, sizeof(double) * g.n, st);
    residual(1);
    k_ref_decide<<<1, 1, 0, st>>>(rc, w.ctlR, h->ctl, 1, h_outer, h_joint, h_inner);
  });
  SeqGraph outer{}, joint{}, jw{}, inner{};
  if (e == cudaSuccess) e = seq_conditional(top, h_outer, cudaGraphCondTypeWhile, &outer);
  if (e == cudaSuccess)
    e = seq_capture(outer, st, [&] {
      if (!a.ld) cudaMemsetAsync(w.H[0], 0, sizeof(float) * E, st);
    });
  // precision state computed together with the first inner solve
  if (e == cudaSuccess) e = seq_conditional(outer, h_joint, cudaGraphCondTypeIf, &joint);
  if (e == cudaSuccess)
    e = seq_capture(joint, st, [&] {
      cudaMemsetAsync(w.MP[0], 0, sizeof(float) * E, st);
      cudaMemsetAsync(w.MP[1], 0, sizeof(float) * E, st);
      if (a.ld) cudaMemsetAsync(w.H[0], 0, sizeof(float) * E, st);
      k32_joint_init<<<(a.n + kBlock - 1) / kBlock, kBlock, 0, st>>>(a.n, a.ad, a.rhs, a.NQ0, a.NP0);
      k_joint_prep<<<1, 1, 0, st>>>(rc, h->ctl, h_jw);
    });
  if (e == cudaSuccess) e = seq_conditional(joint, h_jw, cudaGraphCondTypeWhile, &jw);
  if (e == cudaSuccess)
    e = seq_capture(jw, st, [&] {
      Args32 aj = a;
      aj.cond = h_jw;
      aj.use_cond = 1;
      with_shape(SHj, [&](auto Lc, auto Uc) {
        constexpr int LL = decltype(Lc)::value, UU = decltype(Uc)::value;
        for (int k = 0; k < kLoopK; ++k) launch_joint<LL, UU>(h, aj, st);
      });
    });
  if (e == cudaSuccess)
    e = seq_capture(joint, st, [&] {
      k_joint_after<<<1, 1, 0, st>>>(rc, h->ctl, h_inner);
      // freeze at T fused with round T + 1 (only the freeze if the inner cap is reached)
      Args32 af = a;
      af.cond = h_inner;
      af.use_cond = 1;
      with_shape(SHj, [&](auto Lc, auto Uc) {
        constexpr int LL = decltype(Lc)::value, UU = decltype(Uc)::value;
        launch_freeze<LL, UU>(h, af, st);
      });
      if (a.ld) k32_dense_pack<<<blocks_for(g.n, 1, h->max_blocks), kBlock, 0, st>>>(af, 1);
      k_joint_mark<<<1, 1, 0, st>>>(rc, h->ctl, a.ld ? 1 : 0);
    });
  // the inner solve's frozen-coefficient rounds
  if (e == cudaSuccess) e = seq_conditional(outer, h_inner, cudaGraphCondTypeWhile, &inner);
  if (e == cudaSuccess)
    e = seq_capture(inner, st, [&] {
      Args32 am = a;
      am.cond = h_inner;
      am.use_cond = 1;
      with_shape(SHm, [&](auto Lc, auto Uc) {
        constexpr int LL = decltype(Lc)::value, UU = decltype(Uc)::value;
        for (int k = 0; k < kLoopK; ++k) launch_mean<LL, UU>(h, am, st);
      });
    });
  if (e == cudaSuccess)
    e = seq_capture(outer, st, [&] {
      k_ref_after_inner<<<1, 1, 0, st>>>(rc, h->ctl);
      k64_update_ctl<<<nb1, kBlock, 0, st>>>(g.n, w.X, a.NH0, a.NH1, a.NH2, a.invP, pos, h->ctl, &rc->skip);
      residual(0);
      k_ref_decide<<<1, 1, 0, st>>>(rc, w.ctlR, h->ctl, 0, h_outer, h_joint, h_inner);
    });
  if (e != cudaSuccess) return cuda_fail(e, "build the refinement-loop graph");
  cudaGraphExec_t exec = nullptr;
  e = cudaGraphInstantiate(&exec, root, 0);
  if (e != cudaSuccess) return cuda_fail(e, "instantiate the refinement-loop graph");
  if (h->gRef) cudaGraphExecDestroy(h->gRef);
  if (h->gRefG) cudaGraphDestroy(h->gRefG);
  h->gRef = exec;
  h->gRefG = root;
  root = nullptr;
  return GABP_OK;
}

// solve32_refine for one right-hand side without loading, as one graph launch.
static gabp_status solve32_device_loop(gabp_handle h, const double *B, double *X, double tol, int max_iter,
                                       int *iters, double *relres) {
  Work32 &w = h->w32;
  Graph &g = h->g;
  if (!w.rc) {
    GABP_CUDA(cudaMalloc(&w.rc, sizeof(RefineCtl)));
    GABP_CUDA(cudaMallocHost(&w.rc_host, sizeof(RefineCtl)));
    GABP_CUDA(cudaMalloc(&w.Bd, sizeof(double) * (size_t)g.n));
  }
  gabp_status sd = ensure_dense32(h);
  if (sd != GABP_OK) return sd;
  if ((sd = ensure_sell32(h)) != GABP_OK || (!w.sl_on && (sd = csr_values32(h)) != GABP_OK)) return sd;
  const bool joint = !(w.coef_ready || w.sl.coef_ready) || !h->opt.reuse_precisions;
  if (joint) {
    drop_coef32(h);
    w.dense_packed = false;
    if (!h->opt.overlap_precision) {
      gabp_status s = precision_phase32(h, nullptr);
      if (s != GABP_OK) return s;
    } else {
      diag32(h, nullptr);
      GABP_CUDA(cudaGetLastError());
      if (!w.sl_on && !h->opt.lanes && !h->tuned_Lj32) {
        // the autotuner runs a few joint rounds on scratch state (re-initialised by the graph)
        const size_t E = (size_t)(g.E > 0 ? g.E : 1);
        GABP_CUDA(cudaMemsetAsync(w.rhs32, 0, sizeof(float) * g.n, h->stream));
        GABP_CUDA(cudaMemsetAsync(w.MP[0], 0, sizeof(float) * E, h->stream));
        GABP_CUDA(cudaMemsetAsync(w.MP[1], 0, sizeof(float) * E, h->stream));
        GABP_CUDA(cudaMemsetAsync(w.H[0], 0, sizeof(float) * E, h->stream));
        k32_joint_init<<<(g.n + kBlock - 1) / kBlock, kBlock, 0, h->stream>>>(g.n, g.ad32, w.rhs32, w.NQ[0], w.NP[0]);
        gabp_status s = autotune32(h, K32_JOINT);
        if (s != GABP_OK) return s;
      }
    }
  }
  const bool run_joint = joint && h->opt.overlap_precision;
  gabp_status s = w.dense_ld || w.sl_on ? GABP_OK : autotune32(h, K32_MEAN);
  if (s != GABP_OK || (!run_joint && (s = ready_coef32(h)) != GABP_OK)) return s;
  if (w.dense_ld && !run_joint && (s = dense_pack(h)) != GABP_OK) return s;
  const int SHm = shape32(h, K32_MEAN), SHj = shape32(h, K32_JOINT);
  const int LR = residual_lanes(h);
  const long long key = (long long)SHm | ((long long)SHj << 16) | ((long long)LR << 32) | ((long long)w.dense_ld << 40) |
                        ((long long)w.sl_on << 62);
  if (!h->gRef || h->gRef_key != key) {
    if ((s = build_refine_graph(h, SHm, SHj, LR)) != GABP_OK) return s;
    h->gRef_key = key;
  }
  RefineParams p;
  p.tol = tol;
  p.inner_tol = h->opt.inner_tol;
  p.prec_thr = std::ldexp(1.0, -h->opt.prec_stop_log2);
  p.max_refine = h->opt.max_refine;
  p.max_iter = max_iter;
  p.inner_max = h->opt.inner_max_iter;
  p.prec_cap = kPrecMaxRounds;
  p.joint = run_joint ? 1 : 0;
  GABP_CUDA(cudaMemcpyAsync(w.Bd, B, sizeof(double) * g.n, cudaMemcpyDeviceToDevice, h->stream));
  k_ref_setup<<<1, 1, 0, h->stream>>>(w.rc, p);
  GABP_CUDA(cudaGetLastError());
  GABP_CUDA(cudaGraphLaunch(h->gRef, h->stream));
  GABP_CUDA(cudaMemcpyAsync(X, w.X, sizeof(double) * g.n, cudaMemcpyDeviceToDevice, h->stream));
  GABP_CUDA(cudaMemcpyAsync(w.rc_host, w.rc, sizeof(RefineCtl), cudaMemcpyDeviceToHost, h->stream));
  GABP_CUDA(cudaStreamSynchronize(h->stream));
  const RefineCtl r = *w.rc_host;
  h->prof.launches += 3 + (int64_t)r.launches;  // k_ref_setup, the first residual and decision, the loop
  if (run_joint) {
    if (r.prec_round >= 0) {
      frozen32(h, r.prec_round);
      w.dense_packed = w.dense_ld > 0;
    } else if (r.status != GABP_BREAKDOWN && r.status != GABP_DIVERGED) {
      // stopped before any inner solve (b = 0): the precision state is still provided
      if ((s = precision_phase32(h, nullptr)) != GABP_OK) return s;
    }
  }
  h->stats.rounds += r.total_inner;
  h->stats.refine_steps = r.steps;
  if (iters) *iters = r.total_inner;
  if (relres) *relres = r.bb > 0.0 ? sqrt(r.rr / r.bb) : 0.0;
  return (gabp_status)r.status;
}

gabp_status solve32_refine(gabp_handle h, int R, const double *B, double *X, int64_t ld, double tol,
                           int max_iter, const double *gamma_diag, int *iters, double *relres) {
  NvtxRange nvtx_("gabp fp32 messages + fp64 refinement");
  if (R != 1) return GABP_ERR_INVALID;  // batched path: gabp_solve_batched
  (void)ld;
  gabp_status s = ensure_w32(h, 1);
  if (s != GABP_OK) return s;
  Work32 &w = h->w32;
  Graph &g = h->g;
  h->stats.rounds = 0;
  h->stats.edge_updates = -1;
  h->stats.refine_steps = 0;
  const bool serial = h->opt.schedule == 1 && !gamma_diag;
  if (h->opt.device_loop && h->opt.graphs && !gamma_diag && !h->opt.profile && h->stream && !serial)
    return solve32_device_loop(h, B, X, tol, max_iter, iters, relres);
  // the precision state is cached per handle when no loading is applied; when it
  // has to be computed, it is either computed first (precision-only rounds) or
  // together with the first inner solve (joint rounds, overlap_precision)
  bool joint = false;
  if (serial) { w.dense_ld = 0; w.sl_on = false; }
  else if ((s = ensure_dense32(h)) != GABP_OK || (s = ensure_sell32(h)) != GABP_OK) return s;
  if (!w.sl_on && (s = csr_values32(h)) != GABP_OK) return s;
  if (!(w.coef_ready || w.sl.coef_ready) || gamma_diag || !h->opt.reuse_precisions) {
    drop_coef32(h);
    w.dense_packed = false;
    joint = h->opt.overlap_precision != 0 && !serial;
    if (!joint) {
      if ((s = precision_phase32(h, gamma_diag)) != GABP_OK) return s;
    }
  }
  if (!joint && (s = ready_coef32(h)) != GABP_OK) return s;
  if (gamma_diag) drop_coef32(h);  // do not reuse a loaded state for a plain solve
  if (serial && (s = serial_freeze32(h, w.CF, w.invP)) != GABP_OK) return s;  // coefficients in the serial order
  if (!serial && !w.dense_ld && !w.sl_on && (s = autotune32(h, K32_MEAN)) != GABP_OK) return s;
  if (!serial && w.dense_ld && !joint && (s = dense_pack(h)) != GABP_OK) return s;
  const int SH = shape32(h, K32_MEAN);
  const int LR = residual_lanes(h);
  int nbr = 1;
  GABP_DISPATCH_L(LR, nbr = blocks_for(g.n, kBlock / LL, resident_grid(h->num_sms, k64_residual<LL>)));
  const Args32 a = round_args32(h);
  const int *pos = a.ns ? w.sl.pos : nullptr;
  float *rhs32 = const_cast<float *>(a.rhs);
  GABP_CUDA(cudaMemsetAsync(X, 0, sizeof(double) * g.n, h->stream));
  GABP_CUDA(cudaMemsetAsync(w.ctlR, 0, sizeof(DevCtl), h->stream));
  GABP_DISPATCH_L(LR, (k64_residual<LL><<<nbr, kBlock, 0, h->stream>>>(g.n, g.rowptr, g.col, g.val, B, X, rhs32, a.NH0,
                                                                          w.ctlR, h->partials, 1, pos, nullptr, 1)));
  h->prof.launches += 1;
  GABP_CUDA(cudaGetLastError());
  DevCtl cr;
  GABP_CUDA(cudaMemcpyAsync(&cr, w.ctlR, sizeof(DevCtl), cudaMemcpyDeviceToHost, h->stream));
  GABP_CUDA(cudaStreamSynchronize(h->stream));
  const double bb = cr.bb;
  double rr = cr.rr;
  int total_inner = 0;
  gabp_status result = GABP_NOT_CONVERGED;
  if (bb == 0.0) {
    // x = 0; the precision state is still made available (marginal precisions)
    if (joint && (s = precision_phase32(h, gamma_diag)) != GABP_OK) return s;
    if (gamma_diag) drop_coef32(h);
    if (iters) *iters = 0;
    if (relres) *relres = 0.0;
    return GABP_OK;
  }
  const size_t E = a.ns ? (size_t)w.sl.Es : (size_t)(g.E > 0 ? g.E : 1);
  const double itol = h->opt.inner_tol;
  for (int step = 0; step < h->opt.max_refine; ++step) {
    if (rr <= tol * tol * bb) { result = GABP_OK; break; }
    if (total_inner >= max_iter) break;
    // inner FP32 GaBP on A d = r (messages from zero, Algorithm 1 step 1); the
    // first one may start with the joint rounds, which leave round T's mean state
    const int cap = std::min(h->opt.inner_max_iter, std::max(1, max_iter - total_inner));
    const double it_tol = inner_target(itol, tol, bb, rr);
    if (serial) {  // serial frozen-coefficient sweeps (serial.cu)
      int sweeps = 0, ist = 0;
      if ((s = serial_inner32(h, w.rhs32, cap, it_tol, &sweeps, &ist)) != GABP_OK) return s;
      total_inner += sweeps;
      h->stats.rounds += sweeps;
      if (ist == GABP_DIVERGED) { result = GABP_DIVERGED; break; }
      prof_begin(h);
      if ((s = serial_update32(h, X)) != GABP_OK) return s;
      GABP_DISPATCH_L(LR, (k64_residual<LL><<<nbr, kBlock, 0, h->stream>>>(g.n, g.rowptr, g.col, g.val, B, X, rhs32, a.NH0,
                                                                              w.ctlR, h->partials, 0, pos)));
      prof_end(h);
      h->prof.launches += 2;
      GABP_CUDA(cudaGetLastError());
      GABP_CUDA(cudaMemcpyAsync(&cr, w.ctlR, sizeof(DevCtl), cudaMemcpyDeviceToHost, h->stream));
      GABP_CUDA(cudaStreamSynchronize(h->stream));
      prof_collect(h, PH_REFINE64, 1);
      h->stats.refine_steps = step + 1;
      if (!std::isfinite(cr.rr)) { result = GABP_DIVERGED; rr = cr.rr; break; }
      rr = cr.rr;
      continue;
    }
    int T = 0;
    if (step == 0 && joint) {
      if ((s = joint_phase32(h, gamma_diag, cap, &T)) != GABP_OK) return s;
      // freeze at T fused with the first frozen-coefficient round T + 1
      k_ctl_reset<<<1, 1, 0, h->stream>>>(h->ctl, cap, it_tol * it_tol, T);
      h->prof.launches += 1;
      if ((s = freeze32(h, T)) != GABP_OK) return s;
      if (gamma_diag) drop_coef32(h);  // do not reuse a loaded state for a plain solve
    } else if (!w.dense_ld) {
      GABP_CUDA(cudaMemsetAsync(w.H[0], 0, sizeof(float) * E, h->stream));
    }
    int result_round = T;
    if (T < cap) {
      if (T == 0) {
        k_ctl_reset<<<1, 1, 0, h->stream>>>(h->ctl, cap, it_tol * it_tol, 0);
        h->prof.launches += 1;
      }
      GABP_CUDA(cudaGetLastError());
      with_shape(SH, [&](auto Lc, auto Uc) {
        constexpr int LL = decltype(Lc)::value, UU = decltype(Uc)::value;
        s = run_rounds(h, &h->gH32, &h->gH32_L, w.dense_ld ? -1 : (a.ns ? -2 : SH), [&] {
          launch_mean<LL, UU>(h, a, h->stream);
        }, cap - T, PH_MEAN32, T > 0 ? T + 1 : 0);
      });
      if (s != GABP_OK) return s;
      const DevCtl c = *h->ctl_host;
      result_round = c.result_round;
      if (c.status == GABP_DIVERGED) {
        total_inner += c.round;
        h->stats.rounds += c.round;
        result = GABP_DIVERGED;
        break;
      }
    }
    total_inner += result_round;
    h->stats.rounds += result_round;
    const float *hT = ring3(a.NH0, a.NH1, a.NH2, result_round);
    prof_begin(h);
    k64_update<<<(g.n + kBlock - 1) / kBlock, kBlock, 0, h->stream>>>(g.n, X, hT, a.invP, pos);
    GABP_DISPATCH_L(LR, (k64_residual<LL><<<nbr, kBlock, 0, h->stream>>>(g.n, g.rowptr, g.col, g.val, B, X, rhs32, a.NH0,
                                                                            w.ctlR, h->partials, 0, pos)));
    prof_end(h);
    h->prof.launches += 2;
    GABP_CUDA(cudaGetLastError());
    GABP_CUDA(cudaMemcpyAsync(&cr, w.ctlR, sizeof(DevCtl), cudaMemcpyDeviceToHost, h->stream));
    GABP_CUDA(cudaStreamSynchronize(h->stream));
    prof_collect(h, PH_REFINE64, 1);
    h->stats.refine_steps = step + 1;
    if (!std::isfinite(cr.rr)) { result = GABP_DIVERGED; rr = cr.rr; break; }
    rr = cr.rr;
  }
  if (result != GABP_DIVERGED && rr <= tol * tol * bb) result = GABP_OK;
  if (iters) *iters = total_inner;
  if (relres) *relres = sqrt(rr / bb);
  return result;
}

}  // namespace gabp
