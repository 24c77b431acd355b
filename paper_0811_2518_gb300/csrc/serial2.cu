// serial2.cu -- FP64 serial sweeps of a graph of two colours (grids, trees, bipartite graphs) above the
// sizes that one thread-block cluster runs: plain sweeps and the precision freeze.
//
// With two colours every neighbour of a row has the other colour, so a sweep is two passes over whole rows
// (pass 0: colour 0 fires and the rows of colour 1 are updated; pass 1 the other way round), and a row's
// aggregate after the pass that updated it is at once what it fires with and its aggregate at the end
// of the sweep.  Each pass therefore forms, in one traversal of its rows' slots,
//   the new messages {c, v} (P = -A c, h = -c v; solve64.cu's formula), the row's {P~, h~} and x = h~ / P~,
//   and the residual of its rows: pass 1 of sweep t for x^(t), whose colour 1 it gathers and whose own
//   rows it has just formed; pass 0 of sweep t + 1 for the rows of colour 1, from the gathered colour 0
//   of x^(t) and the row's own previous record.
// The decision about x^(t) falls at the end of pass 0 of sweep t + 1, so colour 1 keeps the records and
// messages of two sweeps.  A sweep was four traversals in four launches (the passes, a second reading
// of every row for the final x, a residual product), with eleven FP64 operations a slot and a division
// on the FP64 pipe; now it is one in two, with five.  Whole solves: 64^3 grid (98 sweeps) 9.2 ->
// 3.84 ms, 128^3 (97) 49.5 -> 18.4.
//
// Layout: Sell64 with the slices of colour 0 first (rows of each colour sorted by degree in windows).
#include "sell64.cuh"

#include <algorithm>
#include <type_traits>

namespace gabp {

namespace {

struct ArgsS2 {
  int n, ns0, ns;
  const int *__restrict__ srow;
  const int *__restrict__ sp;
  const int *__restrict__ sci;
  const int *__restrict__ srev;
  const double *__restrict__ sav;
  const double *__restrict__ ad;
  const double *__restrict__ b;
  double2 *M0, *M1;         // rows of colour 0: M0; of colour 1: M0 / M1 in even / odd sweeps
  NodeRec64 *N0, *N1, *N2;  // colour 0; colour 1 in even / odd sweeps
  double *C;
  int freeze;
  DevCtl *ctl;
  double *partials;
};

// Slots per lane whose loads are issued together, and the blocks per SM of the register budget (as the
// gather form of solve64.cu).
constexpr int kU2 = 3, kMinBlocks2 = 4;

// One slice of a pass.  MODE as in solve64.cu's plain_slice (0 plain, 1 screen, 2 verify and store, 3
// frozen); ZERO: pass 0 of the first sweep, whose reverse messages are zero.  Prev: this pass's rows'
// records of the previous sweep; Mprev: their messages.
template <int PASS, int MODE, bool ZERO>
__device__ __forceinline__ void s2_slice(const ArgsS2 &a, int sl, int lane, const double2 *__restrict__ Min,
                                         const double2 *Mprev, double2 *Mout, const NodeRec64 *__restrict__ Nin,
                                         const NodeRec64 *Prev, NodeRec64 *Nout, double &rr, int &bad, int &moving) {
  const int i = a.srow[sl * 32 + lane];
  const int q0 = a.sp[sl], p0 = q0 + lane, wd = (a.sp[sl + 1] - q0) >> 5;
  double accP = 0.0, acch = 0.0, accr = 0.0;
  for (int j = 0; j < wd; j += kU2) {
    int k[kU2];
    double A[kU2], c[kU2];
    double2 rv[kU2];
    NodeRec64 nk[kU2];
#pragma unroll
    for (int u = 0; u < kU2; ++u) {
      const int pos = p0 + 32 * (j + u);
      k[u] = j + u < wd ? __ldcs(a.sci + pos) : -1;
      if (k[u] >= 0) {
        A[u] = __ldcs(a.sav + pos);
        rv[u] = ZERO ? make_double2(0.0, 0.0) : __ldcs(Min + __ldcs(a.srev + pos));  // j -> k as k holds it
        if (MODE == 3) c[u] = __ldcs(a.C + pos);
        if (MODE == 2) c[u] = Mprev[pos].x;  // the message this one replaces
      }
    }
#pragma unroll
    for (int u = 0; u < kU2; ++u)
      if (k[u] >= 0) nk[u] = Nin[k[u]];  // k's aggregate when it fires
#pragma unroll
    for (int u = 0; u < kU2; ++u) {
      if (k[u] < 0) continue;
      const int pos = p0 + 32 * (j + u);
      if (MODE == 3) {
        const double v = fma(rv[u].x, rv[u].y, nk[u].h);
        __stcs(Mout + pos, make_double2(c[u], v));  // with c, as in solve64.cu
        acch = fma(-c[u], v, acch);
      } else {
        const double2 m = message64(A[u], nk[u], rv[u], bad);
        if (MODE == 2) {
          moving |= ulp_apart(m.x, c[u]);
          a.C[pos] = m.x;
        }
        __stcs(Mout + pos, m);
        accP = fma(-A[u], m.x, accP);
        acch = fma(-m.x, m.y, acch);
      }
      accr = fma(A[u], nk[u].x, accr);
    }
  }
  if (i >= 0) {
    const double bi = a.b[i], d = a.ad[i];
    const NodeRec64 own = Prev[i];
    double x;
    if (MODE == 3) {
      const double h = bi + acch;
      x = h * own.pad;
      Nout[i] = NodeRec64{own.P, h, x, own.pad};
    } else {
      const double P = d + accP, h = bi + acch;
      bad |= is_zero64(P) ? 2 : 0;
      if (MODE == 1) moving |= ulp_apart(P, own.P);
      x = div64(h, P);
      Nout[i] = NodeRec64{P, h, x, MODE == 2 ? rcp64(P) : x};
    }
    const double r = bi - fma(d, PASS == 1 ? x : own.x, accr);
    rr = fma(r, r, rr);
  }
}

// Pass PASS of sweep t, then the sums; in the last block, pass 1 completes the sweep and pass 0 decides
// about the previous one.
template <int PASS, int MODE>
__global__ void __launch_bounds__(kBlock, MODE == 2 ? 3 : kMinBlocks2) ks2_pass(ArgsS2 a) {
  DevCtl *ctl = a.ctl;
  if (ctl->done || (a.freeze && (ctl->stable != PASS || ctl->fstate != MODE - 1))) return;
  const int t = ctl->round + 1;
  double2 *M1 = (t & 1) ? a.M1 : a.M0;                  // colour 1's messages of this sweep
  NodeRec64 *N1 = (t & 1) ? a.N2 : a.N1;                // and records
  const double2 *Min = PASS == 0 ? a.M0 : M1;
  double2 *Mout = PASS == 0 ? M1 : a.M0;
  const double2 *Mprev = PASS == 0 ? ((t & 1) ? a.M0 : a.M1) : a.M0;
  const NodeRec64 *Nin = PASS == 0 ? a.N0 : N1;
  NodeRec64 *Nout = PASS == 0 ? N1 : a.N0;
  const NodeRec64 *Prev = PASS == 0 ? ((t & 1) ? a.N1 : a.N2) : a.N0;
  const WarpPos w = warp_pos();
  const int first = PASS == 0 ? a.ns0 : 0, cnt = PASS == 0 ? a.ns - a.ns0 : a.ns0;
  double rr = 0.0;
  int bad = 0, moving = 0;
  auto rows = [&](auto zero) {
    for (int m = 0; m * w.nwarps < cnt; ++m) {
      const int sl = pass_slice(w, m);
      if (sl < cnt)
        s2_slice<PASS, MODE, decltype(zero)::value>(a, first + sl, w.lane, Min, Mprev, Mout, Nin, Prev, Nout, rr, bad,
                                                    moving);
    }
  };
  if (PASS == 0 && MODE < 2 && t == 1) rows(std::integral_constant<bool, PASS == 0 && MODE < 2>());
  else rows(std::false_type());
  const unsigned fb = __reduce_or_sync(0xffffffffu, (unsigned)bad), fm = __reduce_or_sync(0xffffffffu, (unsigned)moving);
  if (w.lane == 0 && fb) atomicOr(&ctl->edge_bad, (int)fb);
  if (w.lane == 0 && fm) atomicOr(&ctl->fmove, 1);
  double v[1] = {rr}, tot[1];
  block_sum<1>(v);
  if (last_block_reduce<1>(v, a.partials, &ctl->arrive, tot) && threadIdx.x == 0) {
    ctl->stable = 1 - PASS;  // the pass to come (the freeze's state may change after pass 1: not another of its modes)
    if (PASS == 1) {  // the sweep is complete but for the residual of colour 1
      ctl->round = t;
      ctl->xx = tot[0];
      ctl->lam_round = ctl->edge_bad;
      ctl->edge_bad = 0;
      if (a.freeze) {  // the freeze state after this sweep (the first sweep screens nothing)
        if (MODE < 3 && (MODE == 2 || t >= 2)) freeze_step(ctl, MODE - 1, t, (double)ctl->fmove);
        ctl->fmove = 0;
      }
    } else if (t >= 2) {
      const int tchk = t - 1;
      const double r2 = ctl->xx + tot[0];
      ctl->rr = r2;
      int st = -1;
      if (ctl->lam_round) st = GABP_BREAKDOWN;
      else if (!isfinite(r2)) st = GABP_DIVERGED;
      else if (r2 <= ctl->tol2bb) st = GABP_OK;
      else if (tchk >= ctl->max_iter) st = GABP_NOT_CONVERGED;
      if (st >= 0) {
        ctl->status = st;
        ctl->iters = tchk;
        ctl->result_round = tchk;
        ctl->done = 1;
      }
    }
    ctl->arrive = 0;
    __threadfence();
  }
}

// Before the first sweep no message has been sent: colour 0 fires with {A_ii, b_i}.  ||b||^2 and the
// control block of the run.
__global__ void __launch_bounds__(kBlock) ks2_init(ArgsS2 a, const double *__restrict__ b, double *__restrict__ staged,
                                                   double tol, int max_iter) {
  double bb = 0.0;
  for (int q = blockIdx.x * kBlock + threadIdx.x; q < 32 * a.ns; q += gridDim.x * kBlock) {
    const int i = a.srow[q];
    if (i < 0) continue;
    const double bi = b[i], d = a.ad[i];
    staged[i] = bi;
    const double x = bi / d;
    (q < 32 * a.ns0 ? a.N0 : a.N1)[i] = NodeRec64{d, bi, x, x};
    bb = fma(bi, bi, bb);
  }
  double v[1] = {bb}, tot[1];
  block_sum<1>(v);
  if (last_block_reduce<1>(v, a.partials, &a.ctl->arrive, tot) && threadIdx.x == 0) {
    DevCtl *c = a.ctl;
    c->bb = tot[0];
    c->tol2bb = tol * tol * tot[0];
    c->max_iter = max_iter;
    c->status = GABP_NOT_CONVERGED;
    c->done = tot[0] == 0.0;
    c->arrive = 0;
    __threadfence();
  }
}

__global__ void ks2_x(int n, const int *__restrict__ colour, const NodeRec64 *__restrict__ N0,
                      const NodeRec64 *__restrict__ N1, double *__restrict__ out, int precisions) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const NodeRec64 *r = (colour[i] == 0 ? N0 : N1) + i;
  out[i] = precisions ? r->P : r->x;
}

// {P, h} of every compact CSR slot
__global__ void ks2_messages(int n, const int *__restrict__ rp, const int *__restrict__ colour,
                             const int *__restrict__ c2s, const double *__restrict__ av,
                             const double2 *__restrict__ M0, const double2 *__restrict__ M1, double2 *__restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double2 *M = colour[i] == 0 ? M0 : M1;
  for (int e = rp[i]; e < rp[i + 1]; ++e) {
    const double2 m = M[c2s[e]];
    out[e] = make_double2(-av[e] * m.x, -m.x * m.y);
  }
}

// The layout, its values and the state; GABP_NOT_RUN, now and from then on, where there is no room for them
// (the general passes need one message store and no padding).
gabp_status ensure_two(gabp_handle h) {
  WorkS &s = h->ws;
  WorkS2 &w = s.two;
  const Graph &g = h->g;
  const size_t n = (size_t)g.n;
  if (w.refused) return GABP_NOT_RUN;
  auto refuse = [&] {
    cudaGetLastError();
    free_serial2(s);
    w.refused = true;
    return GABP_NOT_RUN;
  };
  if (!w.sl.ready) {
    std::vector<int> rp(n + 1), rows(n);
    GABP_CUDA(cudaMemcpyAsync(rp.data(), g.rp, sizeof(int) * rp.size(), cudaMemcpyDeviceToHost, h->stream));
    GABP_CUDA(cudaMemcpyAsync(rows.data(), s.oid, sizeof(int) * n, cudaMemcpyDeviceToHost, h->stream));
    GABP_CUDA(cudaStreamSynchronize(h->stream));
    const size_t n0 = (size_t)s.cstart[1];
    sort_degree_windows(rp, rows, 0, n0);
    sort_degree_windows(rp, rows, n0, n);
    const size_t p0 = (n0 + 31) / 32 * 32, p1 = (n - n0 + 31) / 32 * 32;
    std::vector<int> srow(p0 + p1, -1);
    std::copy(rows.begin(), rows.begin() + n0, srow.begin());
    std::copy(rows.begin() + n0, rows.end(), srow.begin() + p0);
    w.ns0 = (int)(p0 / 32);
    if (build_sell64(h, w.sl, rp, srow, nullptr) != GABP_OK) return refuse();
  } else if (!w.sl.vals_ok) {
    const gabp_status vs = sell64_values(h, w.sl);
    if (vs != GABP_OK) return vs;
  }
  const size_t Es = (size_t)std::max(w.sl.Es, 1);
  bool room = true;
  auto get = [&](auto *&p, size_t m) { room = room && (p || cudaMalloc(&p, sizeof(*p) * m) == cudaSuccess); };
  for (int q = 0; q < 2; ++q) get(w.M[q], Es);
  for (int q = 0; q < 3; ++q) get(w.N[q], n);
  get(w.b, n);
  if (h->opt.freeze_precisions) get(w.C, Es);
  return room ? GABP_OK : refuse();
}

// Where the general passes (2 lanes a row from 8 slots a row, 4 from 24) are the faster ones: rows that are long for
// a lane each, and too few of them to hide that behind other warps.  Bipartite graphs of two equal sides, whole solves
// in ms, general / these: 24 slots a row or more, 2 x 6,000 rows of 40 2.95 / 4.70, 2 x 10,000 of 25 2.87 / 3.65, 2 x
// 20,000 of 100 8.43 / 9.64, 2 x 40,000 of 100 15.6 / 12.1 and of 40 7.40 / 5.29; 16 slots, 2 x 3,000 rows 2.35 / 2.10.
// With the freeze, whose empty launches weigh on these: 8 slots a row or more, 2 x 20,000 rows of 16 2.36 / 3.14, 2 x
// 40,000 of 100 14.1 / 14.8 and of 40 6.75 / 6.49, 2 x 60,000 of 16 4.63 / 3.55; below 8, 2 x 6,000 rows 2.10 / 1.59.
bool two_pays(gabp_handle h) {
  const int slices = h->g.n / 32;
  return h->opt.freeze_precisions ? h->g.avg_deg < 8.0 || slices >= 20 * h->num_sms
                                  : h->g.avg_deg < 24.0 || slices >= 16 * h->num_sms;
}

ArgsS2 args_two(gabp_handle h) {
  WorkS2 &w = h->ws.two;
  ArgsS2 a;
  a.n = h->g.n; a.ns0 = w.ns0; a.ns = w.sl.ns;
  a.srow = w.sl.srow; a.sp = w.sl.sp; a.sci = w.sl.sci; a.srev = w.sl.srev; a.sav = w.sl.sav;
  a.ad = h->g.ad; a.b = w.b;
  a.M0 = w.M[0]; a.M1 = w.M[1]; a.N0 = w.N[0]; a.N1 = w.N[1]; a.N2 = w.N[2];
  a.C = w.C; a.freeze = h->opt.freeze_precisions; a.ctl = h->ctl; a.partials = h->partials;
  return a;
}

template <int PASS, int MODE>
void launch_two(gabp_handle h, const ArgsS2 &a) {
  const int ns = PASS == 0 ? a.ns - a.ns0 : a.ns0;
  ks2_pass<PASS, MODE><<<blocks_for(ns, kBlock / 32, resident_grid(h->num_sms, ks2_pass<PASS, MODE>)), kBlock, 0,
                         h->stream>>>(a);
}

}  // namespace

void free_serial2(WorkS &s) {
  WorkS2 &w = s.two;
  free_sell64(w.sl);
  for (int q = 0; q < 2; ++q) cudaFree(w.M[q]);
  for (int q = 0; q < 3; ++q) cudaFree(w.N[q]);
  cudaFree(w.C); cudaFree(w.b);
  if (w.graph) cudaGraphExecDestroy(w.graph);
  w = WorkS2{};
}

gabp_status solve64_two_colours(gabp_handle h, const double *b, double *x, double tol, int max_iter, int *iters,
                                double *relres) {
  if (!two_pays(h)) return GABP_NOT_RUN;
  gabp_status st = ensure_two(h);
  if (st != GABP_OK) return st;
  Graph &g = h->g;
  WorkS &s = h->ws;
  WorkS2 &w = s.two;
  const ArgsS2 a = args_two(h);
  const int cap = std::max(1, max_iter);
  GABP_CUDA(cudaMemsetAsync(h->ctl, 0, sizeof(DevCtl), h->stream));
  ks2_init<<<blocks_for(g.n, kBlock, h->max_blocks), kBlock, 0, h->stream>>>(a, b, w.b, tol, cap);
  GABP_CUDA(cudaGetLastError());
  h->prof.launches += 1;
  if ((st = read_ctl(h)) != GABP_OK) return st;
  if (h->ctl_host->done) return GABP_NOT_RUN;  // b = 0
  h->stats.edge_updates = -1;
  h->stats.refine_steps = 0;
  // one sweep; with the freeze each pass as its three modes, of which the state picks one (it changes
  // after pass 1 only, so a sweep runs in one state)
  st = run_rounds(h, &w.graph, &w.graph_key, a.freeze, [&] {
    if (a.freeze) {
      launch_two<0, 3>(h, a); launch_two<0, 2>(h, a); launch_two<0, 1>(h, a);
      launch_two<1, 3>(h, a); launch_two<1, 2>(h, a); launch_two<1, 1>(h, a);
    } else {
      launch_two<0, 0>(h, a); launch_two<1, 0>(h, a);
    }
  }, cap + 1, PH_FP64);
  if (st != GABP_OK) return st;
  const DevCtl c = *h->ctl_host;
  const int n1 = (g.n + kBlock - 1) / kBlock;
  ks2_x<<<n1, kBlock, 0, h->stream>>>(g.n, s.colour, w.N[0], w.N[1 + (c.result_round & 1)], x, 0);
  GABP_CUDA(cudaGetLastError());
  GABP_CUDA(cudaStreamSynchronize(h->stream));
  h->prof.launches += 1;
  h->stats.rounds = c.result_round;
  h->stats.freeze_round = a.freeze ? c.fround : 0;
  h->stats.freeze_checks = a.freeze ? c.fchecks : 0;
  s.valid = true;
  s.last_two = true;
  s.result_round = c.result_round;
  if (iters) *iters = c.iters;
  if (relres) *relres = std::sqrt(c.rr / c.bb);
  return (gabp_status)c.status;
}

gabp_status two_colours_messages(gabp_handle h, double2 *M_input_layout) {
  WorkS &s = h->ws;
  ks2_messages<<<(h->g.n + kBlock - 1) / kBlock, kBlock, 0, h->stream>>>(
      h->g.n, h->g.rp, s.colour, s.two.sl.c2s, h->g.av, s.two.M[0], s.two.M[s.result_round & 1], M_input_layout);
  GABP_CUDA(cudaGetLastError());
  return GABP_OK;
}

gabp_status two_colours_marginals(gabp_handle h, double *Pi) {
  WorkS &s = h->ws;
  ks2_x<<<(h->g.n + kBlock - 1) / kBlock, kBlock, 0, h->stream>>>(h->g.n, s.colour, s.two.N[0],
                                                                   s.two.N[1 + (s.result_round & 1)], Pi, 1);
  GABP_CUDA(cudaGetLastError());
  GABP_CUDA(cudaStreamSynchronize(h->stream));
  return GABP_OK;
}

}  // namespace gabp
