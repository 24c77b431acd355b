// batched.cu -- many right-hand sides in one launch sequence: FP32 mean messages
// for R right-hand sides sharing one converged precision state, FP64 iterative
// refinement per column.
//
// The precision messages depend on A only (eq_prec and eq_prec_message have no
// b in them), so the FP32 precision phase and the frozen coefficient pairs of
// solve32.cu serve every right-hand side.  The mean messages of round t are
//   h_{k->i}^{(t)} = c_in (h~_k^{(t-1)} - h_{i->k}^{(t-1)}),
// run for RP columns at once, and the message store, E x RP floats, is the traffic.  Only the
// messages of EVEN rounds are stored, one array:
//   even t   row i forms the reverse message of round t-1 again from what it held at t-2,
//            h_{i->k}^{(t-1)} = c_out (h~_i^{(t-2)} - h_{k->i}^{(t-2)}), its own slot, which it
//            overwrites with h_{k->i}^{(t)};
//   odd t    the reverse message of round t-1 is the stored one of the reverse edge, read from row
//            k's slot; nothing is written but the aggregates.
// A pair of rounds moves three messages per slot where the recompute form in every round (two
// stores) moves four.  A message row is RP contiguous floats, so the gather pays without locality, too (random
// graphs, whole solves with four messages / three: 2^20 rows of degree 16, 64 columns 50.9 / 42.2 ms, 128 columns 104 /
// 82.6, 8 columns 32.0 / 27.4; 200,003 rows 10.6 / 8.6; 2^20 rows of degree 6, one column 24.3 / 22.1).
// Layout: slot-major, column-minor -- H[e][r], NH[i][r] -- so a warp that owns a
// row reads one coefficient pair and one column index per slot (broadcast) and
// moves RP contiguous floats for the slot's messages and for the sender's
// aggregate: every edge-array access and every gather is a coalesced 128-512 B
// row.  One warp per row; lane l owns columns [l*VEC, l*VEC+VEC).
#include "gabp_internal.cuh"
#include "devutil.cuh"

#include <algorithm>
#include <cmath>
#include <vector>

namespace gabp {

namespace {

template <int VEC>
__device__ __forceinline__ void ldv(const float *p, float (&v)[VEC]) {
  if constexpr (VEC == 1) {
    v[0] = *p;
  } else if constexpr (VEC == 2) {
    const float2 q = *reinterpret_cast<const float2 *>(p);
    v[0] = q.x; v[1] = q.y;
  } else {
    const float4 q = *reinterpret_cast<const float4 *>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  }
}
template <int VEC>
__device__ __forceinline__ void ldv_cs(const float *p, float (&v)[VEC]) {
  if constexpr (VEC == 1) {
    v[0] = __ldcs(p);
  } else if constexpr (VEC == 2) {
    const float2 q = __ldcs(reinterpret_cast<const float2 *>(p));
    v[0] = q.x; v[1] = q.y;
  } else {
    const float4 q = __ldcs(reinterpret_cast<const float4 *>(p));
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  }
}
template <int VEC>
__device__ __forceinline__ void stv(float *p, const float (&v)[VEC]) {
  if constexpr (VEC == 1) {
    *p = v[0];
  } else if constexpr (VEC == 2) {
    *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]);
  } else {
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
  }
}
template <int VEC>
__device__ __forceinline__ void stv_cs(float *p, const float (&v)[VEC]) {
  if constexpr (VEC == 1) {
    __stcs(p, v[0]);
  } else if constexpr (VEC == 2) {
    __stcs(reinterpret_cast<float2 *>(p), make_float2(v[0], v[1]));
  } else {
    __stcs(reinterpret_cast<float4 *>(p), make_float4(v[0], v[1], v[2], v[3]));
  }
}

struct ArgsB {
  int n, RP;
  const int *__restrict__ rp;
  const int *__restrict__ ci;
  const int *__restrict__ rev;
  const float2 *__restrict__ CF;
  const float *__restrict__ invP;
  float *H;  // [E][RP] messages of the latest even round
  float *NH0, *NH1, *NH2;
  const float *rhs;
  DevCtl *ctl;
  double *red;  // [2][gridDim][RP] per-block per-column partial sums
  double *col;  // [4][RP] per-column results (0: dxx, 1: xx)
};

__device__ __forceinline__ float *ring3b(float *a, float *b, float *c, int t) {
  int m = t % 3;
  return m == 0 ? a : (m == 1 ? b : c);
}

// Per-column block reduction of NV per-thread vectors acc[j][v] (column l*VEC+v)
// over the block's warps, written to red[j][blockIdx][col].  Then the last block
// sums the columns over blocks into col[j][...].  Returns true in the last block.
template <int VEC, int NV>
__device__ bool col_reduce(const double (&acc)[NV][VEC], int RP, double *red, double *colout, unsigned int *arrive) {
  extern __shared__ double shc[];  // [NV][warps][RP]
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = kBlock / 32;
#pragma unroll
  for (int j = 0; j < NV; ++j)
#pragma unroll
    for (int v = 0; v < VEC; ++v) shc[(j * nw + w) * RP + l * VEC + v] = acc[j][v];
  __syncthreads();
  for (int c = threadIdx.x; c < NV * RP; c += kBlock) {
    const int j = c / RP, r = c % RP;
    double s = 0.0;
    for (int q = 0; q < nw; ++q) s += shc[(j * nw + q) * RP + r];
    red[((size_t)j * gridDim.x + blockIdx.x) * RP + r] = s;
  }
  __shared__ bool s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned int prev = atomicAdd(arrive, 1u);
    s_last = (prev == gridDim.x - 1);
  }
  __syncthreads();
  if (!s_last) return false;
  __threadfence();
  for (int c = threadIdx.x; c < NV * RP; c += kBlock) {
    const int j = c / RP, r = c % RP;
    double s = 0.0;
    for (int bI = 0; bI < (int)gridDim.x; ++bI) s += __ldcg(red + ((size_t)j * gridDim.x + bI) * RP + r);
    colout[j * RP + r] = s;
  }
  __threadfence();
  __syncthreads();
  return true;
}

// Slots of a row whose loads are issued together, and the blocks per SM of the register budget.  A
// round is bound by HBM (128^3 grid, 64 columns: 6.9 GB on average, 1.01 ms at the measured copy rate) and
// by the bytes its warps keep in flight: 2 slots and 6 blocks 1.33 ms per round (1.68 with four messages a
// pair of rounds); 7 or 8 blocks the same, 3 slots with 6 / 5 / 4 blocks 1.37 / 1.42 / 1.74, 1 with 8 1.47.
#ifndef GABP_KB_U
#define GABP_KB_U 2
#endif
#ifndef GABP_KB_MINB
#define GABP_KB_MINB 6
#endif
template <int VEC>
constexpr int kBU = VEC == 4 ? 2 : GABP_KB_U;
// Rounds that last as long as their longest row, one warp waiting for its loads (few rows, or a hub among many), take more
// slots of a row together.  With 2, the rounds that read the reverse messages through rev cost such graphs more than
// the store they save; whole solves in ms with four messages a pair of rounds / with three / with three and 8 slots, 16
// columns: 200 rows of 40 slots 2.51 / 2.71 / 2.37, 1,000 rows of 100 4.55 / 4.31 / 3.24, 60,000 rows of
// 6 with a hub of 1,000 45.8 / 47.0 / 25.1, 100,000 rows of a heavy tail 168 / 182 / 86.
constexpr int kBULong = 8;
// A slot of the longest row takes 0.35 us of a round with 2 slots at a time; the round's bytes as below.
static bool long_row_round(const Graph &g, int max_deg, int RP) {
  const double bytes = (double)g.E * (6.0 * RP + 14.0) + (double)g.n * (16.0 * RP + 8.0);
  return 0.35 * max_deg > bytes / 6.8e6;
}

// Rounds by what their reverse messages come from: none in round 1 (zero messages), the row's own
// aggregate in round 2 (its stored messages are the zero ones, not read), then as above.
enum BKind { kBFirst, kBSecond, kBEven, kBOdd };

// NU slots e .. e + NU - 1 of one row: messages k -> i of this round added to acc, stored in even rounds.
template <int VEC, BKind KIND, int NU>
__device__ __forceinline__ void kb_slots(const ArgsB &a, int e, int c0, const float *__restrict__ Hm1,
                                         const float (&hi2)[VEC], float (&acc)[VEC]) {
  const int RP = a.RP;
  int k[NU], rv[NU];
  float2 cf[NU];
  float hs[NU][VEC], hk[NU][VEC];
#pragma unroll
  for (int u = 0; u < NU; ++u) {
    k[u] = a.ci[e + u];
    cf[u] = a.CF[e + u];
    if (KIND == kBOdd) rv[u] = a.rev[e + u];
  }
#pragma unroll
  for (int u = 0; u < NU; ++u) {
    if (KIND == kBEven) ldv_cs<VEC>(a.H + (size_t)(e + u) * RP + c0, hs[u]);
    if (KIND == kBOdd) ldv_cs<VEC>(a.H + (size_t)rv[u] * RP + c0, hs[u]);
    ldv<VEC>(Hm1 + (size_t)k[u] * RP + c0, hk[u]);
  }
#pragma unroll
  for (int u = 0; u < NU; ++u) {
    float hn[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
      const float hout = KIND == kBFirst ? 0.f                               // message i -> k at t-1
                         : KIND == kBOdd ? hs[u][v]
                                         : cf[u].y * (hi2[v] - (KIND == kBEven ? hs[u][v] : 0.f));
      hn[v] = cf[u].x * (hk[u][v] - hout);                                   // message k -> i at t
      acc[v] += hn[v];
    }
    if (KIND == kBEven || KIND == kBSecond) stv_cs<VEC>(a.H + (size_t)(e + u) * RP + c0, hn);
  }
}

template <int VEC, BKind KIND, int NU>
__device__ __forceinline__ void kb_rows(const ArgsB &a, const float *__restrict__ Hm1, const float *__restrict__ Hm2,
                                        float *__restrict__ Ht, float (&acc2)[2][VEC]) {
  const int RP = a.RP;
  const int c0 = (threadIdx.x & 31) * VEC;
  const int warp = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * kBlock) >> 5;
  for (int i = warp; i < a.n; i += nwarps) {
    float hi2[VEC], acc[VEC];
    if (KIND == kBEven || KIND == kBSecond) ldv<VEC>(Hm2 + (size_t)i * RP + c0, hi2);
#pragma unroll
    for (int v = 0; v < VEC; ++v) acc[v] = 0.f;
    int e = a.rp[i];
    const int e1 = a.rp[i + 1];
    for (; e + NU <= e1; e += NU) kb_slots<VEC, KIND, NU>(a, e, c0, Hm1, hi2, acc);
    if (NU > 4 && e + 4 <= e1) { kb_slots<VEC, KIND, 4>(a, e, c0, Hm1, hi2, acc); e += 4; }
    if (NU > 2 && e + 2 <= e1) { kb_slots<VEC, KIND, 2>(a, e, c0, Hm1, hi2, acc); e += 2; }
    for (; e < e1; ++e) kb_slots<VEC, KIND, 1>(a, e, c0, Hm1, hi2, acc);
    float rh[VEC], hp[VEC], hnew[VEC];
    ldv<VEC>(a.rhs + (size_t)i * RP + c0, rh);
    ldv<VEC>(Hm1 + (size_t)i * RP + c0, hp);
    const float ip = a.invP[i];
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
      hnew[v] = rh[v] + acc[v];
      const float x = hnew[v] * ip, dx = (hnew[v] - hp[v]) * ip;
      acc2[0][v] = fmaf(dx, dx, acc2[0][v]);
      acc2[1][v] = fmaf(x, x, acc2[1][v]);
    }
    stv<VEC>(Ht + (size_t)i * RP + c0, hnew);
  }
}

// Round t of the batched frozen-precision mean iteration (one warp per row).
// Stops when every column with a nonzero iterate has ||dx_r|| <= inner_tol ||x_r||.
template <int VEC, int NU>
__global__ void __launch_bounds__(kBlock, NU > 2 ? 2 : GABP_KB_MINB) kb_mean(ArgsB a) {
  DevCtl *ctl = a.ctl;
  if (ctl->done) return;
  const int t = ctl->round + 1;
  const int RP = a.RP;
  const float *__restrict__ Hm1 = ring3b(a.NH0, a.NH1, a.NH2, t + 2);
  const float *__restrict__ Hm2 = ring3b(a.NH0, a.NH1, a.NH2, t + 1);
  float *__restrict__ Ht = ring3b(a.NH0, a.NH1, a.NH2, t);
  float acc2[2][VEC];
#pragma unroll
  for (int v = 0; v < VEC; ++v) acc2[0][v] = acc2[1][v] = 0.f;
  if (t & 1) {
    if (t == 1) kb_rows<VEC, kBFirst, NU>(a, Hm1, Hm2, Ht, acc2);
    else kb_rows<VEC, kBOdd, NU>(a, Hm1, Hm2, Ht, acc2);
  } else {
    if (t == 2) kb_rows<VEC, kBSecond, NU>(a, Hm1, Hm2, Ht, acc2);
    else kb_rows<VEC, kBEven, NU>(a, Hm1, Hm2, Ht, acc2);
  }
  double accd[2][VEC];
#pragma unroll
  for (int v = 0; v < VEC; ++v) {
    accd[0][v] = (double)acc2[0][v];
    accd[1][v] = (double)acc2[1][v];
  }
  if (col_reduce<VEC, 2>(accd, RP, a.red, a.col, &ctl->arrive) && threadIdx.x == 0) {
    ctl->round = t;
    int notdone = 0;
    bool finite = true;
    for (int r = 0; r < RP; ++r) {
      const double dxx = a.col[r], xx = a.col[RP + r];
      if (!isfinite(dxx) || !isfinite(xx)) finite = false;
      if (xx > 0.0 && !(dxx <= ctl->tol2bb * xx)) ++notdone;
    }
    ctl->rr = (double)notdone;
    if (ctl->no_stop) {
    } else if (!finite) {
      ctl->status = GABP_DIVERGED; ctl->iters = t; ctl->result_round = t; ctl->done = 1;
    } else if (t >= 2 && notdone == 0) {
      ctl->status = GABP_OK; ctl->iters = t; ctl->result_round = t; ctl->done = 1;
    } else if (t >= ctl->max_iter) {
      ctl->status = GABP_NOT_CONVERGED; ctl->iters = t; ctl->result_round = t; ctl->done = 1;
    }
    ctl->arrive = 0;
    __threadfence();
  }
}

// R = B - A X in FP64 for all columns (one warp per row, full CSR with the
// diagonal); FP32 copies seed the next inner solve; per-column ||r||^2.
template <int VEC>
__global__ void __launch_bounds__(kBlock) kb_residual(int n, int RP, const int *__restrict__ rowptr,
                                                     const int *__restrict__ col, const double *__restrict__ val,
                                                     const double *__restrict__ Bt, const double *__restrict__ X,
                                                     float *__restrict__ rhs, float *__restrict__ nh0, double *red,
                                                     double *colout, unsigned int *arrive) {
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * kBlock) >> 5;
  const int c0 = lane * VEC;
  double rrd[1][VEC];
#pragma unroll
  for (int v = 0; v < VEC; ++v) rrd[0][v] = 0.0;
  for (int i = warp; i < n; i += nwarps) {
    double ax[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) ax[v] = 0.0;
    for (int p = rowptr[i]; p < rowptr[i + 1]; ++p) {
      const double A = val[p];
      const double *xr = X + (size_t)col[p] * RP + c0;
#pragma unroll
      for (int v = 0; v < VEC; ++v) ax[v] = fma(A, xr[v], ax[v]);
    }
    float rf[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
      const double r = Bt[(size_t)i * RP + c0 + v] - ax[v];
      rrd[0][v] = fma(r, r, rrd[0][v]);
      rf[v] = (float)r;
    }
    stv<VEC>(rhs + (size_t)i * RP + c0, rf);
    stv<VEC>(nh0 + (size_t)i * RP + c0, rf);
  }
  if (col_reduce<VEC, 1>(rrd, RP, red, colout, arrive) && threadIdx.x == 0) {
    *arrive = 0;  // colout[r] now holds column r's ||b_r - A x_r||^2
    __threadfence();
  }
}

// X[i][r] += h~_i^{(T)}[r] / P~_i
template <int VEC>
__global__ void kb_update(int n, int RP, double *__restrict__ X, const float *__restrict__ hT,
                          const float *__restrict__ invP) {
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * blockDim.x) >> 5;
  for (int i = warp; i < n; i += nwarps) {
    const float ip = invP[i];
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
      const size_t q = (size_t)i * RP + lane * VEC + v;
      X[q] += (double)(hT[q] * ip);
    }
  }
}

// Column-major user arrays <-> row-major [n][RP] work arrays (32 x 32 tiles).
__global__ void kb_gather_cols(int n, int R, int RP, const double *__restrict__ B, int64_t ld,
                               double *__restrict__ Bt) {
  __shared__ double tile[32][33];
  const int i0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  for (int q = threadIdx.y; q < 32; q += blockDim.y) {
    const int r = r0 + q, i = i0 + threadIdx.x;
    tile[q][threadIdx.x] = (r < R && i < n) ? B[(size_t)r * ld + i] : 0.0;
  }
  __syncthreads();
  for (int q = threadIdx.y; q < 32; q += blockDim.y) {
    const int i = i0 + q, r = r0 + threadIdx.x;
    if (i < n && r < RP) Bt[(size_t)i * RP + r] = tile[threadIdx.x][q];
  }
}

__global__ void kb_scatter_cols(int n, int R, int RP, const double *__restrict__ Xt, double *__restrict__ X,
                                int64_t ld) {
  __shared__ double tile[32][33];
  const int i0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  for (int q = threadIdx.y; q < 32; q += blockDim.y) {
    const int i = i0 + q, r = r0 + threadIdx.x;
    tile[q][threadIdx.x] = (i < n && r < RP) ? Xt[(size_t)i * RP + r] : 0.0;
  }
  __syncthreads();
  for (int q = threadIdx.y; q < 32; q += blockDim.y) {
    const int r = r0 + q, i = i0 + threadIdx.x;
    if (r < R && i < n) X[(size_t)r * ld + i] = tile[threadIdx.x][q];
  }
}

// ---------------------------------------------------------------------------- serial schedule, R right-hand sides
// Pass c of a serial frozen-coefficient mean sweep for RP columns (one warp per
// new row, lane l owns columns [l*VEC, l*VEC+VEC)); the layout, the order and
// the recompute identity are those of serial.cu.  Per-column sums of the pass
// go to acc[2][RP]; after the last pass every column with a nonzero iterate must
// have its estimated error (step x q/(1-q), q the step ratio of the last two
// sweeps, taken between 1 and 4 steps) within itol ||x_r||.
struct ArgsBS {
  int n, C, RP;
  const int *__restrict__ co;
  const int *__restrict__ sci;
  const int *__restrict__ scol;
  const int *__restrict__ srp;
  const float2 *__restrict__ sCF;
  const float *__restrict__ sinvP;
  const float *__restrict__ srhs;  // [n][RP] new order
  const int *__restrict__ srev;
  int n1, e1;                      // two colours: the first row of colour 1 and its first slot
  float *sH;                       // [E][RP] serial slot order (two colours: the slots from e1 on)
  float *hfire;                    // [n][RP] new order
  DevCtl *ctl;
  double *red;
  double *col;                     // [2][RP] pass sums, then [2][RP] sweep sums, [RP] previous step
};

// As above for the serial sweeps: 3 slots and 5 blocks (two colours, 128^3 grid, 64 columns: 1.49 ms per
// sweep, 1.82 with four messages a pair of slots); 2 and 6 the same, 3 and 6 1.51, 3 and 4 1.58, 4 and 5 1.59.
#ifndef GABP_KBS_U
#define GABP_KBS_U 3
#endif
#ifndef GABP_KBS_MINB
#define GABP_KBS_MINB 5
#endif
constexpr int kBsU = GABP_KBS_U;  // slots of a row whose loads are issued together

// The end of a pass: per-column sums over the grid; the last block adds them to the sweep's and, after
// the sweep's last pass, takes the per-column decision.
template <int VEC>
__device__ __forceinline__ void kbs_finish(const ArgsBS &a, const float (&acc2)[2][VEC], bool last) {
  DevCtl *ctl = a.ctl;
  const int RP = a.RP;
  double accd[2][VEC];
#pragma unroll
  for (int v = 0; v < VEC; ++v) {
    accd[0][v] = (double)acc2[0][v];
    accd[1][v] = (double)acc2[1][v];
  }
  if (col_reduce<VEC, 2>(accd, a.RP, a.red, a.col, &ctl->arrive)) {
    // the last block: add the pass to the sweep's per-column sums
    double *sw = a.col + 2 * RP, *prev = a.col + 4 * RP;
    for (int r = threadIdx.x; r < 2 * RP; r += kBlock) sw[r] += a.col[r];
    __syncthreads();
    if (threadIdx.x == 0) {
      if (last) {  // the sweep is complete: per-column decision
        const int t = ctl->round + 1;
        ctl->round = t;
        int notdone = 0;
        bool finite = true;
        for (int r = 0; r < RP; ++r) {
          const double dd = sw[r], xx = sw[RP + r], pv = prev[r];
          if (!isfinite(dd) || !isfinite(xx)) finite = false;
          double f2 = 1.0;
          if (t >= 3 && pv > 0.0) {
            const double q = sqrt(dd / pv);
            f2 = q < 0.8 ? fmax(1.0, (q / (1.0 - q)) * (q / (1.0 - q))) : 16.0;
          }
          if (xx > 0.0 && !(dd * f2 <= ctl->tol2bb * xx)) ++notdone;
          prev[r] = dd;
          sw[r] = 0.0;
          sw[RP + r] = 0.0;
        }
        ctl->rr = (double)notdone;
        if (!finite) {
          ctl->status = GABP_DIVERGED; ctl->iters = t; ctl->result_round = t; ctl->done = 1;
        } else if (t >= 2 && notdone == 0) {
          ctl->status = GABP_OK; ctl->iters = t; ctl->result_round = t; ctl->done = 1;
        } else if (t >= ctl->max_iter) {
          ctl->status = GABP_NOT_CONVERGED; ctl->iters = t; ctl->result_round = t; ctl->done = 1;
        }
      }
      ctl->arrive = 0;
      __threadfence();
    }
  }
}

template <int VEC>
__global__ void __launch_bounds__(kBlock, GABP_KBS_MINB) kbs_pass(ArgsBS a, int c, int skip0, int skipn) {
  DevCtl *ctl = a.ctl;
  if (ctl->done) return;
  const int RP = a.RP;
  const int cn = c + 1 == a.C ? 0 : c + 1;
  const int nv = a.n - skipn;
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * kBlock) >> 5;
  const int c0 = lane * VEC;
  float acc2[2][VEC];
#pragma unroll
  for (int v = 0; v < VEC; ++v) acc2[0][v] = acc2[1][v] = 0.f;
  for (int vr = warp; vr < nv; vr += nwarps) {
    const int j = vr < skip0 ? vr : vr + skipn;
    float hj[VEC], acc[VEC];
    ldv<VEC>(a.hfire + (size_t)j * RP + c0, hj);
#pragma unroll
    for (int v = 0; v < VEC; ++v) acc[v] = 0.f;
    const int s0 = a.co[(size_t)c * a.n + j], s1 = a.co[(size_t)(c + 1) * a.n + j];
    int e = s0;
    for (; e + kBsU <= s1; e += kBsU) {  // kBsU slots with their loads issued together
      int k[kBsU];
      float2 cf[kBsU];
      float hs[kBsU][VEC], hk[kBsU][VEC];
#pragma unroll
      for (int u = 0; u < kBsU; ++u) {
        k[u] = a.sci[e + u];
        cf[u] = a.sCF[e + u];
      }
#pragma unroll
      for (int u = 0; u < kBsU; ++u) {
        ldv_cs<VEC>(a.sH + (size_t)(e + u) * RP + c0, hs[u]);
        ldv<VEC>(a.hfire + (size_t)k[u] * RP + c0, hk[u]);
      }
#pragma unroll
      for (int u = 0; u < kBsU; ++u) {
        float hn[VEC];
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
          hn[v] = cf[u].x * (hk[u][v] - cf[u].y * (hj[v] - hs[u][v]));  // message k -> j, k firing now
          acc[v] += hn[v];                                              // (reverse message recomputed)
        }
        stv_cs<VEC>(a.sH + (size_t)(e + u) * RP + c0, hn);
      }
    }
    for (; e < s1; ++e) {
      const int k = a.sci[e];
      const float2 cf = a.sCF[e];
      float hs[VEC], hk[VEC], hn[VEC];
      ldv_cs<VEC>(a.sH + (size_t)e * RP + c0, hs);
      ldv<VEC>(a.hfire + (size_t)k * RP + c0, hk);
#pragma unroll
      for (int v = 0; v < VEC; ++v) {
        const float hout = cf.y * (hj[v] - hs[v]);  // message j -> k when j last fired
        hn[v] = cf.x * (hk[v] - hout);              // message k -> j, k firing now
        acc[v] += hn[v];
      }
      stv_cs<VEC>(a.sH + (size_t)e * RP + c0, hn);
    }
    if (a.scol[j] == cn) {  // j fires next: its aggregate over the whole row
      for (int e = a.srp[j]; e < s0; ++e) {
        float hs[VEC];
        ldv<VEC>(a.sH + (size_t)e * RP + c0, hs);
#pragma unroll
        for (int v = 0; v < VEC; ++v) acc[v] += hs[v];
      }
      for (int e = s1; e < a.srp[j + 1]; ++e) {
        float hs[VEC];
        ldv<VEC>(a.sH + (size_t)e * RP + c0, hs);
#pragma unroll
        for (int v = 0; v < VEC; ++v) acc[v] += hs[v];
      }
      float rh[VEC], hnew[VEC];
      ldv<VEC>(a.srhs + (size_t)j * RP + c0, rh);
      const float ip = a.sinvP[j];
#pragma unroll
      for (int v = 0; v < VEC; ++v) {
        hnew[v] = rh[v] + acc[v];
        const float x = hnew[v] * ip, dx = (hnew[v] - hj[v]) * ip;
        acc2[0][v] = fmaf(dx, dx, acc2[0][v]);
        acc2[1][v] = fmaf(x, x, acc2[1][v]);
      }
      stv<VEC>(a.hfire + (size_t)j * RP + c0, hnew);
    }
  }
  kbs_finish<VEC>(a, acc2, c == a.C - 1);
}

// Pass C of a sweep of two colours (grids, trees, the augmented least-squares systems), where a pass
// visits whole rows of the other colour and nothing else.  Only the messages into colour 1 are kept:
//   pass 0 (colour 0 fires, rows of colour 1)  as kbs_pass: the slot's own message, overwritten;
//   pass 1 (colour 1 fires, rows of colour 0)  the reverse message j -> k is the one pass 0 has just
//          stored in row k, read from there; the messages into colour 0 are used and not stored.
// A sweep moves three messages per pair of slots instead of four, and what a cavity takes out is the
// message its aggregate added, where c_out (hj - h) rounds it anew: after equal sweeps the error is smaller (64^3 grid, 16
// columns, 122 sweeps in two steps 2.6e-11 where kbs_pass has 3.4e-11, 182 sweeps 3.3e-14 and 4.3e-14), and
// the update's norm passes the stop as soon as the iteration has converged, while kbs_pass took 124 to 154 sweeps by
// the seed and ended at the smaller errors of the later sweeps.  The first sweep starts from zero
// messages: hfire of colour 1 is 0 and the store is not read.
template <int VEC, int PASS, bool START, int NU>
__device__ __forceinline__ void kbs2_slots(const ArgsBS &a, int e, int c0, const float (&hj)[VEC], float (&acc)[VEC]) {
  const int RP = a.RP;
  int k[NU], q[NU];
  float2 cf[NU];
  float hs[NU][VEC], hk[NU][VEC];
#pragma unroll
  for (int u = 0; u < NU; ++u) {
    k[u] = a.sci[e + u];
    cf[u] = a.sCF[e + u];
    q[u] = (PASS == 0 ? e + u : a.srev[e + u]) - a.e1;
  }
#pragma unroll
  for (int u = 0; u < NU; ++u) {
    if (!START || PASS == 1) ldv_cs<VEC>(a.sH + (size_t)q[u] * RP + c0, hs[u]);
    ldv<VEC>(a.hfire + (size_t)k[u] * RP + c0, hk[u]);
  }
#pragma unroll
  for (int u = 0; u < NU; ++u) {
    float hn[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
      const float hout = PASS == 1 ? hs[u][v] : START ? 0.f : cf[u].y * (hj[v] - hs[u][v]);
      hn[v] = cf[u].x * (hk[u][v] - hout);
      acc[v] += hn[v];
    }
    if (PASS == 0) stv_cs<VEC>(a.sH + (size_t)q[u] * RP + c0, hn);
  }
}

template <int VEC, int PASS, bool START>
__device__ __forceinline__ void kbs2_rows(const ArgsBS &a, int j0, int j1, float (&acc2)[2][VEC]) {
  constexpr int NU = VEC == 4 ? 2 : kBsU;
  const int RP = a.RP;
  const int c0 = (threadIdx.x & 31) * VEC;
  const int warp = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * kBlock) >> 5;
  for (int j = j0 + warp; j < j1; j += nwarps) {
    float hj[VEC], acc[VEC];
    ldv<VEC>(a.hfire + (size_t)j * RP + c0, hj);
#pragma unroll
    for (int v = 0; v < VEC; ++v) acc[v] = 0.f;
    int e = a.srp[j];
    const int e1 = a.srp[j + 1];
    for (; e + NU <= e1; e += NU) kbs2_slots<VEC, PASS, START, NU>(a, e, c0, hj, acc);
    for (; e < e1; ++e) kbs2_slots<VEC, PASS, START, 1>(a, e, c0, hj, acc);
    float rh[VEC], hnew[VEC];
    ldv<VEC>(a.srhs + (size_t)j * RP + c0, rh);
    const float ip = a.sinvP[j];
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
      hnew[v] = rh[v] + acc[v];
      const float x = hnew[v] * ip, dx = (hnew[v] - hj[v]) * ip;
      acc2[0][v] = fmaf(dx, dx, acc2[0][v]);
      acc2[1][v] = fmaf(x, x, acc2[1][v]);
    }
    stv<VEC>(a.hfire + (size_t)j * RP + c0, hnew);
  }
}

template <int VEC, int PASS>
__global__ void __launch_bounds__(kBlock, GABP_KBS_MINB) kbs2_pass(ArgsBS a) {
  DevCtl *ctl = a.ctl;
  if (ctl->done) return;
  float acc2[2][VEC];
#pragma unroll
  for (int v = 0; v < VEC; ++v) acc2[0][v] = acc2[1][v] = 0.f;
  const int j0 = PASS == 0 ? a.n1 : 0, j1 = PASS == 0 ? a.n : a.n1;
  if (PASS == 0 && ctl->round == 0) kbs2_rows<VEC, PASS, true>(a, j0, j1, acc2);
  else kbs2_rows<VEC, PASS, false>(a, j0, j1, acc2);
  kbs_finish<VEC>(a, acc2, PASS == 1);
}

// new-order rows of an [n][RP] FP32 array from the input order; the inner
// solve starts with h~ = r
// (rows from n1 on: with 0, they have not fired)
__global__ void kbs_init(int n, int n1, int RP, const int *__restrict__ oid, const float *__restrict__ rhs,
                         float *__restrict__ srhs, float *__restrict__ hfire) {
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * blockDim.x) >> 5;
  for (int j = warp; j < n; j += nwarps) {
    const size_t src = (size_t)oid[j] * RP, dst = (size_t)j * RP;
    for (int r = lane; r < RP; r += 32) {
      const float v = rhs[src + r];
      srhs[dst + r] = v;
      hfire[dst + r] = j < n1 ? v : 0.f;
    }
  }
}

// X[oid[j]][r] += h~_j^fire[r] / P~_j
__global__ void kbs_update(int n, int RP, const int *__restrict__ oid, const float *__restrict__ hfire,
                           const float *__restrict__ sinvP, double *__restrict__ X) {
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * blockDim.x) >> 5;
  for (int j = warp; j < n; j += nwarps) {
    const float ip = sinvP[j];
    const size_t src = (size_t)j * RP, dst = (size_t)oid[j] * RP;
    for (int r = lane; r < RP; r += 32) X[dst + r] += (double)(hfire[src + r] * ip);
  }
}

__global__ void kbs_ctl_reset(DevCtl *c, int max_iter, double tol2, double *col, int RP) {
  c->round = 0;
  c->done = 0;
  c->status = GABP_NOT_CONVERGED;
  c->iters = 0;
  c->result_round = 0;
  c->max_iter = max_iter;
  c->tol2bb = tol2;
  c->arrive = 0;
  c->no_stop = 0;
  for (int r = 2 * RP; r < 5 * RP; ++r) col[r] = 0.0;  // sweep sums and previous steps
}

__global__ void __launch_bounds__(kBlock) kb_max_degree(int n, const int *__restrict__ rp, unsigned *most) {
  unsigned d = 0;
  for (int i = blockIdx.x * kBlock + threadIdx.x; i < n; i += gridDim.x * kBlock) d = max(d, (unsigned)(rp[i + 1] - rp[i]));
  d = __reduce_max_sync(0xffffffffu, d);
  if ((threadIdx.x & 31) == 0) atomicMax(most, d);
}

__global__ void kb_ctl_reset(DevCtl *c, int max_iter, double tol2) {
  c->round = 0;
  c->done = 0;
  c->status = GABP_NOT_CONVERGED;
  c->iters = 0;
  c->result_round = 0;
  c->max_iter = max_iter;
  c->check_from = 1;
  c->stable = 0;
  c->tol2bb = tol2;
  c->arrive = 0;
  c->no_stop = 0;
}

}  // namespace

struct WorkB {
  int RP = 0;
  int max_deg = 0;  // longest row
  float *H = nullptr;
  float *NH[3] = {nullptr, nullptr, nullptr};
  float *rhs = nullptr;
  double *X = nullptr, *Bt = nullptr;
  double *red = nullptr, *col = nullptr;
  unsigned int *arrive = nullptr;
  cudaGraphExec_t graph = nullptr;
  long long graph_key = -1;
  float *sH = nullptr, *hfire = nullptr, *srhs = nullptr;  // serial schedule: [E][RP], [n][RP], [n][RP]
  cudaGraphExec_t sgraph = nullptr;
  long long sgraph_key = -1;
};

void free_wb(gabp_handle h) {
  WorkB *w = h->wb;
  if (!w) return;
  cudaFree(w->H);
  for (int j = 0; j < 3; ++j) cudaFree(w->NH[j]);
  cudaFree(w->rhs); cudaFree(w->X); cudaFree(w->Bt); cudaFree(w->red); cudaFree(w->col); cudaFree(w->arrive);
  cudaFree(w->sH); cudaFree(w->hfire); cudaFree(w->srhs);
  if (w->graph) cudaGraphExecDestroy(w->graph);
  if (w->sgraph) cudaGraphExecDestroy(w->sgraph);
  delete w;
  h->wb = nullptr;
}

static gabp_status ensure_wb(gabp_handle h, int RP) {
  if (h->wb && h->wb->RP == RP) return GABP_OK;
  free_wb(h);
  h->wb = new WorkB();
  WorkB *w = h->wb;
  const size_t n = (size_t)h->g.n;
  for (int j = 0; j < 3; ++j) GABP_CUDA(cudaMalloc(&w->NH[j], sizeof(float) * n * RP));
  GABP_CUDA(cudaMalloc(&w->rhs, sizeof(float) * n * RP));
  GABP_CUDA(cudaMalloc(&w->X, sizeof(double) * n * RP));
  GABP_CUDA(cudaMalloc(&w->Bt, sizeof(double) * n * RP));
  GABP_CUDA(cudaMalloc(&w->red, sizeof(double) * 2 * (size_t)h->max_blocks * RP));
  GABP_CUDA(cudaMalloc(&w->col, sizeof(double) * 5 * RP));
  GABP_CUDA(cudaMalloc(&w->arrive, sizeof(unsigned int)));
  GABP_CUDA(cudaMemsetAsync(w->arrive, 0, sizeof(unsigned int), h->stream));
  kb_max_degree<<<blocks_for(h->g.n, kBlock, h->max_blocks), kBlock, 0, h->stream>>>(h->g.n, h->g.rp, w->arrive);
  GABP_CUDA(cudaGetLastError());
  GABP_CUDA(cudaMemcpyAsync(&w->max_deg, w->arrive, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
  GABP_CUDA(cudaMemsetAsync(w->arrive, 0, sizeof(unsigned int), h->stream));
  GABP_CUDA(cudaStreamSynchronize(h->stream));
  w->RP = RP;
  return GABP_OK;
}

template <int VEC>
static gabp_status batched_chunk(gabp_handle h, int R, const double *B, double *X, int64_t ld, double tol,
                                 int max_iter, int *iters, double *relres_host, int *worst) {
  constexpr int RP = 32 * VEC;
  gabp_status s = ensure_wb(h, RP);
  if (s != GABP_OK) return s;
  WorkB &w = *h->wb;
  Graph &g = h->g;
  Work32 &w32 = h->w32;
  const size_t E = (size_t)(g.E > 0 ? g.E : 1);
  const size_t shmem = sizeof(double) * 2 * (kBlock / 32) * RP;
  // a full wave of one-warp-per-row blocks
  auto grid_of = [&](auto kern) {
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, kBlock, shmem) != cudaSuccess || nb < 1) {
      cudaGetLastError();
      nb = 1;
    }
    return blocks_for(g.n, kBlock / 32, nb * h->num_sms);
  };
  void (*const mean)(ArgsB) =
      VEC < 4 && long_row_round(g, w.max_deg, RP) ? kb_mean<VEC, VEC < 4 ? kBULong : kBU<VEC>> : kb_mean<VEC, kBU<VEC>>;
  const int nb_mean = grid_of(mean);
  const int nb_res = grid_of(kb_residual<VEC>);
  dim3 tb(32, 8), tg((g.n + 31) / 32, RP / 32);
  kb_gather_cols<<<tg, tb, 0, h->stream>>>(g.n, R, RP, B, ld, w.Bt);
  GABP_CUDA(cudaMemsetAsync(w.X, 0, sizeof(double) * g.n * RP, h->stream));
  kb_residual<VEC><<<nb_res, kBlock, shmem, h->stream>>>(g.n, RP, g.rowptr, g.col, g.val, w.Bt, w.X, w.rhs, w.NH[0],
                                                         w.red, w.col, w.arrive);
  h->prof.launches += 2;
  GABP_CUDA(cudaGetLastError());
  std::vector<double> colh(4 * RP);
  auto read_cols = [&]() -> gabp_status {
    GABP_CUDA(cudaMemcpyAsync(colh.data(), w.col, sizeof(double) * RP, cudaMemcpyDeviceToHost, h->stream));
    GABP_CUDA(cudaStreamSynchronize(h->stream));
    return GABP_OK;
  };
  if ((s = read_cols()) != GABP_OK) return s;
  std::vector<double> bb(R), rr(R);
  for (int r = 0; r < R; ++r) bb[r] = rr[r] = colh[r];
  ArgsB a;
  const bool serial = h->opt.schedule == 1;
  if (!serial && !w.H) GABP_CUDA(cudaMalloc(&w.H, sizeof(float) * E * RP));
  a.n = g.n; a.RP = RP; a.rp = g.rp; a.ci = g.ci; a.rev = g.rev; a.CF = w32.CF; a.invP = w32.invP;
  a.H = w.H; a.NH0 = w.NH[0]; a.NH1 = w.NH[1]; a.NH2 = w.NH[2];
  a.rhs = w.rhs; a.ctl = h->ctl; a.red = w.red; a.col = w.col;
  const double itol = h->opt.inner_tol;
  ArgsBS as;
  int nb_ser = 1, nb_two[2] = {1, 1};
  bool two = false;  // two colours
  if (serial) {
    if ((s = serial_freeze32(h, w32.CF, w32.invP)) != GABP_OK) return s;
    WorkS &ws = h->ws;
    two = ws.C == 2;
    as.n1 = two ? ws.cstart[1] : g.n;
    as.e1 = two ? ws.srp_h[as.n1] : 0;
    if (!w.sH) {
      GABP_CUDA(cudaMalloc(&w.sH, sizeof(float) * (E - as.e1) * RP));
      GABP_CUDA(cudaMalloc(&w.hfire, sizeof(float) * g.n * RP));
      GABP_CUDA(cudaMalloc(&w.srhs, sizeof(float) * g.n * RP));
    }
    as.n = g.n; as.C = ws.C; as.RP = RP; as.co = ws.co; as.sci = ws.sci; as.scol = ws.scol; as.srp = ws.srp;
    as.srev = ws.srev; as.sCF = ws.sCF; as.sinvP = ws.sinvP; as.srhs = w.srhs; as.sH = w.sH; as.hfire = w.hfire;
    as.ctl = h->ctl; as.red = w.red; as.col = w.col;
    nb_ser = grid_of(kbs_pass<VEC>);
    nb_two[0] = grid_of(kbs2_pass<VEC, 0>);
    nb_two[1] = grid_of(kbs2_pass<VEC, 1>);
  }
  int total_inner = 0;
  auto all_done = [&]() {
    for (int r = 0; r < R; ++r)
      if (bb[r] > 0.0 && !(rr[r] <= tol * tol * bb[r])) return false;
    return true;
  };
  bool diverged = false;
  for (int step = 0; step < h->opt.max_refine && !all_done() && total_inner < max_iter; ++step) {
    if (serial && !two) GABP_CUDA(cudaMemsetAsync(w.sH, 0, sizeof(float) * E * RP, h->stream));
    const int cap = std::min(h->opt.inner_max_iter, std::max(1, max_iter - total_inner));
    double worst_ratio = 0.0;  // the column furthest from its target sets the inner tolerance
    for (int r = 0; r < R; ++r)
      if (bb[r] > 0.0) worst_ratio = std::max(worst_ratio, rr[r] / bb[r]);
    const double it_tol = inner_target(itol, tol, 1.0, worst_ratio);
    if (serial) {
      WorkS &ws = h->ws;
      kbs_init<<<std::max(1, (g.n + 7) / 8), kBlock, 0, h->stream>>>(g.n, as.n1, RP, ws.oid, w.rhs, w.srhs,
                                                                             w.hfire);
      kbs_ctl_reset<<<1, 1, 0, h->stream>>>(h->ctl, cap, it_tol * it_tol, w.col, RP);
      h->prof.launches += 2;
      GABP_CUDA(cudaGetLastError());
      s = run_rounds(h, &w.sgraph, &w.sgraph_key, RP | (ws.C << 16), [&] {
        if (two) {
          kbs2_pass<VEC, 0><<<nb_two[0], kBlock, shmem, h->stream>>>(as);
          kbs2_pass<VEC, 1><<<nb_two[1], kBlock, shmem, h->stream>>>(as);
          return;
        }
        for (int c = 0; c < ws.C; ++c)
          kbs_pass<VEC><<<nb_ser, kBlock, shmem, h->stream>>>(as, c, ws.cstart[c], ws.cstart[c + 1] - ws.cstart[c]);
      }, cap, PH_MEAN32);
    } else {
      kb_ctl_reset<<<1, 1, 0, h->stream>>>(h->ctl, cap, it_tol * it_tol);
      h->prof.launches += 1;
      GABP_CUDA(cudaGetLastError());
      s = run_rounds(h, &w.graph, &w.graph_key, RP, [&] { mean<<<nb_mean, kBlock, shmem, h->stream>>>(a); },
                     cap, PH_MEAN32);
    }
    if (s != GABP_OK) return s;
    const DevCtl c = *h->ctl_host;
    total_inner += c.round;
    h->stats.rounds += c.round;
    h->stats.edge_updates += (int64_t)c.round * g.E * R;
    if (c.status == GABP_DIVERGED) { diverged = true; break; }
    float *hT = w.NH[c.result_round % 3];
    prof_begin(h);
    if (serial)
      kbs_update<<<std::max(1, (g.n + 7) / 8), kBlock, 0, h->stream>>>(g.n, RP, h->ws.oid, w.hfire, h->ws.sinvP, w.X);
    else
      kb_update<VEC><<<std::max(1, (g.n + 7) / 8), kBlock, 0, h->stream>>>(g.n, RP, w.X, hT, w32.invP);
    kb_residual<VEC><<<nb_res, kBlock, shmem, h->stream>>>(g.n, RP, g.rowptr, g.col, g.val, w.Bt, w.X, w.rhs,
                                                           w.NH[0], w.red, w.col, w.arrive);
    prof_end(h);
    h->prof.launches += 2;
    GABP_CUDA(cudaGetLastError());
    if ((s = read_cols()) != GABP_OK) return s;
    prof_collect(h, PH_REFINE64, 1);
    h->stats.refine_steps += 1;
    for (int r = 0; r < R; ++r) {
      rr[r] = colh[r];
      if (!std::isfinite(rr[r])) diverged = true;
    }
    if (diverged) break;
  }
  dim3 sg((g.n + 31) / 32, RP / 32);
  kb_scatter_cols<<<sg, tb, 0, h->stream>>>(g.n, R, RP, w.X, X, ld);
  h->prof.launches += 1;
  GABP_CUDA(cudaGetLastError());
  GABP_CUDA(cudaStreamSynchronize(h->stream));
  int st = GABP_OK;
  for (int r = 0; r < R; ++r) {
    const double rel = bb[r] > 0.0 ? std::sqrt(rr[r] / bb[r]) : 0.0;
    if (relres_host) relres_host[r] = rel;
    if (diverged) st = std::max(st, (int)GABP_DIVERGED);
    else if (bb[r] > 0.0 && !(rr[r] <= tol * tol * bb[r])) st = std::max(st, (int)GABP_NOT_CONVERGED);
  }
  *worst = std::max(*worst, st);
  *iters += total_inner;
  return GABP_OK;
}

gabp_status solve_batched32(gabp_handle h, int nrhs, const double *B, double *X, int64_t ld, double tol,
                            int max_iter, int *iters, double *relres_host) {
  NvtxRange nvtx_("gabp batched right-hand sides");
  if (nrhs < 1 || ld < h->g.n) return GABP_ERR_INVALID;
  gabp_status s = ensure_w32(h, 1);
  if (s != GABP_OK) return s;
  h->stats.rounds = 0;
  h->stats.edge_updates = 0;
  h->stats.refine_steps = 0;
  if (h->opt.reuse_precisions && (s = csr_coef32(h)) != GABP_OK) return s;
  if (!h->w32.coef_ready || !h->opt.reuse_precisions) {
    drop_coef32(h);
    if ((s = precision_phase32(h, nullptr)) != GABP_OK) return s;
    h->stats.edge_updates += h->stats.rounds * (int64_t)h->g.E;  // precision rounds serve every column
  }
  int worst = GABP_OK, total = 0;
  for (int r0 = 0; r0 < nrhs; r0 += 128) {
    const int R = std::min(128, nrhs - r0);
    const double *Bc = B + (size_t)r0 * ld;
    double *Xc = X + (size_t)r0 * ld;
    double *rel = relres_host ? relres_host + r0 : nullptr;
    if (R <= 32) s = batched_chunk<1>(h, R, Bc, Xc, ld, tol, max_iter, &total, rel, &worst);
    else if (R <= 64) s = batched_chunk<2>(h, R, Bc, Xc, ld, tol, max_iter, &total, rel, &worst);
    else s = batched_chunk<4>(h, R, Bc, Xc, ld, tol, max_iter, &total, rel, &worst);
    if (s != GABP_OK) return s;
  }
  if (iters) *iters = total;
  h->last_path = 1;
  return (gabp_status)worst;
}

}  // namespace gabp
