// multichip.cu -- many independent systems, each solved from its first round to its last by one SM that
// takes it from a queue, with the node aggregates in shared memory.
//
// A global round of the grid-persistent kernels (multigrid.cu) streams every running system's slots, gathers each
// slot's sender through L2 (one request a slot, as many as the streams need together) and ends at a grid
// barrier.  Here a system belongs to one CTA with the aggregates of the last two rounds in its shared
// memory: gathers are shared-memory loads, the round's barrier is the CTA's own, and what streams is the
// slots alone, 18 bytes each (coefficients 8, sender position 2, message read and write 8).  A warp
// fetches the chunks of its slices by bulk copies into its part of a ring, several ahead (one SM's share of
// the HBM rate times the copies' ~1.8 us of latency is 80 KB in flight), into the next round too: what
// that round streams was written a round ago.
// Bound by HBM when every SM has a system (152 graphs of 16384 rows and degree 6: 54 us a round, 5.9 TB/s of
// slots and row vectors; the grid-persistent kernel 138), by one SM's rate of 2.4 ns a row of degree 6 and round when
// few have.  Systems above kTRowsMost rows go to the grid-persistent kernel.  512 geometric graphs of 1024
// to 65536 rows to 1e-10: 22.0 -> 16.0 ms, 9 of it for the 38 largest on the grid-persistent kernel.
//
// Rows are addressed by position (slice, lane) of the sliced layout within their system, so own rows'
// accesses are contiguous; padding slots hold zero coefficients, padding rows a unit precision and a zero
// right-hand side.  The rounds, decisions and their order are multigrid.cu's (precision rounds,
// coefficients, FP64 residual, inner rounds, update), each system on its own.
#include "sell64.cuh"

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

namespace gabp {

namespace {

constexpr int kTThreads = 512, kTWarps = kTThreads / 32;
constexpr int kTPrecCap = 300;       // precision-round cap per system (multigrid.cu's)
constexpr int kTU = 4;               // lines of a chunk; slots per lane whose loads are issued together
// A mean round's slots come in chunks of up to kTU lines of 32 slots, each line {c_in, c_out} 256 bytes,
// sender positions 64, messages 128; a chunk's coefficient lines and then its position lines lie together
// (kChunkCF bytes for a full one), the messages in their chain.
constexpr int kLineCF = 320, kLineH = 128, kChunkCF = kTU * kLineCF, kStageBytes = kChunkCF + kTU * kLineH;
constexpr size_t kTSmem = 227328;    // dynamic shared memory of a CTA (222 KB): chunk ring, slice table, aggregates
constexpr int kStagesMin = 3, kStagesMax = 7;  // chunks of a warp in the ring: what the aggregates leave room for
// positions of the largest system: aggregates of two rounds and the slice table, 8 1/4 bytes each, beside the
// smallest ring
constexpr int kTRowsMost = (int)((kTSmem - (size_t)kTWarps * kStagesMin * kStageBytes - 64) / 33 * 4 / 32 * 32);
constexpr long long kTWaitLimit = 4000000000LL;  // clock cycles (~2 s) before a wait gives up

struct TeamArgs {
  const int *__restrict__ srow;              // [32 ns] row of each position, -1 for padding
  const int *__restrict__ sp;                // [ns + 1] first slot of each slice
  const int2 *__restrict__ sys;              // [nsys] first slice and slices of each system
  unsigned char *blk;                        // [10 Es] chunks of coefficients and sender positions
  const float *__restrict__ av;              // [Es]
  const float *__restrict__ adp;             // [32 ns] A_ii by position (1 for padding)
  const int *__restrict__ rowptr;
  const int *__restrict__ col;
  const double *__restrict__ val;
  float *MP0, *MP1, *H0, *H1;                // [Es] precision and mean chains
  float *rhsp, *invPp;                       // [32 ns] by position
  const double *b;
  double *x;
  const int *order;                          // systems by descending size
  int njobs;
  int *queue;                                // [0] next system, [1] a wait gave up
  int *status, *iters, *refine;
  double *relres;
  double tol, inner_tol, prec_thr;
  int inner_max, max_refine, max_iter;
};

__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long *bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned long long *bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_load(void *dst, const void *src, unsigned bytes, unsigned long long *bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}
__device__ __forceinline__ bool mbar_done(unsigned long long *bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Waits for the phase; gives up after kTWaitLimit, or at once when another wait has, and raises *err.
__device__ __noinline__ void mbar_wait_slow(unsigned long long *bar, unsigned parity, int *err) {
  const long long t0 = clock64();
  while (!mbar_done(bar, parity)) {
    if (*(volatile int *)err || clock64() - t0 > kTWaitLimit) {
      atomicExch(err, 1);
      return;
    }
  }
}
// This thread's writes to global memory come before later bulk copies (another proxy) by the CTA.
__device__ __forceinline__ void fence_bulk() { asm volatile("fence.proxy.async;" ::: "memory"); }

// What a precision round's flags decide, the same bits in every thread.
struct TeamFlags {
  unsigned m, f;
};

// A positive factor as m 2^e with the top bit of m set (m = 0: zero).
struct TeamFactor {
  unsigned long long m;
  int e;
};

struct TeamShared {
  float2 part[2][kTWarps];
  uint2 flag[2][kTWarps];
  double rr[kTWarps];
  TeamFactor tol2;  // the inner solve's squared tolerance
  int job;
  unsigned long long bar[kTWarps][kStagesMax];  // one phase per chunk
  TeamArgs args;  // the launch's arguments, read from here in the solves
};

// Posts this thread's flags, passes the CTA's barrier, and joins what all warps posted.
__device__ __forceinline__ TeamFlags team_flags(TeamShared &sh, int parity, unsigned m, unsigned f) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  m = __reduce_max_sync(0xffffffffu, m);
  f = __reduce_or_sync(0xffffffffu, f);
  if (lane == 0) sh.flag[parity][w] = make_uint2(m, f);
  __syncthreads();
  const uint2 g = lane < kTWarps ? sh.flag[parity][lane] : make_uint2(0u, 0u);
  return TeamFlags{__reduce_max_sync(0xffffffffu, g.x), __reduce_or_sync(0xffffffffu, g.y)};
}

// A sum over the warps of their FP32 values (not negative), on the integer units: the 24-bit significands are
// aligned to the largest value's, 32 bits below its last place kept, and added exactly: s 2^(e - 182).  A sum
// over a whole system overflows FP32 long before its entries do, and FP64 additions hold a scheduler 64 cycles
// each (one warp's, with a second barrier: 0.4 to 0.8 us a round of 10 to 45).
struct TeamSum {
  unsigned long long s;
  int e;  // 255: a value is not finite
};
__device__ __forceinline__ TeamSum team_sum(float v) {
  const unsigned u = __float_as_uint(v) & 0x7fffffffu;
  const int em = max(1, (int)(__reduce_max_sync(0xffffffffu, u) >> 23)), eu = max(1, (int)(u >> 23));
  const unsigned long long m = (u & 0x7fffffu) | (u >= 0x800000u ? 0x800000u : 0u);
  const unsigned long long x = em - eu < 56 ? (m << 32) >> (em - eu) : 0ull;  // below 2^56
  const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)x & 0xfffffffu);
  const unsigned hi = __reduce_add_sync(0xffffffffu, (unsigned)(x >> 28));
  return TeamSum{lo + ((unsigned long long)hi << 28), em};
}

// f as a factor.
__device__ __forceinline__ TeamFactor team_factor(double f) {
  if (!(f > 0.0)) return TeamFactor{0ull, 0};
  int e;
  const double r = frexp(f, &e);  // f = r 2^e, r in [1/2, 1)
  return TeamFactor{(unsigned long long)(r * 0x1p53) << 11, e - 64};
}
// a <= f b, to 2^-62.
__device__ __forceinline__ bool team_below(const TeamSum &a, const TeamFactor &f, const TeamSum &b) {
  if (a.s == 0ull) return true;
  if (b.s == 0ull || f.m == 0ull) return false;
  const int la = __clzll((long long)a.s), lb = __clzll((long long)b.s);
  const unsigned long long A = a.s << la;
  unsigned long long P = __umul64hi(f.m, b.s << lb);  // f b = P 2^64 at b's exponent, less lb, and f's
  int ep = 64 + f.e + b.e - lb;
  if (!(P >> 63)) {
    P <<= 1;
    --ep;
  }
  const int ea = a.e - la;
  return ea != ep ? ea < ep : A <= P;
}

// The decision from all warps' sums p; out of line, to leave the rounds their registers.
__device__ __noinline__ int team_decide(float2 p, const TeamFactor &f) {
  const TeamSum a = team_sum(p.x), b = team_sum(p.y);
  return (a.e >= 255 || b.e >= 255 ? 1 : 0) | (team_below(a, f, b) ? 2 : 0);
}

// Posts this thread's squared update and iterate, passes the CTA's barrier, and decides: bit 0 a sum is not
// finite, bit 1 the update is small against the iterate.  Most rounds are far from that, which FP32 sums of the 16
// values tell (16 2^-24 off; the bound is 2^-16 wide, and values near FP32's smallest go the exact way).
// The tolerance is sh.tol2; above: an FP32 value 2^-16 above it.
__device__ __forceinline__ int team_stop(TeamShared &sh, int parity, float va, float vb, float above) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  va = warp_sum(va);
  vb = warp_sum(vb);
  if (lane == 0) sh.part[parity][w] = make_float2(va, vb);
  __syncthreads();
  const float2 p = lane < kTWarps ? sh.part[parity][lane] : make_float2(0.f, 0.f);
  const float fa = warp_sum(p.x), fb = warp_sum(p.y);
  if (isfinite(fa) && isfinite(fb) && fa > 0x1p-100f && fa > above * fb) return 0;
  return team_decide(p, sh.tol2);
}

__device__ __forceinline__ double team_sum64(TeamShared &sh, double v) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  v = warp_sum(v);
  if (lane == 0) sh.rr[w] = v;
  __syncthreads();
  const double t = warp_sum(lane < kTWarps ? sh.rr[lane] : 0.0);
  __syncthreads();  // sh.rr is posted again only after every reader is done
  return t;
}

// One system's solve.  phases: the next phase's parity of each of this warp's barriers, a bit each.
__device__ __noinline__ unsigned team_solve(TeamShared &sh, unsigned char *smem, int sys, unsigned phases) {
  const TeamArgs &a = sh.args;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int s0 = a.sys[sys].x, ns = a.sys[sys].y, np = 32 * ns;
  const int base = 32 * s0, slot0 = a.sp[s0];
  int2 *meta = reinterpret_cast<int2 *>(smem);                 // slices: first slot (from slot0), width
  const int nmeta = (ns + 1) / 2 * 2;                           // even: what follows is 16-byte aligned
  float *const h0 = reinterpret_cast<float *>(meta + nmeta), *const h1 = h0 + np;  // aggregates, even / odd rounds
  const size_t used = sizeof(int2) * nmeta + sizeof(float) * 2 * np;
  const int S = min(kStagesMax, (int)((kTSmem - used) / ((size_t)kTWarps * kStageBytes)));
  unsigned char *const ringw = reinterpret_cast<unsigned char *>(h1 + np) + (size_t)w * S * kStageBytes;
  unsigned long long *const bar = sh.bar[w];
  float *const rhs = a.rhsp + base, *const invP = a.invPp + base;
  unsigned char *const blk = a.blk + (size_t)10 * slot0;
  const float *__restrict__ av = a.av + slot0;
  for (int m = threadIdx.x; m < ns; m += kTThreads)
    meta[m] = make_int2(a.sp[s0 + m] - slot0, (a.sp[s0 + m + 1] - a.sp[s0 + m]) >> 5);
  // line j of a slice of width wd from slot q: its coefficients, its senders
  auto cf_line = [&](int q, int j) { return blk + (size_t)10 * q + (j / kTU) * kChunkCF + (j % kTU) * 256; };
  auto k_line = [&](int q, int j, int wd) {
    return blk + (size_t)10 * q + (j / kTU) * kChunkCF + min(kTU, wd - j / kTU * kTU) * 256 + (j % kTU) * 64;
  };
  int parity = 0;
  int status = GABP_NOT_CONVERGED, steps = 0, inner = 0, Tp = 0;
  double rr = 0.0, bb = 0.0;
  // round 0: P~ = A_ii, no messages; x = 0
  for (int p = threadIdx.x; p < np; p += kTThreads) {
    const int i = a.srow[base + p];
    h0[p] = a.adp[base + p];
    if (i >= 0) a.x[i] = 0.0;
  }
  __syncthreads();

  // Precision round t; ZERO: the chain's message of round t - 2 is zero (rounds 1 and 2).
  auto prec_round = [&](int t, auto zero) {
    constexpr bool ZERO = decltype(zero)::value;
    float *__restrict__ Mc = ((t & 1) ? a.MP1 : a.MP0) + slot0;
    const float *__restrict__ Mo = ((t & 1) ? a.MP0 : a.MP1) + slot0;
    const float *hp = (t & 1) ? h0 : h1;
    float *hn = (t & 1) ? h1 : h0;  // holds round t - 2 of the own rows until they are written
    unsigned bad = 0, rel = 0;
    for (int m = w; m < ns; m += kTWarps) {
      const int p = 32 * m + lane;
      const int2 mt = meta[m];
      const int q0 = mt.x + lane;
      const float Pi2 = t >= 2 ? hn[p] : 0.f, ad = a.adp[base + p];
      float acc = 0.f;
      for (int j = 0; j < mt.y; j += kTU) {
        int k[kTU];
        float A[kTU], Ps[kTU], Pp[kTU];
#pragma unroll
        for (int u = 0; u < kTU; ++u)
          if (j + u < mt.y) {
            const int pos = q0 + 32 * (j + u);
            k[u] = __ldcs(reinterpret_cast<const unsigned short *>(k_line(mt.x, j + u, mt.y)) + lane);
            A[u] = __ldcs(av + pos);
            Ps[u] = ZERO ? 0.f : __ldcs(Mc + pos);
            Pp[u] = ZERO && t == 1 ? 0.f : __ldcs(Mo + pos);
          }
#pragma unroll
        for (int u = 0; u < kTU; ++u)
          if (j + u < mt.y) {
            const float A2 = A[u] * A[u];
            float Pout = 0.f;
            if (t >= 2) {
              const float d1 = Pi2 - Ps[u];
              bad |= (d1 == 0.f);
              Pout = -__fdividef(A2, d1);
            }
            const float d2 = hp[k[u]] - Pout;
            bad |= (d2 == 0.f);
            const float Pn = -__fdividef(A2, d2);
            __stcs(Mc + q0 + 32 * (j + u), Pn);
            acc += Pn;
            const float dP = fabsf(Pn - Pp[u]);  // >= 0 or NaN: the bit patterns order as the values
            rel = max(rel, __float_as_uint(dP == 0.f ? 0.f : fabsf(__fdividef(dP, Pn))));
          }
      }
      const float P = ad + acc;
      bad |= (P == 0.f);
      hn[p] = P;
    }
    parity ^= 1;
    return team_flags(sh, parity, rel & 0x7fffffffu, bad);
  };

  // The fetch cursor over this warp's chunks: slice and chunk of it (an empty slice has one, of no lines),
  // round; the ring's stages to fill and to use next and how many are on their way.
  int pm = w, pc = 0, ft = 1, sf = 0, su = 0, out = 0;
  // Fetches the next chunk, if it lies in a round up to tmax; false if not.
  auto fetch = [&](int tmax) {
    if (w >= ns || ft > tmax) return false;
    const int2 mt = meta[pm];
    const bool zero = ft <= 2;
    if (lane == 0) {
      const unsigned lines = (unsigned)min(kTU, mt.y - pc * kTU);
      unsigned char *dst = ringw + sf * kStageBytes;
      mbar_expect(bar + sf, lines * (zero ? kLineCF : kLineCF + kLineH));
      if (lines) {
        bulk_load(dst, blk + (size_t)10 * mt.x + pc * kChunkCF, lines * kLineCF, bar + sf);
        if (!zero)
          bulk_load(dst + kChunkCF, ((ft & 1) ? a.H1 : a.H0) + slot0 + mt.x + 32 * kTU * pc, lines * kLineH, bar + sf);
      }
    }
    sf = sf + 1 == S ? 0 : sf + 1;
    ++out;
    if (++pc * kTU >= mt.y) {
      pc = 0;
      pm += kTWarps;
      if (pm >= ns) { pm = w; ++ft; }
    }
    return true;
  };
  // Waits for the chunk to use next; it is given back by release().
  auto arrive = [&]() {
    const unsigned ph = (phases >> su) & 1u;
    if (!mbar_done(bar + su, ph)) mbar_wait_slow(bar + su, ph, a.queue + 1);
  };
  auto release = [&]() {
    phases ^= 1u << su;
    su = su + 1 == S ? 0 : su + 1;
    --out;
    __syncwarp();  // every lane has read the stage before it is filled again
  };

  auto mean_round = [&](int t, float above, auto zero) {
    constexpr bool ZERO = decltype(zero)::value;
    float *__restrict__ Hc = ((t & 1) ? a.H1 : a.H0) + slot0;
    const float *hp = (t & 1) ? h0 : h1;
    float *hn = (t & 1) ? h1 : h0;
    float dxx = 0.f, xx = 0.f;
    while (out < S && fetch(t + 1)) {}
    float rh = 0.f, ip = 0.f;
    if (w < ns) {
      rh = rhs[32 * w + lane];
      ip = invP[32 * w + lane];
    }
    for (int m = w; m < ns; m += kTWarps) {
      const int p = 32 * m + lane;
      const int2 mt = meta[m];
      float rh2 = 0.f, ip2 = 0.f;  // the next slice's, on their way
      if (m + kTWarps < ns) {
        rh2 = rhs[p + 32 * kTWarps];
        ip2 = invP[p + 32 * kTWarps];
      }
      const float hi2 = t >= 2 ? hn[p] : 0.f, hprev = hp[p];
      float acc = 0.f;
      int j = 0;
      do {
        const int lines = min(kTU, mt.y - j);
        arrive();
        const unsigned char *src = ringw + su * kStageBytes;
        const float2 *cfs = reinterpret_cast<const float2 *>(src) + lane;
        const unsigned short *ks = reinterpret_cast<const unsigned short *>(src + lines * 256) + lane;
        const float *hcs = reinterpret_cast<const float *>(src + kChunkCF) + lane;
        float hk[kTU];
#pragma unroll
        for (int u = 0; u < kTU; ++u)
          if (u < lines) hk[u] = hp[ks[32 * u]];
#pragma unroll
        for (int u = 0; u < kTU; ++u)
          if (u < lines) {
            const float2 cf = cfs[32 * u];
            const float hout = t >= 2 ? cf.y * (hi2 - (ZERO ? 0.f : hcs[32 * u])) : 0.f;
            const float hm = cf.x * (hk[u] - hout);
            __stcs(Hc + mt.x + 32 * (j + u) + lane, hm);
            acc += hm;
          }
        release();
        fetch(t + 1);
        j += kTU;
      } while (j < mt.y);
      const float hnew = rh + acc, dx = (hnew - hprev) * ip, x = hnew * ip;
      hn[p] = hnew;
      dxx = fmaf(dx, dx, dxx);
      xx = fmaf(x, x, xx);
      rh = rh2;
      ip = ip2;
    }
    fence_bulk();  // the messages written here are fetched for round t + 2, from the next round on
    parity ^= 1;
    return team_stop(sh, parity, dxx, xx, above);
  };

  bool run = true;
  {
    int stable = 0;
    for (int t = 1;; ++t) {
      const TeamFlags r = t <= 2 ? prec_round(t, std::true_type()) : prec_round(t, std::false_type());
      const float rel = __uint_as_float(r.m);
      stable = (double)rel <= a.prec_thr ? stable + 1 : 0;  // a NaN is not stationary
      Tp = t;
      if (r.f) { status = GABP_BREAKDOWN; run = false; break; }
      if (!(rel <= 1e30f)) { status = GABP_DIVERGED; run = false; break; }
      if (stable >= 2 || t >= kTPrecCap) break;
    }
  }
  if (run) {  // frozen coefficients; padding slots give zeros
    const float *Ms = ((Tp & 1) ? a.MP1 : a.MP0) + slot0;
    const float *hp = (Tp & 1) ? h1 : h0;
    for (int m = w; m < ns; m += kTWarps) {
      const int p = 32 * m + lane;
      const int2 mt = meta[m];
      const float Pi = hp[p];
#pragma unroll 4
      for (int j = 0; j < mt.y; ++j) {
        const int pos = mt.x + lane + 32 * j;
        const int k = reinterpret_cast<const unsigned short *>(k_line(mt.x, j, mt.y))[lane];
        const float A = av[pos];
        const float cout = -A / (Pi - Ms[pos]);
        const float cin = -A / (hp[k] - cout * A);
        reinterpret_cast<float2 *>(cf_line(mt.x, j))[lane] = make_float2(cin, cout);
      }
      invP[p] = 1.f / Pi;
    }
    fence_bulk();  // the coefficients are fetched by the mean rounds
    __syncthreads();
  }
  while (run) {
    // r = b - A x in FP64 (x = 0 at first: r = b)
    double v = 0.0;
    for (int p = threadIdx.x; p < np; p += kTThreads) {
      const int i = a.srow[base + p];
      float rf = 0.f;
      if (i >= 0) {
        double ax = 0.0;
        if (steps > 0) {
          const int e1 = a.rowptr[i + 1];
#pragma unroll 4
          for (int e = a.rowptr[i]; e < e1; ++e) ax = fma(a.val[e], __ldcg(a.x + a.col[e]), ax);
        }
        const double r = a.b[i] - ax;
        rf = (float)r;
        v = fma(r, r, v);
      }
      rhs[p] = rf;
      h0[p] = rf;
    }
    rr = team_sum64(sh, v);
    if (steps == 0) bb = rr;
    if (bb == 0.0 || rr <= a.tol * a.tol * bb) { status = GABP_OK; break; }
    if (!isfinite(rr)) { status = GABP_DIVERGED; break; }
    if (steps >= a.max_refine || inner >= a.max_iter) { status = GABP_NOT_CONVERGED; break; }
    const double itol = fmin(a.inner_tol, fmax(1e-6, 0.1 * a.tol * sqrt(bb / rr)));
    const float it2 = fmaxf((float)(itol * itol), 0x1p-126f) * (1.f + 0x1p-16f);  // and a little above it
    if (threadIdx.x == 0) sh.tol2 = team_factor(itol * itol);
    const int cap = min(a.inner_max, max(1, a.max_iter - inner));
    int t = 1;
    bool ok = true;
    pm = w; pc = 0; ft = 1;
    for (;; ++t) {
      const int r = t <= 2 ? mean_round(t, it2, std::true_type()) : mean_round(t, it2, std::false_type());
      if (r & 1) { ok = false; break; }
      if ((t >= 2 && (r & 2)) || t >= cap) break;
    }
    while (out > 0) {  // chunks fetched for a round that does not come
      arrive();
      release();
    }
    inner += t;
    if (!ok) { status = GABP_DIVERGED; break; }
    const float *hp = (t & 1) ? h1 : h0;
    for (int p = threadIdx.x; p < np; p += kTThreads) {
      const int i = a.srow[base + p];
      if (i >= 0) a.x[i] += (double)(hp[p] * invP[p]);
    }
    steps += 1;
    __syncthreads();  // the next residual gathers x
  }
  if (threadIdx.x == 0) {
    a.status[sys] = status;
    a.iters[sys] = Tp + inner;
    a.refine[sys] = steps;
    a.relres[sys] = bb > 0.0 ? sqrt(rr / bb) : 0.0;
  }
  __syncthreads();  // the shared memory is free for the next system
  return phases;
}

__global__ void __launch_bounds__(kTThreads, 1) kt_solve(TeamArgs args) {
  extern __shared__ __align__(128) unsigned char tbuf[];
  __shared__ TeamShared sh;
  if (threadIdx.x == 0) sh.args = args;
  if (threadIdx.x < kTWarps * kStagesMax) mbar_init(&sh.bar[0][0] + threadIdx.x);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  fence_bulk();
  __syncthreads();
  unsigned phases = 0;
  for (;;) {
    if (threadIdx.x == 0) sh.job = atomicAdd(sh.args.queue, 1);
    __syncthreads();
    const int job = sh.job;
    __syncthreads();
    if (job >= sh.args.njobs) break;
    phases = team_solve(sh, tbuf, sh.args.order[job], phases);
  }
}

// Position in its system of every row; the chunks' sender positions; A_ii by position.
__global__ void kt_positions(int nq, const int *__restrict__ srow, const int *__restrict__ ssys,
                             const int2 *__restrict__ sys, int *__restrict__ posof) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nq) return;
  const int i = srow[q];
  if (i >= 0) posof[i] = q - 32 * sys[ssys[q >> 5]].x;
}
__global__ void kt_slots(int nq, const int *__restrict__ sp, const int *__restrict__ ssys,
                         const int2 *__restrict__ sys, const int *__restrict__ sci, const int *__restrict__ posof,
                         unsigned char *__restrict__ blk) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nq) return;
  const int sl = q >> 5, own = q - 32 * sys[ssys[sl]].x, lane = q & 31;
  const int wd = (sp[sl + 1] - sp[sl]) >> 5;
  unsigned char *b = blk + (size_t)10 * sp[sl];
  for (int j = 0; j < wd; ++j) {
    const int k = sci[sp[sl] + 32 * j + lane], c = j / kTU, lines = min(kTU, wd - c * kTU);
    reinterpret_cast<unsigned short *>(b + c * kChunkCF + lines * 256 + (j % kTU) * 64)[lane] =
        (unsigned short)(k >= 0 ? posof[k] : own);
  }
}
__global__ void kt_diag(int nq, const int *__restrict__ srow, const double *__restrict__ ad, float *__restrict__ adp) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < nq) adp[q] = srow[q] >= 0 ? (float)ad[srow[q]] : 1.f;
}

}  // namespace

void free_team(TeamSell &t) {
  cudaFree(t.sys); cudaFree(t.blk); cudaFree(t.adp); cudaFree(t.node); cudaFree(t.order);
  t = TeamSell{};
}

// Systems of at most this many rows can be solved by one SM each (0: not on this device).
int team_rows(gabp_handle h) {
  int optin = 0;
  cudaFuncAttributes fa;
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, h->device);
  if (cudaFuncGetAttributes(&fa, kt_solve) != cudaSuccess || kTSmem + fa.sharedSizeBytes > (size_t)optin) {
    cudaGetLastError();
    return 0;
  }
  return kTRowsMost;
}

// Solves the systems from place `from` of the layout's order on (at most kTRowsMost rows each).
gabp_status solve_systems_team(gabp_handle h, int nsys, const int *off, int from, const double *b, double *x, double tol,
                               int max_iter, int *d_status, int *d_iters, int *d_refine, double *d_relres,
                               float *ms_out) {
  gabp_status st = ensure_gsell(h, nsys, off, true);
  if (st != GABP_OK) return st;
  Graph &g = h->g;
  GSell *L = h->gsl;
  TeamSell &T = L->team;
  const int nq = 32 * L->ns, nb = (nq + kBlock - 1) / kBlock;
  if (off[L->order[from] + 1] - off[L->order[from]] > kTRowsMost) {
    set_last_error("gabp_solve_systems: a system is too large for one SM");
    return GABP_ERR_INVALID;
  }
  if (T.njobs != nsys - from) {
    free_team(T);
    std::vector<int2> sys(nsys);
    int s0 = 0;
    for (int s : L->order) {
      sys[s] = make_int2(s0, (off[s + 1] - off[s] + 31) / 32);
      s0 += sys[s].y;
    }
    int *posof = nullptr;
    GABP_CUDA(cudaMalloc(&posof, sizeof(int) * g.n));
    struct F {
      int *p;
      ~F() { cudaFree(p); }
    } fr{posof};
    GABP_CUDA(cudaMalloc(&T.sys, sizeof(int2) * nsys));
    GABP_CUDA(cudaMalloc(&T.order, sizeof(int) * (nsys + 2)));
    GABP_CUDA(cudaMalloc(&T.blk, (size_t)10 * std::max(L->Es, 32)));
    GABP_CUDA(cudaMalloc(&T.adp, sizeof(float) * nq));
    GABP_CUDA(cudaMalloc(&T.node, sizeof(float) * 2 * (size_t)nq));
    GABP_CUDA(cudaMemcpyAsync(T.sys, sys.data(), sizeof(int2) * nsys, cudaMemcpyHostToDevice, h->stream));
    GABP_CUDA(cudaMemcpyAsync(T.order, L->order.data() + from, sizeof(int) * (nsys - from), cudaMemcpyHostToDevice,
                              h->stream));
    kt_positions<<<nb, kBlock, 0, h->stream>>>(nq, L->srow, L->ssys, T.sys, posof);
    kt_slots<<<nb, kBlock, 0, h->stream>>>(nq, L->sp, L->ssys, T.sys, L->sci, posof, T.blk);
    GABP_CUDA(cudaGetLastError());
    GABP_CUDA(cudaStreamSynchronize(h->stream));
    T.njobs = nsys - from;
  }
  TeamArgs a;
  a.srow = L->srow; a.sp = L->sp; a.sys = T.sys; a.blk = T.blk; a.av = L->sav; a.adp = T.adp;
  a.rowptr = g.rowptr; a.col = g.col; a.val = g.val;
  a.MP0 = L->MP[0]; a.MP1 = L->MP[1]; a.H0 = L->H[0]; a.H1 = L->H[1];
  a.rhsp = T.node; a.invPp = T.node + nq;
  a.b = b; a.x = x;
  a.order = T.order; a.njobs = T.njobs; a.queue = T.order + nsys;
  a.status = d_status; a.iters = d_iters; a.refine = d_refine; a.relres = d_relres;
  a.tol = tol; a.inner_tol = h->opt.inner_tol; a.prec_thr = std::ldexp(1.0, -h->opt.prec_stop_log2);
  a.inner_max = h->opt.inner_max_iter; a.max_refine = h->opt.max_refine; a.max_iter = max_iter;
  GABP_CUDA(cudaFuncSetAttribute(kt_solve, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTSmem));
  GABP_CUDA(cudaMemsetAsync(a.queue, 0, 2 * sizeof(int), h->stream));
  kt_diag<<<nb, kBlock, 0, h->stream>>>(nq, L->srow, g.ad, T.adp);
  cudaEvent_t e0 = h->prof.e0, e1 = h->prof.e1;
  cudaEventRecord(e0, h->stream);
  kt_solve<<<std::min(h->num_sms, T.njobs), kTThreads, kTSmem, h->stream>>>(a);
  GABP_CUDA(cudaGetLastError());
  cudaEventRecord(e1, h->stream);
  h->prof.launches += 2;
  int gave_up = 0;
  GABP_CUDA(cudaMemcpyAsync(&gave_up, a.queue + 1, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
  GABP_CUDA(cudaStreamSynchronize(h->stream));
  GABP_CUDA(cudaEventElapsedTime(ms_out, e0, e1));
  if (gave_up) {
    set_last_error("gabp_solve_systems: a wait for a bulk copy gave up");
    return GABP_TIMEOUT;
  }
  return GABP_OK;
}

}  // namespace gabp
