// devutil.cuh -- small device helpers shared by the solver's kernels.
#pragma once
#include <cuda_runtime.h>
#include "gabp_internal.cuh"

namespace gabp {

// IEEE division, kept out of line so that the common paths of div64 and rcp64 do not
// carry its instructions.
static __device__ __noinline__ double div64_slow(double a, double d) { return a / d; }

// Division off the FP64 pipe.  GB300 retires two FP64 operations per SM and clock (a warp's
// FP64 instruction holds its scheduler's unit for 64 cycles) and bounds the FP64 rounds with
// them, while the integer units stand idle: a quotient formed with integer instructions
// (about 45 a warp) replaces four FP64 ones (three of a reciprocal iteration, one product).
//
// Reciprocal of d's 53-bit significand m in [1, 2): seed y (24 bits, PTX rcp.approx.ftz.f32 of
// m cut to 24 bits, so |m y - 1| < 2^-21.5 with a margin), then the geometric series
//   1 / m = y / (1 + s) = y (1 - s + s^2 - ...),   s = m y - 1  (exact, s^3 < 2^-64),
// in fixed point.  Units: y 2^-24, m 2^-52, so m y wraps modulo 2^64 at 2^76 = 1 and its low
// 64 bits, read as signed, are s itself.  Returns 1 / m in units of 2^-63 (error a few units).
__device__ __forceinline__ unsigned long long rcp_sig64(unsigned dh, unsigned dl) {
  float yf;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(__uint_as_float(0x3f800000u | ((dh & 0xfffffu) << 3) | (dl >> 29))));
  const unsigned y = __float_as_uint(yf) - 0x3e800000u;  // y in (2^23, 2^24]: [0.5, 1] in units of 2^-24
  const unsigned mh = (dh & 0xfffffu) | 0x100000u;
  const long long s = (long long)((unsigned long long)dl * y + ((unsigned long long)(mh * y) << 32));
  const int s32 = (int)(s >> 24);                                    // s in units of 2^-52
  const long long t = s + (long long)__mulhi(s32, s32) * -16;        // s - s^2, units of 2^-76
  const long long w = (long long)(int)(t >> 32) * (int)y + (long long)__umulhi((unsigned)t, y);  // y t, units of 2^-68
  return ((unsigned long long)(y << 7) << 32) - (unsigned long long)(w >> 5);
}

// Exponent field of a high word, and whether quotients of two such operands are certain to be normal
// (zero, subnormal, inf, NaN and the outer exponents take the IEEE division).
__device__ __forceinline__ int exp_field64(unsigned hi) { return (int)((hi >> 20) & 0x7ffu); }
__device__ __forceinline__ bool plain_exp64(int e) { return (unsigned)(e - 523) <= 1000u; }

// a / d within 0.51 units in the last place (IEEE division's 0.50): the significands' 64-bit
// product a (1 / d), normalised, rounded to 53 bits and put together with the exponent.
__device__ __forceinline__ double div64(double a, double d) {
  unsigned ah, al, dh, dl;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(al), "=r"(ah) : "d"(a));
  asm("mov.b64 {%0, %1}, %2;" : "=r"(dl), "=r"(dh) : "d"(d));
  const unsigned long long z = rcp_sig64(dh, dl);
  const unsigned mh = ((ah & 0xfffffu) | 0x100000u) << 11 | (al >> 21), ml = al << 11;  // units of 2^-63
  const unsigned zh = (unsigned)(z >> 32), zl = (unsigned)z;
  const unsigned long long q =
      (unsigned long long)mh * zh + ((unsigned long long)__umulhi(mh, zl) + __umulhi(ml, zh));  // units of 2^-62
  const int sh = (unsigned)(q >> 32) < 0x40000000u ? 1 : 0;  // quotient of the significands below 1
  const unsigned long long r = (q + (unsigned)(512 >> sh)) >> (10 - sh);
  const int ea = exp_field64(ah), ed = exp_field64(dh);
  const unsigned rh = ((unsigned)(r >> 32) + ((unsigned)(ea - ed + 1022 - sh) << 20)) ^ ((ah ^ dh) & 0x80000000u);
  double v;
  asm("mov.b64 %0, {%1, %2};" : "=d"(v) : "r"((unsigned)r), "r"(rh));
  if (!plain_exp64(ea) || !plain_exp64(ed)) v = div64_slow(a, d);
  return v;
}

// 1 / d in the same way (no product).
__device__ __forceinline__ double rcp64(double d) {
  unsigned dh, dl;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(dl), "=r"(dh) : "d"(d));
  const unsigned long long r = (rcp_sig64(dh, dl) + 512u) >> 10;  // 2^52 .. 2^53 (1 / 1 carries into the exponent)
  const int ed = exp_field64(dh);
  const unsigned rh = ((unsigned)(r >> 32) + ((unsigned)(2044 - ed) << 20)) ^ (dh & 0x80000000u);
  double v;
  asm("mov.b64 %0, {%1, %2};" : "=d"(v) : "r"((unsigned)r), "r"(rh));
  if (!plain_exp64(ed)) v = div64_slow(1.0, d);
  return v;
}

// d == +0 or -0, tested on the bit pattern.  The two 32-bit halves come out of an
// inline move so the test stays on the integer pipe: written on the 64-bit pattern
// in C, it is recognised as d == 0.0 and becomes an FP64 compare, one more
// instruction per message on the FP64 pipe that bounds the FP64 rounds.
__device__ __forceinline__ bool is_zero64(double d) {
  unsigned lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "d"(d));
  return ((hi << 1) | lo) == 0u;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// max that keeps a NaN from either side (fmax drops it): a NaN change or
// residual must never read as "small".
template <typename T>
__device__ __forceinline__ T nan_max(T a, T b) {
  return (a > b || a != a) ? a : b;
}

// |now - prev| / |now| with 0 for an unchanged value (an explicitly stored zero
// coupling keeps a zero message: 0/0 must not read as a NaN change).
__device__ __forceinline__ float rel_change(float now, float prev) {
  const float d = fabsf(now - prev);
  return d == 0.f ? 0.f : d / fabsf(now);
}

template <typename T>
__device__ __forceinline__ T warp_max(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = nan_max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Sum over the L lanes of a sub-warp (L a power of two dividing 32); every lane
// of the warp must call it.
template <int L, typename T>
__device__ __forceinline__ T sub_sum(T v) {
#pragma unroll
  for (int o = L / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, L);
  return v;
}

// Block-wide sum of NV doubles over NT threads.  Result valid in thread 0.  The threads' values meet in
// shared memory and one warp a value adds them: 12 FP64 instructions a block of 256 threads (7 a lane, 5
// in the butterfly), where a butterfly in every warp first issued 45, each 64 cycles of a scheduler.
template <int NV, int NT>
__device__ __forceinline__ void block_sum_nt(double (&v)[NV]) {
  __shared__ double sh[NV][NT], res[NV];
  constexpr int NW = NT / 32;
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
#pragma unroll
  for (int j = 0; j < NV; ++j) sh[j][threadIdx.x] = v[j];
  __syncthreads();
  for (int j = w; j < NV; j += NW) {
    double s[NW];
#pragma unroll
    for (int q = 0; q < NW; ++q) s[q] = sh[j][l + 32 * q];
#pragma unroll
    for (int o = NW / 2; o > 0; o >>= 1)
#pragma unroll
      for (int q = 0; q < o; ++q) s[q] += s[q + o];
    s[0] = warp_sum(s[0]);
    if (l == 0) res[j] = s[0];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int j = 0; j < NV; ++j) v[j] = res[j];
  }
}

// Block-wide max of NV doubles over NT threads.  Result valid in thread 0.
template <int NV, int NT>
__device__ __forceinline__ void block_max_nt(double (&v)[NV]) {
  __shared__ double sh[NV][NT / 32];
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
#pragma unroll
  for (int j = 0; j < NV; ++j) {
    double s = warp_max(v[j]);
    if (l == 0) sh[j][w] = s;
  }
  __syncthreads();
  if (w == 0) {
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      double s = l < NT / 32 ? sh[j][l] : -1.0;
      v[j] = warp_max(s);
    }
  }
  __syncthreads();
}

// Block-wide sum of NV doubles (kBlock threads).  Result valid in thread 0.
template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV]) {
  block_sum_nt<NV, kBlock>(v);
}

// Publish this block's NV partial values (thread 0 holds them) into
// partials[j * gridDim.x + blockIdx.x] and find out whether this block is the
// last of the grid to finish.  In the last block, tot[] (valid in thread 0)
// receives the sums over all blocks, taken in a fixed order (deterministic).
template <int NV>
__device__ __forceinline__ bool last_block_reduce(double (&v)[NV], double *partials, unsigned int *arrive,
                                                  double (&tot)[NV]) {
  __shared__ bool s_last;
  if (threadIdx.x == 0) {
#pragma unroll
    for (int j = 0; j < NV; ++j) partials[j * gridDim.x + blockIdx.x] = v[j];
    __threadfence();
    unsigned int prev = atomicAdd(arrive, 1u);
    s_last = (prev == gridDim.x - 1);
  }
  __syncthreads();
  if (!s_last) return false;
  __threadfence();
#pragma unroll
  for (int j = 0; j < NV; ++j) tot[j] = 0.0;
  // deterministic: each thread's stripe is fixed; the block tree is fixed
  for (int bI = threadIdx.x; bI < (int)gridDim.x; bI += kBlock) {
#pragma unroll
    for (int j = 0; j < NV; ++j) tot[j] += __ldcg(partials + j * gridDim.x + bI);
  }
  block_sum<NV>(tot);
  return true;
}

}  // namespace gabp
