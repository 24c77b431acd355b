// sell64.cuh -- what the FP64 round kernels on the sliced layout share: the message formula, the order in
// which warps take slices, the layout's construction.
#pragma once
#include <vector>

#include "devutil.cuh"

namespace gabp {

constexpr int kSellWindow = 4096;  // rows sorted by degree within windows of this many (a multiple of 32)

// Warp / lane of the calling thread and the number of warps in the grid.
struct WarpPos {
  int lane, warp, nwarps;
};
__device__ __forceinline__ WarpPos warp_pos() {
  return WarpPos{(int)(threadIdx.x & 31), (int)((blockIdx.x * kBlock + threadIdx.x) >> 5),
                 (int)((gridDim.x * kBlock) >> 5)};
}

// The slice a warp takes in its pass m over the grid (ns or more: none).  Inside a window of kSellWindow
// rows the slices get narrower (rows sorted by degree), and a fixed stride would hand a warp slices of
// like width in every pass (28 % of the round with idle warps on the 2^20 random graph); turning each
// pass by the golden section of a window's 128 slices spreads every warp's slices over the window:
// 307 -> 240 us per round there, unchanged on grids.
__device__ __forceinline__ int pass_slice(const WarpPos &w, int m) {
  constexpr int kSlices = kSellWindow / 32, kGolden = 79;  // 128 / 1.618
  const int turn = (kGolden + kSlices - w.nwarps % kSlices) % kSlices;
  return m * w.nwarps + (w.warp + m * turn) % w.nwarps;
}

// Message k -> i of round t as {c, v} from node k's record at t-1 and the reverse message rv
// (i -> k at t-1).  bad: a cavity precision P_{k\i} of exactly 0.
__device__ __forceinline__ double2 message64(double A, const NodeRec64 &nk, const double2 &rv, int &bad) {
  const double den = fma(A, rv.x, nk.P);  // cavity precision P_{k\i}
  bad |= is_zero64(den);
  return make_double2(div64(A, den), fma(rv.x, rv.y, nk.h));
}

// Host: rows[b .. e) in windows of kSellWindow, each ordered by degree (descending, stable).
void sort_degree_windows(const std::vector<int> &rp, std::vector<int> &rows, size_t b, size_t e);
// Host: the layout of the given slice rows (32 a slice, -1 for none; rp: row offsets of the off-diagonal
// CSR) on the handle's graph; synchronises.  Values: sell64_values after gabp_set_values.
gabp_status build_sell64(gabp_handle h, Sell64 &S, const std::vector<int> &rp, const std::vector<int> &srow,
                         std::vector<int> *sp_out);
gabp_status sell64_values(gabp_handle h, Sell64 &S);
void free_sell64(Sell64 &S);

}  // namespace gabp
