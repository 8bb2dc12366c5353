// Dispatch of the register-tiled tanh-drift kernel (lax_td_tile.cuh).
#include "hj_internal.cuh"

namespace hj {

hj_status launch_tile_d32(const SolveArgs<float>& a, cudaStream_t s);
hj_status launch_tile_d64(const SolveArgs<float>& a, cudaStream_t s);
hj_status launch_tile_d104(const SolveArgs<float>& a, cudaStream_t s);
hj_status launch_tile_d128(const SolveArgs<float>& a, cudaStream_t s);

namespace {

// Warps a point takes with j-tiles in whole blocks of four, rounded up to a power of two:
// up to 8 with eight-node tiles (about 240 registers), 16 with four-node tiles (128
// registers); 0 if it does not fit.  This is the range of (d, N) that the kernel serves;
// the launch itself takes as many warps as the tiles fill.  It is not the largest that
// would fit (d = 100, N = 65..80 fills 8 warps of eight-node tiles and is left to the
// shared-memory kernel, whose sums round in another order): points served by either
// kernel give the bits that they always gave.
int group_warps(int d, int N, int TJ) {
  const int TIc = (d + 3) / 4, TJc = (N + TJ - 1) / TJ;
  const int w = (4 * TIc * ((TJc + 3) / 4) + 31) / 32;
  const int g = w <= 1 ? 1 : w <= 2 ? 2 : w <= 4 ? 4 : w <= 8 ? 8 : w <= 16 ? 16 : 0;
  return (g == 16 && TJ != 4) ? 0 : g;
}

}  // namespace

// Runs the register-tiled kernel when it applies (FP32, tanh drift, a point in
// at most 16 warps of four-node tiles, d <= 64, or 8 of eight-node tiles);
// HJ_ERR_UNSUPPORTED otherwise, and the caller takes the shared-memory kernel.
hj_status launch_td_tile_solver(const SolveArgs<float>& a, cudaStream_t s) {
  if (a.inner_steps != 1 || a.A == nullptr || a.At == nullptr) return HJ_ERR_UNSUPPORTED;
  if (a.d < 1 || a.d > kMaxD || a.N < 1 || a.N > kMaxN) return HJ_ERR_UNSUPPORTED;
  if (a.d <= 64) {                   // 16 warps of eight-node tiles never fit where four-node ones do not
    if (group_warps(a.d, a.N, 4) == 0) return HJ_ERR_UNSUPPORTED;
    return a.d <= 32 ? launch_tile_d32(a, s) : launch_tile_d64(a, s);
  }
  if (group_warps(a.d, a.N, 8) == 0) return HJ_ERR_UNSUPPORTED;
  return a.d <= 104 ? launch_tile_d104(a, s) : launch_tile_d128(a, s);
}

}  // namespace hj
