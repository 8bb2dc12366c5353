// Register-tiled tanh-drift kernel, d <= 64: tiles of 4 nodes.
#include "lax_td_tile.cuh"

namespace hj {

hj_status launch_tile_d64(const SolveArgs<float>& a, cudaStream_t s) {
  if (a.N <= 32) return launch_tile<4, 64, 36>(a, s);
  if (a.N <= 64) return launch_tile<4, 64, 68>(a, s);
  if (a.N <= 128) return launch_tile<4, 64, 132>(a, s);
  if (a.N <= 256) return launch_tile<4, 64, 260>(a, s);
  return HJ_ERR_UNSUPPORTED;
}

}  // namespace hj
