// Register-tiled tanh-drift kernel, d <= 32: tiles of 4 nodes.
#include "lax_td_tile.cuh"

namespace hj {

hj_status launch_tile_d32(const SolveArgs<float>& a, cudaStream_t s) {
  if (a.N <= 32) return launch_tile<4, 32, 36>(a, s);
  if (a.N <= 64) return launch_tile<4, 32, 68>(a, s);
  if (a.N <= 128) return launch_tile<4, 32, 132>(a, s);
  if (a.N <= 256) return launch_tile<4, 32, 260>(a, s);
  return HJ_ERR_UNSUPPORTED;
}

}  // namespace hj
