// Register-tiled tanh-drift kernel, d <= 128: tiles of 8 nodes.
#include "lax_td_tile.cuh"

namespace hj {

hj_status launch_tile_d128(const SolveArgs<float>& a, cudaStream_t s) {
  if (a.N <= 32) return launch_tile<8, 128, 36>(a, s);
  if (a.N <= 64) return launch_tile<8, 128, 68>(a, s);
  return HJ_ERR_UNSUPPORTED;
}

}  // namespace hj
