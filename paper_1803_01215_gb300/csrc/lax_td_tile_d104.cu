// Register-tiled tanh-drift kernel, d <= 104: tiles of 8 nodes.
#include "lax_td_tile.cuh"

namespace hj {

hj_status launch_tile_d104(const SolveArgs<float>& a, cudaStream_t s) {
  if (a.N <= 32) return launch_tile<8, 104, 36>(a, s);
  if (a.N <= 64) return launch_tile<8, 104, 68>(a, s);
  if (a.N <= 128) return launch_tile<8, 104, 132>(a, s);
  return HJ_ERR_UNSUPPORTED;
}

}  // namespace hj
