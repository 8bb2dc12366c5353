// Register-tiled tanh-drift kernel, d <= 104: tiles of 8 nodes.
// A row stride of A below 128 leaves shared memory for more points where the groups are
// one warp: d = 72, N = 8 eight of them beside A against four (8000 points: 6.64 ms,
// 7.77 with the stride 128; d = 70, N = 7 5.86 and 6.98).  From N = 9 on, and above d =
// 72, the two strides measured the same (d = 72..104, N = 8..96): the class could end
// anywhere between.
#include "lax_td_tile.cuh"

namespace hj {

hj_status launch_tile_d104(const SolveArgs<float>& a, cudaStream_t s) {
  if (a.N <= 32) return launch_tile<8, 104, 36>(a, s);
  if (a.N <= 64) return launch_tile<8, 104, 68>(a, s);
  if (a.N <= 128) return launch_tile<8, 104, 132>(a, s);
  return HJ_ERR_UNSUPPORTED;
}

}  // namespace hj
