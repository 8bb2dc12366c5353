// Register-resident eikonal kernel: two coordinates per thread, a cluster of two CTAs per point, a uniform batch
// (the node count at compile time), FP32.
#include "lax_eik_reg.cuh"

namespace hj {

hj_status launch_reg_exact_cluster(const SolveArgs<float>& a, int threads, cudaStream_t s) {
  return launch_reg_exact<2, 2>(a, threads, s);
}

}  // namespace hj
