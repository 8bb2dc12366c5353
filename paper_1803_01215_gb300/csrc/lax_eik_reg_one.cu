// Register-resident eikonal kernel: one coordinate per thread, a uniform batch
// (the node count at compile time), FP32.
#include "lax_eik_reg.cuh"

namespace hj {

hj_status launch_reg_exact_one(const SolveArgs<float>& a, int threads, cudaStream_t s) {
  return launch_reg_exact<1, 1>(a, threads, s);
}

}  // namespace hj
