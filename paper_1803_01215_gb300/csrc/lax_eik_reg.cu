// Dispatch of the register-resident eikonal kernel (lax_eik_reg.cuh), and its
// instantiations for ragged batches, N in 11..16 and FP64.
//
// A uniform batch with N = 16 takes the sixteen-node form without node guards: with them
// its per-node state does not stay in registers (d = 100, 600 points: 11.1 ms without,
// 28.6 with; d = 400, 150 points: 20.3 and 39.2).
#include "lax_eik_reg.cuh"

namespace hj {

// Runs the register-resident eikonal kernel when it applies (static bump,
// backward Euler; FP32: d <= 512 with N <= 16, d <= 1024 with N <= 10 and, on a
// cluster of two CTAs, d <= 2048 with N <= 10; FP64: d <= 512 with N <= 10);
// HJ_ERR_UNSUPPORTED otherwise, and the caller takes the shared-memory kernel.
template <typename T>
hj_status launch_eik_reg_solver(const SolveArgs<T>& a, cudaStream_t s) {
  if (a.eik_moving || a.scheme != HJ_SCHEME_BE || a.formulation != HJ_FORM_LAX ||
      a.inner_steps != 1 || a.xb == nullptr)
    return HJ_ERR_UNSUPPORTED;
  if (a.d < 1 || a.N < 1 || a.N > 16) return HJ_ERR_UNSUPPORTED;
  auto threads_for = [](int coords) { return (coords + 31) / 32 * 32; };
  if constexpr (sizeof(T) == 8) {             // FP64 state fits the registers at one coordinate, N <= 10
    if (a.d > kRegMaxThreads || a.N > 10) return HJ_ERR_UNSUPPORTED;
    return (a.Nv == nullptr && a.N == 10) ? launch_reg<T, 1, 10, true, 1>(a, threads_for(a.d), s)
                                          : launch_reg<T, 1, 10, false, 1>(a, threads_for(a.d), s);
  } else {
    const bool uniform = a.Nv == nullptr;     // every point has a.N nodes: no node guards
    if (a.N <= 10) {
      // two coordinates per thread from d = 64 (half the threads per point, the
      // same work per barrier: d = 100 ran 13.5 against 15.2 ms), one below
      if (a.d < 64) {
        const int t = threads_for(a.d);
        return uniform ? launch_reg_exact_one(a, t, s) : launch_reg<T, 1, 10, false, 1>(a, t, s);
      }
      if (a.d <= 2 * kRegMaxThreads) {
        const int t = threads_for((a.d + 1) / 2);
        return uniform ? launch_reg_exact_two(a, t, s) : launch_reg<T, 2, 10, false, 1>(a, t, s);
      }
      if (a.d <= 4 * kRegMaxThreads) {        // two CTAs, each half of the coordinates
        const int t = threads_for(((a.d + 1) / 2 + 1) / 2);
        return uniform ? launch_reg_exact_cluster(a, t, s) : launch_reg<T, 2, 10, false, 2>(a, t, s);
      }
      return HJ_ERR_UNSUPPORTED;
    }
    if (a.d > kRegMaxThreads) return HJ_ERR_UNSUPPORTED;
    return uniform && a.N == 16 ? launch_reg<T, 1, 16, true, 1>(a, threads_for(a.d), s)
                                : launch_reg<T, 1, 16, false, 1>(a, threads_for(a.d), s);
  }
}

template hj_status launch_eik_reg_solver<float>(const SolveArgs<float>&, cudaStream_t);
template hj_status launch_eik_reg_solver<double>(const SolveArgs<double>&, cudaStream_t);

}  // namespace hj
