// The mixed-precision tracking kernels of batches with a step budget (one loop, see
// run_tracker): default group width below a warp, dense degree 2 (n = 1..12) and 3
// (n = 1..8), term tables (n = 1..16).  Wider groups have one loop in any case.
#include "dense_kernel.cuh"
#include "term_param.cuh"

namespace hc {

template <int DEG, int N>
KernelRef pick_dense_budget(int n) {
  if constexpr (N == 0)
    return KernelRef{nullptr, 0};
  else
    return n == N ? dense_ref<DEG, HC_PREC_MIXED, N, 0, F_BUDGET>()
                  : pick_dense_budget<DEG, N - 1>(n);
}

template <int N>
KernelRef pick_term_budget(int n) {
  if constexpr (N == 0)
    return KernelRef{nullptr, 0};
  else
    return n == N ? term_ref<HC_PREC_MIXED, N, 0, F_BUDGET>() : pick_term_budget<N - 1>(n);
}

KernelRef budget_kernel(bool terms, int deg, int n) {
  if (terms) return pick_term_budget<16>(n);
  if (deg == 2) return pick_dense_budget<2, 12>(n);
  if (deg == 3) return pick_dense_budget<3, 8>(n);
  return KernelRef{nullptr, 0};
}

}  // namespace hc
