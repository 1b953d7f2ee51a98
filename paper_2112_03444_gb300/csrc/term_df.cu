// Parameter-homotopy (term table) tracking kernels in double-float
// arithmetic (HC_PREC_DF), n = 1..24 (the last re-tracking tier of the mixed
// pipeline, and precision HC_PREC_DF).  lanes = 0: the warps per path that suit
// n; 32: one warp per path (beside a resident launch, whose free block slots
// may take no larger block).
#include "term_block.cuh"

namespace hc {

// Two warps for up to 8 unknowns, four above: the terms of an equation grow
// with n, and a round takes one per thread.
template <int N>
KernelRef pick_term_df(int n, int lanes) {
  if constexpr (N == 0) {
    return KernelRef{nullptr, 0};
  } else {
    constexpr int NW = N <= 4 ? 1 : N <= 8 ? 2 : 4;
    if (n == N) return lanes == 32 ? term_df_ref<N, 1>() : term_df_ref<N, NW>();
    return pick_term_df<N - 1>(n, lanes);
  }
}

KernelRef term_ref_df(int n, int lanes) { return pick_term_df<24>(n, lanes); }

}  // namespace hc
