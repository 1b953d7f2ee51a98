// Parameter-homotopy (term table) tracking kernels in double-float
// arithmetic (HC_PREC_DF), n = 1..24 (the last re-tracking tier of the mixed
// pipeline, and precision HC_PREC_DF).  lanes = 0: the warps per path that suit
// n; 32: one warp per path (beside a resident launch, whose free block slots
// may take no larger block).
#include "term_block.cuh"

namespace hc {

template <int N>
KernelRef pick_term_df(int n, int lanes) {
  if constexpr (N == 0) {
    return KernelRef{nullptr, 0};
  } else {
    if (n == N) return lanes == 32 ? term_df_ref<N, 1>() : term_df_ref<N, term_df_warps(N)>();
    return pick_term_df<N - 1>(n, lanes);
  }
}

KernelRef term_ref_df(int n, int lanes) { return pick_term_df<24>(n, lanes); }

}  // namespace hc
