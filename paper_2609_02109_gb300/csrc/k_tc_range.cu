// The bf16 tensor-core scorer (k_tc.cuh) of the d_L 8, 64-64 shape with its model loop
// unrolled, range mode, with and without the lists' shared bar.
#include "k_tc.cuh"

namespace mf {

namespace {

template <bool SB>
TcFn pick_n(int n_models) {
  switch (n_models) {
    case 3: return k_score_tc<kTcRange, 8, 4, 1, 5, 4, 16, false, false, 3, kXmBf16, SB>;
    case 4: return k_score_tc<kTcRange, 8, 4, 1, 5, 4, 16, false, false, 4, kXmBf16, SB>;
    case 5: return k_score_tc<kTcRange, 8, 4, 1, 5, 4, 16, false, false, 5, kXmBf16, SB>;
    case 6: return k_score_tc<kTcRange, 8, 4, 1, 5, 4, 16, false, false, 6, kXmBf16, SB>;
    default: return k_score_tc<kTcRange, 8, 4, 1, 5, 4, 16, false, false, 7, kXmBf16, SB>;
  }
}

}  // namespace

TcFn tc_kernel_nm_range(int n_models, bool shared_bar) {
  return shared_bar ? pick_n<true>(n_models) : pick_n<false>(n_models);
}

}  // namespace mf
