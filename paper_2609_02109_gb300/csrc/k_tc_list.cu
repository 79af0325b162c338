// The bf16 tensor-core scorer (k_tc.cuh) of the d_L 8, 64-64 shape with its model loop
// unrolled, list mode.
#include "k_tc.cuh"

namespace mf {

TcFn tc_kernel_nm_list(int n_models) {
  switch (n_models) {
    case 3: return k_score_tc<kTcList, 8, 4, 1, 5, 4, 16, false, false, 3, kXmBf16>;
    case 4: return k_score_tc<kTcList, 8, 4, 1, 5, 4, 16, false, false, 4, kXmBf16>;
    case 5: return k_score_tc<kTcList, 8, 4, 1, 5, 4, 16, false, false, 5, kXmBf16>;
    case 6: return k_score_tc<kTcList, 8, 4, 1, 5, 4, 16, false, false, 6, kXmBf16>;
    default: return k_score_tc<kTcList, 8, 4, 1, 5, 4, 16, false, false, 7, kXmBf16>;
  }
}

}  // namespace mf
