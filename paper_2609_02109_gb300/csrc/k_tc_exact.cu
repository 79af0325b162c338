// The exact fp32 variant of the tensor-core scorer (k_tc.cuh), d_L 8, 64-64.
#include "k_tc.cuh"

namespace mf {

namespace {

// S1 = k1 / 8, S2 = h1 / 8 + 1 (the b2 step), S3 = hl / 8: K = 8 steps of kind::tf32.
template <int MODE, bool MP, bool UT>
TcFn exact() {
  return k_score_tc<MODE, 16, 8, 2, 9, 8, 16, MP, UT, 0, kXmTf32>;
}

template <int MODE>
TcFn pick_mode(bool mp, bool util) {
  if (mp) return util ? exact<MODE, true, true>() : exact<MODE, true, false>();
  return util ? exact<MODE, false, true>() : exact<MODE, false, false>();
}

}  // namespace

TcFn tc_kernel_exact(int mode, bool mp, bool util) {
  return mode == kTcRange ? pick_mode<kTcRange>(mp, util) : pick_mode<kTcList>(mp, util);
}

}  // namespace mf
