// The exact fp32 variants of the tensor-core scorer (k_tc.cuh), d_L 8, 64-64.
#include "k_tc.cuh"

namespace mf {

namespace {

template <int MODE, bool MP, bool UT>
TcFn pick_exact(int xm) {
  // S1 = k1 / K, S2 = h1 / K + 1 (the b2 step), S3 = hl / K with K = 8 (tf32) or 16 (fp16).
  // (A compile-time model count with register digits, which serves bf16, is slower here:
  // 24^6 32.9 ms against 31.4 with the run-time loop.)
  return xm == kXmTf32 ? k_score_tc<MODE, 16, 8, 2, 9, 8, 16, MP, UT, 0, kXmTf32>
                       : k_score_tc<MODE, 8, 4, 1, 5, 4, 16, MP, UT, 0, kXmHalf>;
}

template <int MODE>
TcFn pick_mode(int xm, bool mp, bool util) {
  if (mp) return util ? pick_exact<MODE, true, true>(xm) : pick_exact<MODE, true, false>(xm);
  return util ? pick_exact<MODE, false, true>(xm) : pick_exact<MODE, false, false>(xm);
}

}  // namespace

TcFn tc_kernel_exact(int xm, int mode, bool mp, bool util) {
  return mode == kTcRange ? pick_mode<kTcRange>(xm, mp, util) : pick_mode<kTcList>(xm, mp, util);
}

}  // namespace mf
