// fqt_gemm_pair.cu -- the instances of k_gemm that run on CTA pairs
// (cta_group::2, 256 x 256 super tiles); run_gemm in fqt_gemm.cu chooses
// between them and the single-CTA instances.
#include "fqt_gemm_core.cuh"

namespace fqt {

GemmKernel gemm_pair_kernel(int mode, int nb, int form) {
  if (mode == MODE_PARTIAL) return k_gemm<MODE_PARTIAL, 1, 0, true>;
#define FQT_GXP(NBV)                                                         \
  case NBV:                                                                  \
    return form == 2   ? k_gemm<MODE_GRADX, NBV, 2, true>                    \
           : form == 1 ? k_gemm<MODE_GRADX, NBV, 1, true>                    \
                       : k_gemm<MODE_GRADX, NBV, 0, true>;
  switch (nb) {
    FQT_GXP(1)
    FQT_GXP(4)
    FQT_GXP(8)
    FQT_GXP(16)
    FQT_GXP(32)
    FQT_GXP(64)
  }
#undef FQT_GXP
  return nullptr;
}

}  // namespace fqt
