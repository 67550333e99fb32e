// CUDA-core kernels: Poisson on tetrahedra, P1..P4 (FP64: poisson_fixed.cu).
#include <type_traits>

#include "simt_dispatch.cuh"

namespace ffc {
int launch_simt_tet_poisson(const LaunchArgs& a, int precision, bool assemble) {
  if (a.f->d != 3 || a.f->kind != FFC_POISSON) return FFC_EUNSUPPORTED;
  if (precision == FFC_FP64) return launch_poisson_fixed(a, assemble);
  return precision == FFC_FP32 ? simt_by_degree<3, FFC_POISSON, 4, float>(a, assemble) : FFC_EUNSUPPORTED;
}
}  // namespace ffc
