// CUDA-core kernels: mass and Poisson on triangles, P1..P4 (FP64 Poisson: poisson_fixed.cu).
#include <type_traits>

#include "simt_dispatch.cuh"

namespace ffc {
int launch_simt_tri(const LaunchArgs& a, int precision, bool assemble) {
  if (a.f->d != 2) return FFC_EUNSUPPORTED;
  if (a.f->kind == FFC_MASS) return simt_by_precision<2, FFC_MASS, 4>(a, precision, assemble);
  if (a.f->kind == FFC_POISSON) {
    if (precision == FFC_FP64) return launch_poisson_fixed(a, assemble);
    if (precision == FFC_FP32) return simt_by_degree<2, FFC_POISSON, 4, float>(a, assemble);
  }
  return FFC_EUNSUPPORTED;
}
}  // namespace ffc
