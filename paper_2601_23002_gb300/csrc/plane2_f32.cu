// k_plane_prec2 (the one-field preconditioning pass on two-block clusters),
// float plans: reached with OFDFT_CPASS=0 only, so one kernel with every radix.
#include "plane.cuh"

namespace ofdft {

template <>
PlaneKernel<float> plane_prec2_kernel<float>(unsigned) {
  return k_plane_prec2<float, kAllRadices>;
}

}  // namespace ofdft
