// k_plane_prec2 (the one-field preconditioning pass on two-block clusters),
// double plans: the FP64 162^3 grid, and with OFDFT_CPASS=0 smaller ones, so one kernel with every radix.
#include "plane.cuh"

namespace ofdft {

template <>
PlaneKernel<double> plane_prec2_kernel<double>(unsigned) {
  return k_plane_prec2<double, kAllRadices>;
}

}  // namespace ofdft
