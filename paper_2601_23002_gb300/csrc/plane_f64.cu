// k_plane instantiated for the radix sets of the grids of 8 to 20 points per side
// (bit r set: radix r used by the fewest-pass factorisation of n), double plans;
// larger grids take the compile-time passes (cpass_f64.cu), or with
// OFDFT_CPASS=0 the kernel with every radix.
#include "plane.cuh"

namespace ofdft {

template <>
PlaneKernel<double> plane_kernel<double>(unsigned mask) {
  switch (mask) {
    case 0x28u: return k_plane<double, 0x28u>;         // 15
    case 0x100u: return k_plane<double, 0x100u>;       // 8
    case 0x200u: return k_plane<double, 0x200u>;       // 9
    case 0x204u: return k_plane<double, 0x204u>;       // 18
    case 0x400u: return k_plane<double, 0x400u>;       // 10
    case 0x404u: return k_plane<double, 0x404u>;       // 20
    case 0x1000u: return k_plane<double, 0x1000u>;     // 12
    case 0x10000u: return k_plane<double, 0x10000u>;   // 16
    default: return k_plane<double, kAllRadices>;
  }
}

}  // namespace ofdft
