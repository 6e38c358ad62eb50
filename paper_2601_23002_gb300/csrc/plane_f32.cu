// k_plane instantiated for the radix sets of the grids of 8 to 20 points per side
// (bit r set: radix r used by the fewest-pass factorisation of n), float plans;
// larger grids take the compile-time passes (cpass_f32.cu), or with
// OFDFT_CPASS=0 the kernel with every radix.
#include "plane.cuh"

namespace ofdft {

template <>
PlaneKernel<float> plane_kernel<float>(unsigned mask) {
  switch (mask) {
    case 0x28u: return k_plane<float, 0x28u>;         // 15
    case 0x100u: return k_plane<float, 0x100u>;       // 8
    case 0x200u: return k_plane<float, 0x200u>;       // 9
    case 0x204u: return k_plane<float, 0x204u>;       // 18
    case 0x400u: return k_plane<float, 0x400u>;       // 10
    case 0x404u: return k_plane<float, 0x404u>;       // 20
    case 0x1000u: return k_plane<float, 0x1000u>;     // 12
    case 0x10000u: return k_plane<float, 0x10000u>;   // 16
    default: return k_plane<float, kAllRadices>;
  }
}

}  // namespace ofdft
