// The compile-time passes of FP32 plans.  Compiled in parts (CPASS_PART 0..5, a share of
// the grid sizes each), since every size has kernels of its own.
#include <initializer_list>
#include "cpass.cuh"

namespace ofdft {

#define OFDFT_CP(N)                                                   \
  case N: {                                                           \
    static const CPass<float> p = make_cpass<float, N>();            \
    return &p;                                                        \
  }

#define OFDFT_CAT2(a, b) a##b
#define OFDFT_CAT(a, b) OFDFT_CAT2(a, b)
const CPass<float>* OFDFT_CAT(cpass_f32_, CPASS_PART)(int n) {
  switch (n) {
#if CPASS_PART == 0
    OFDFT_CP(24) OFDFT_CP(36) OFDFT_CP(50) OFDFT_CP(75) OFDFT_CP(90) OFDFT_CP(160) OFDFT_CP(250)
#elif CPASS_PART == 1
    OFDFT_CP(25) OFDFT_CP(40) OFDFT_CP(54) OFDFT_CP(72) OFDFT_CP(96) OFDFT_CP(150) OFDFT_CP(240)
#elif CPASS_PART == 2
    OFDFT_CP(27) OFDFT_CP(45) OFDFT_CP(60) OFDFT_CP(80) OFDFT_CP(128) OFDFT_CP(144) OFDFT_CP(225)
#elif CPASS_PART == 3
    OFDFT_CP(30) OFDFT_CP(32) OFDFT_CP(48) OFDFT_CP(64) OFDFT_CP(108) OFDFT_CP(135) OFDFT_CP(216)
#elif CPASS_PART == 4
    OFDFT_CP(81) OFDFT_CP(100) OFDFT_CP(120) OFDFT_CP(192) OFDFT_CP(200)
#else
    OFDFT_CP(125) OFDFT_CP(162) OFDFT_CP(180) OFDFT_CP(243)
#endif
    default: return nullptr;
  }
}

#if CPASS_PART == 0
const CPass<float>* cpass_f32_1(int n);
const CPass<float>* cpass_f32_2(int n);
const CPass<float>* cpass_f32_3(int n);
const CPass<float>* cpass_f32_4(int n);
const CPass<float>* cpass_f32_5(int n);
template <> const CPass<float>* cpass_kernels<float>(int n) {
  for (auto* part : {cpass_f32_0, cpass_f32_1, cpass_f32_2, cpass_f32_3, cpass_f32_4, cpass_f32_5})
    if (const CPass<float>* p = part(n)) return p;
  return nullptr;
}
#endif

}  // namespace ofdft
