// Mixed-radix line passes, part D of the plan lists.
#include "k_mixed.cuh"

namespace fft3 {
extern const MixedKernels g_mixed_j_d[] = {FFT3_MIXED_J_D(FFT3_MIXED_ROW_J){0, nullptr}};
extern const MixedKernels g_mixed_c_d[] = {FFT3_MIXED_C_D(FFT3_MIXED_ROW_C){0, nullptr}};
} // namespace fft3
