// Mixed-radix line passes, part A of the plan lists.
#include "k_mixed.cuh"

namespace fft3 {
extern const MixedKernels g_mixed_j_a[] = {FFT3_MIXED_J_A(FFT3_MIXED_ROW_J){0, nullptr}};
extern const MixedKernels g_mixed_c_a[] = {FFT3_MIXED_C_A(FFT3_MIXED_ROW_C){0, nullptr}};
} // namespace fft3
