// Mixed-radix line passes, part C of the plan lists.
#include "k_mixed.cuh"

namespace fft3 {
extern const MixedKernels g_mixed_j_c[] = {FFT3_MIXED_J_C(FFT3_MIXED_ROW_J){0, nullptr}};
extern const MixedKernels g_mixed_c_c[] = {FFT3_MIXED_C_C(FFT3_MIXED_ROW_C){0, nullptr}};
} // namespace fft3
