// Mixed-radix line passes, part C of the plan list.
#include "k_mixed.cuh"

namespace fft3 {
extern const MixedKernels g_mixed_kernels_c[] = {FFT3_MIXED_PLANS_C(FFT3_MIXED_ROW){0, nullptr, nullptr}};
} // namespace fft3
