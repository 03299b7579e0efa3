// Mixed-radix line passes, part A of the plan list.
#include "k_mixed.cuh"

namespace fft3 {
extern const MixedKernels g_mixed_kernels_a[] = {FFT3_MIXED_PLANS_A(FFT3_MIXED_ROW){0, nullptr, nullptr}};
} // namespace fft3
