// Mixed-radix line passes, part D of the plan list.
#include "k_mixed.cuh"

namespace fft3 {
extern const MixedKernels g_mixed_kernels_d[] = {FFT3_MIXED_PLANS_D(FFT3_MIXED_ROW){0, nullptr, nullptr}};
} // namespace fft3
