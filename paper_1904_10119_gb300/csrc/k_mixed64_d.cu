// complex128 mixed-radix passes, part D of the plan list.
#include "k_mixed64.cuh"

namespace fft3 {
extern const Mixed64Kernels g_mixed64_d[] = {FFT3_MIXED64_D(FFT3_MIXED64_ROW){0, nullptr, nullptr}};
} // namespace fft3
