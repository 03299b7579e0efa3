// complex128 mixed-radix passes, part B of the plan list.
#include "k_mixed64.cuh"

namespace fft3 {
extern const Mixed64Kernels g_mixed64_b[] = {FFT3_MIXED64_B(FFT3_MIXED64_ROW){0, nullptr, nullptr}};
} // namespace fft3
