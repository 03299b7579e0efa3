// complex128 mixed-radix passes, part C of the plan list.
#include "k_mixed64.cuh"

namespace fft3 {
extern const Mixed64Kernels g_mixed64_c[] = {FFT3_MIXED64_C(FFT3_MIXED64_ROW){0, nullptr, nullptr}};
} // namespace fft3
