// k_mixed64.cuh -- the complex128 passes (k_pass64.cuh) of one part of the
// mixed-radix plans (mixed64_plans.h); each part is its own translation unit so
// that they compile in parallel.
#pragma once

#include "k_pass64.cuh"
#include "mixed64_plans.h"

#define FFT3_MIXED64_ROW(N, T, LPT, SH, PITCH, ...)                                             \
    {N, (const void *)&fft3::k_pass_j64<N, T, fft3::Radices<__VA_ARGS__>, LPT, SH, PITCH>,     \
     (const void *)&fft3::k_pass_c64<N, T, fft3::Radices<__VA_ARGS__>, fft3::kLpt64Strided, fft3::groups64(T)>},
