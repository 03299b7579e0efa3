// k_mixed.cuh -- the line passes of pass_kernels.cuh instantiated for one part
// of the mixed-radix plan list (mixed_plans.h); each part is its own
// translation unit so that they compile in parallel.
#pragma once

#include "mixed_plans.h"
#include "pass_kernels.cuh"
#include "plans.h"

#define FFT3_MIXED_ROW(N, T, ...)                                                                      \
    {N, (const void *)&fft3::k_pass_j<N, T, fft3::Radices<__VA_ARGS__>, fft3::lpt_j(T), false>,       \
     (const void *)&fft3::k_pass_c<N, T, fft3::Radices<__VA_ARGS__>, fft3::mixed_lpt_c(N, T)>},
