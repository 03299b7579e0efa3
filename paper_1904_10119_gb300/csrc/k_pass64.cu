// k_pass64.cu -- the complex128 passes (k_pass64.cuh) of the power-of-two plans,
// and the integer twiddle generator.
#include "k_pass64.cuh"

namespace fft3 {

template <int N, int T, class Rad>
constexpr const void *pass_c64_ptr()
{
    if constexpr (T * kLpt64Strided <= 1024)
        return (const void *)&k_pass_c64<N, T, Rad, kLpt64Strided, groups64(T)>;
    else
        return nullptr;
}

#define FFT3_KERNEL64_ROW(ID, N, T, ...)                                                              \
    {ID, (const void *)&k_pass_j64<N, T, Radices<__VA_ARGS__>, lpt_j64(T)>,                           \
     pass_c64_ptr<N, T, Radices<__VA_ARGS__>>()},

static const Fixed64Kernels g_fixed64[] = {FFT3_FIXED_PLANS_A(FFT3_KERNEL64_ROW)
                                               FFT3_FIXED_PLANS_B(FFT3_KERNEL64_ROW)};

const Fixed64Kernels *fixed64_kernels(int id)
{
    for (const Fixed64Kernels &k : g_fixed64)
        if (k.id == id)
            return &k;
    return nullptr;
}

// Twiddles of the integer stages: w_n^m * 2^62 for the listed exponents.
__global__ void k_roots_fix(int n, const int64_t *m, int64_t count, root62 *o)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x)
        o[i] = root_fix(m[i], n);
}

} // namespace fft3
