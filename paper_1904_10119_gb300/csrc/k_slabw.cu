// k_slabw.cu -- the 2D DFT of n0 x n1 slabs (Section 2.3, slab-pencil), one slab
// at a time per block of 256 threads, with compile-time line transforms: x lines
// from global memory through warp registers into shared memory, y lines in place
// there (slab_warp.cuh), the slab copied out with 16-byte stores.  For slabs whose
// sides are lengths of FFT3_SLABZ_WARP_PLANS (8 to 128 points); other slabs run
// k_slab, whose radix lists are data.
// What bounds it: latency (one slab's loads, rows, columns and stores follow each
// other in a block).  64^3: slab pass and z pass 10.3 us, with k_slab 14.4.
#include "pass_kernels.cuh"
#include "slab_warp.cuh"

namespace fft3 {

__global__ void __launch_bounds__(kSzThreads, 3) k_slab_warp(PassArgs a)
{
    extern __shared__ __align__(16) float2 smem[];
    const int n0 = a.L[0].n, n1 = a.L[1].n, P = n0 | 1;
    // the tables w_n^m (m < n) of the two lengths, read through L1
    const float2 *twx = a.tw + a.L[0].tw_off, *twy = a.tw + a.L[1].tw_off;
    const int off[16] = {};
    const bool conj = a.conj != 0;
    pdl_wait();
    for (int64_t tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
        const int64_t sa = tile % a.g.A, sb = tile / a.g.A;
        sz_run_rows_warp(n0, a.in + sa * a.g.ia + sb * a.g.ib, smem, P, n1, twx, off, conj);
        __syncthreads();
        sz_run_cols_warp(n1, smem, P, n0, n0, n1 * P, twy, off);
        __syncthreads();
        sz_copy_out(smem, P, n0, n1, a.out + sa * a.g.oa + sb * a.g.ob, conj);
        __syncthreads();
    }
}

} // namespace fft3
