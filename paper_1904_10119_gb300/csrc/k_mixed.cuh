// k_mixed.cuh -- the line passes of pass_kernels.cuh for the plans of
// mixed_plans.h, with the tile, occupancy and shared layout each plan names;
// each part of the list is its own translation unit so that they compile in
// parallel.
#pragma once

#include "mixed_plans.h"
#include "pass_kernels.cuh"

namespace fft3 {

template <int SH>
struct SmemLineMixed { // position p at p + (p >> SH), SH = 0: p
    float2 *p;
    __device__ __forceinline__ static int pos(int j)
    {
        if constexpr (SH > 0)
            return j + (j >> SH);
        else
            return j;
    }
    __device__ __forceinline__ float2 operator()(int j) const { return p[pos(j)]; }
    __device__ __forceinline__ void operator()(int k, float2 v) const { p[pos(k)] = v; }
};

// Contiguous lines (ij == 1, ok == 1).  What bounds it: memory up to about 200
// points (two stages), instructions and the shared-memory exchanges of three
// stages beyond; the rates stand in mixed_plans.h.
template <int N, int T, int LPT, int MB, int SH, int PITCH, class Rad>
__global__ void __launch_bounds__(T *LPT, MB) k_mixed_j(PassArgs a)
{
    static_assert(MB <= 32, "an SM holds 32 blocks; a larger bound is ignored");
    extern __shared__ float2 smem[];
    float2 *tw = smem;
    float2 *buf = smem + tw_slots(a.tw_len);
    load_twiddles(tw, a.tw, a.tw_len);
    pdl_wait();
    const int t = threadIdx.x % T, l = threadIdx.x / T;
    const bool conj = a.conj != 0;
    for (int64_t tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
        __syncthreads();
        const TileId id = decode_tile(tile, a.tiles_c, a.g.A, LPT);
        const int64_t c = id.c0 + l;
        const bool valid = c < a.g.C;
        GLoad1 src{a.in + c * a.g.ic + id.a * a.g.ia + id.b * a.g.ib, valid, conj};
        GStore1 dst{a.out + c * a.g.oc + id.a * a.g.oa + id.b * a.g.ob, valid, conj};
        SmemLineMixed<SH> sm{buf + l * PITCH};
        EngineFixed<N, T, 1, Rad>::template run<true, false>(t, src, sm, dst, tw);
    }
}

// Strided columns (ic == 1, oc == 1), position-major shared layout.
template <int N, int T, int LPT, int MB, class Rad>
__global__ void __launch_bounds__(T *LPT, MB) k_mixed_c(PassArgs a)
{
    static_assert(MB <= 32, "an SM holds 32 blocks; a larger bound is ignored");
    extern __shared__ float2 smem[];
    float2 *tw = smem;
    float2 *buf = smem + tw_slots(a.tw_len);
    load_twiddles(tw, a.tw, a.tw_len);
    pdl_wait();
    const int l = threadIdx.x % LPT, t = threadIdx.x / LPT;
    const bool conj = a.conj != 0;
    for (int64_t tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
        __syncthreads();
        const TileId id = decode_tile(tile, a.tiles_c, a.g.A, LPT);
        const int64_t c = id.c0 + l;
        const bool valid = c < a.g.C;
        GLoad src{a.in + c * a.g.ic + id.a * a.g.ia + id.b * a.g.ib, a.g.ij, valid, conj};
        GStore dst{a.out + c * a.g.oc + id.a * a.g.oa + id.b * a.g.ob, a.g.ok, valid, conj};
        SmemCol<LPT> sm{buf + l};
        EngineFixed<N, T, 1, Rad>::template run<true, false>(t, src, sm, dst, tw);
    }
}

} // namespace fft3

#define FFT3_MIXED_ROW_J(N, T, LPT, MB, SH, PITCH, ...) \
    {N, (const void *)&fft3::k_mixed_j<N, T, LPT, MB, SH, PITCH, fft3::Radices<__VA_ARGS__>>},
#define FFT3_MIXED_ROW_C(N, T, LPT, MB, ...) \
    {N, (const void *)&fft3::k_mixed_c<N, T, LPT, MB, fft3::Radices<__VA_ARGS__>>},
