// slab_warp.cuh -- the x and y lines of n0 x n1 slabs in one block: rows from
// global memory through the registers of a few lanes of a warp (warp_fft.cuh)
// into shared memory, columns in place there, the slabs copied out.  Used by the
// slab executor of batched plans (k_slabz.cu) and the slab pass of single plans
// (k_slabw.cu); line lengths of FFT3_SLABZ_WARP_PLANS.
#pragma once

#include "seg_plans.h"
#include "warp_fft.cuh"

namespace fft3 {

namespace {

constexpr int kSzThreads = 256;

// Rows of the stacked slabs (x lines) straight from global memory into the
// shared buffer (rows `pitch` values apart, pitch odd): a row in the
// registers of L/2 lanes (warp_fft.cuh), 512 / L rows per round, no barrier;
// `w` is the table w_N^m (m < N).
template <int N, int R, int L>
__device__ __noinline__ void sz_rows_warp(const float2 *src, float2 *A, int pitch, int rows, const float2 *w,
                                          bool conj)
{
    using WL = WarpLine<N, R, L>;
    constexpr int RPR = kSzThreads / WL::W; // rows per round
    const int u = threadIdx.x % WL::W, l = threadIdx.x / WL::W;
    typename WL::Tw tw;
    WL::load_tw(tw, w, u);
    for (int r0 = 0; r0 < rows; r0 += RPR) {
        const int row = r0 + l;
        const bool valid = row < rows;
        pk2 v[2][R];
        WL::load(v, src + (int64_t)(valid ? row : 0) * N, u, valid, conj);
        WL::run(v, tw, u);
        if (valid) {
            float2 *ar = A + row * pitch;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int k0 = R * WL::rev(2 * u + e);
#pragma unroll
                for (int k = 0; k < R; ++k)
                    ar[k0 + k] = v[e][k];
            }
        }
    }
}

// Columns of the stacked slabs (y lines) in the registers of L/2 lanes
// (warp_fft.cuh): the lanes of a column read different rows of the buffer
// (pitch odd: conflict free), adjacent lane groups take adjacent columns, and
// each group writes its column's outputs back in place (a group owns its
// column: no barrier).
template <int N, int R, int L>
__device__ __noinline__ void sz_cols_warp(float2 *A, int pitch, int cols, int w, int slab_stride, const float2 *tw_w)
{
    using WL = WarpLine<N, R, L>;
    constexpr int CPR = kSzThreads / WL::W; // columns per round
    const int u = threadIdx.x % WL::W, l = threadIdx.x / WL::W;
    typename WL::Tw tw;
    WL::load_tw(tw, tw_w, u);
    for (int c0 = 0; c0 < cols; c0 += CPR) {
        const int c = c0 + l;
        const bool valid = c < cols;
        const int cs = valid ? c / w : 0, cc = valid ? c - cs * w : 0;
        float2 *p = A + cs * slab_stride + cc;
        pk2 v[2][R];
        WL::load_strided(v, p, pitch, u, valid, false);
        WL::run(v, tw, u);
        WL::store_strided(v, p, pitch, u, valid, false);
    }
}

// The stacked slabs (rows of n0 values, n0 even, `pitch` apart) to dst, where
// they are contiguous: each thread moves pairs of values of a row, 16-byte
// stores when dst is 16-byte aligned; conjugated for the inverse.
__device__ __noinline__ void sz_copy_out(const float2 *A, int pitch, int n0, int rows, float2 *dst, bool conj)
{
    const int half = n0 >> 1, rpp = kSzThreads / half; // rows per pass
    const int rr = threadIdx.x / half, x = 2 * (threadIdx.x - rr * half);
    if (rr >= rpp)
        return;
    const bool v4 = (reinterpret_cast<uintptr_t>(dst) & 15) == 0;
    for (int r = rr; r < rows; r += rpp) {
        float2 a = A[r * pitch + x], b = A[r * pitch + x + 1];
        if (conj) {
            a = cconj(a);
            b = cconj(b);
        }
        float2 *q = dst + (int64_t)r * n0 + x;
        if (v4) {
            *reinterpret_cast<float4 *>(q) = make_float4(a.x, a.y, b.x, b.y);
        } else {
            q[0] = a;
            q[1] = b;
        }
    }
}

__device__ __forceinline__ void sz_run_rows_warp(int n0, const float2 *src, float2 *A, int pitch, int rows,
                                                 const float2 *tw, const int *off, bool conj)
{
    int k = 0;
#define FFT3_SZ_WROW(N, R, L)                                                        \
    if (n0 == N) {                                                                   \
        sz_rows_warp<N, R, L>(src, A, pitch, rows, tw + off[k], conj);              \
        return;                                                                      \
    }                                                                                \
    ++k;
    FFT3_SLABZ_WARP_PLANS(FFT3_SZ_WROW)
#undef FFT3_SZ_WROW
}

__device__ __forceinline__ void sz_run_cols_warp(int n1, float2 *A, int pitch, int cols, int w, int slab_stride,
                                                 const float2 *tw, const int *off)
{
    int k = 0;
#define FFT3_SZ_WCOL(N, R, L)                                                        \
    if (n1 == N) {                                                                   \
        sz_cols_warp<N, R, L>(A, pitch, cols, w, slab_stride, tw + off[k]);          \
        return;                                                                      \
    }                                                                                \
    ++k;
    FFT3_SLABZ_WARP_PLANS(FFT3_SZ_WCOL)
#undef FFT3_SZ_WCOL
}

} // namespace

} // namespace fft3
