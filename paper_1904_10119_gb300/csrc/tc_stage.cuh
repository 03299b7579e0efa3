// tc_stage.cuh -- a radix-16 Stockham stage computed on the tensor cores in
// split BF16.
//
// The 16-point DFT of a butterfly is a dense product y = W x with
// W[k][r] = w_16^{kr}.  In real arithmetic, with x = (xr, xi) and
// W = Wr + i Wi, the outputs are yr = Wr xr - Wi xi and yi = Wi xr + Wr xi:
// one 32 x 32 real matrix applied to 32-element columns.  Eight butterflies
// form the N = 8 columns of an m16n8k16 BF16 MMA with FP32 accumulation; the
// 32 x 32 matrix is 2 x 2 blocks of 16 x 16 (rows: yr | yi, columns: xr | xi).
// Both operands are split into a high and a low BF16 part, v = v_hi + v_lo
// with v_hi = bf16(v) and v_lo = bf16(v - v_hi), and three products are
// accumulated: W_hi x_hi + W_hi x_lo + W_lo x_hi (W_lo x_lo is dropped).
// Twiddles are applied to x in FP32 before the split.
//
// Fragment layouts of mma.sync.m16n8k16 (g = lane / 4, t = lane % 4):
//   A (16 x 16, row-major): {a0,a1} = (g, 2t..2t+1), {a2,a3} = (g+8, 2t..),
//                           {a4,a5} = (g, 2t+8..), {a6,a7} = (g+8, 2t+8..)
//   B (16 x 8, column):     {b0,b1} = (2t..2t+1, g), {b2,b3} = (2t+8.., g)
//   C (16 x 8):             {c0,c1} = (g, 2t..2t+1), {c2,c3} = (g+8, 2t..)
// so thread (g, t) supplies inputs r in {2t, 2t+1, 2t+8, 2t+9} of butterfly
// g of its group and receives outputs k in {g, g+8} of butterflies 2t, 2t+1.
#pragma once

#include <cuda_bf16.h>

#include "fft_engine.cuh"

namespace fft3 {

__device__ __forceinline__ uint32_t bf16x2_bits(__nv_bfloat16 lo, __nv_bfloat16 hi)
{
    return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

// (x0, x1) -> packed high parts and packed low parts.
__device__ __forceinline__ void split_pair(float x0, float x1, uint32_t &hi, uint32_t &lo)
{
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(x1), "f"(x0));
    const float l0 = x0 - __uint_as_float(hi << 16), l1 = x1 - __uint_as_float(hi & 0xffff0000u);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(l1), "f"(l0));
}

__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
                 "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The real-ified DFT_16 as split-BF16 A fragments of this lane.
struct TcW {
    uint32_t hi[2][2][4], lo[2][2][4]; // [row block: yr|yi][column block: xr|xi][register]
};

// w16[m] = w_16^m (float32, from the FP64 generator).
__device__ __forceinline__ void tc_build_w(TcW &w, const float2 *w16)
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int mb = 0; mb < 2; ++mb)
#pragma unroll
        for (int kb = 0; kb < 2; ++kb)
#pragma unroll
            for (int reg = 0; reg < 4; ++reg) {
                const int i = g + ((reg & 1) ? 8 : 0);
                const int j0 = 2 * t + ((reg & 2) ? 8 : 0);
                float v[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float2 c = w16[(i * (j0 + e)) & 15];
                    // blocks: (yr,xr) = Wr, (yr,xi) = -Wi, (yi,xr) = Wi, (yi,xi) = Wr
                    v[e] = (mb == kb) ? c.x : (mb == 0 ? -c.y : c.y);
                }
                split_pair(v[0], v[1], w.hi[mb][kb][reg], w.lo[mb][kb][reg]);
            }
}

// Butterfly (line, q) of group `grp`, lane group g (GROUP_LINES: a group is
// 8 adjacent lines at one q; otherwise 8 adjacent q of one line).
template <int NB, int LPT, bool GROUP_LINES>
__device__ __forceinline__ void tc_butterfly(int grp, int n, int &line, int &q)
{
    if constexpr (GROUP_LINES) {
        q = grp / (LPT / 8);
        line = (grp % (LPT / 8)) * 8 + n;
    } else {
        line = grp / (NB / 8);
        q = (grp % (NB / 8)) * 8 + n;
    }
}

// One radix-16 stage of lines of N points on the tensor cores: the NB*LPT
// butterflies (line, q) of a tile, in groups of 8, each warp taking every
// nwarps-th group.  Src and Dst are tile accessors acc(line, pos) and must not
// alias (the stage streams group by group; the caller ping-pongs buffers).
// `warp` / `nwarps`: this warp's index among the warps sharing the stage (by
// default every warp of the block).
template <int N, int NS, int LPT, bool GROUP_LINES, class Src, class Dst>
__device__ __forceinline__ void tc_stage16(const Src &src, const Dst &dst, const float2 *tw, const TcW &w,
                                           int warp = -1, int nwarps = 0)
{
    constexpr int NB = N / 16;
    constexpr int NGROUPS = NB * LPT / 8;
    const int lane = threadIdx.x & 31;
    if (warp < 0) {
        warp = threadIdx.x >> 5;
        nwarps = blockDim.x >> 5;
    }
    const int g = lane >> 2, t = lane & 3;
    for (int grp = warp; grp < NGROUPS; grp += nwarps) {
        int line, q;
        tc_butterfly<NB, LPT, GROUP_LINES>(grp, g, line, q);
        float2 v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int r = 2 * t + (e & 1) + ((e & 2) ? 8 : 0);
            float2 x = src(line, q + r * NB);
            if constexpr (NS > 1) {
                if (r > 0)
                    x = cmul(x, tw[(r - 1) * NS + (q % NS)]);
            }
            v[e] = x;
        }
        uint32_t bh[2][2], bl[2][2]; // [xr|xi][register]
        split_pair(v[0].x, v[1].x, bh[0][0], bl[0][0]);
        split_pair(v[2].x, v[3].x, bh[0][1], bl[0][1]);
        split_pair(v[0].y, v[1].y, bh[1][0], bl[1][0]);
        split_pair(v[2].y, v[3].y, bh[1][1], bl[1][1]);
        float d[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
        for (int mb = 0; mb < 2; ++mb)
#pragma unroll
            for (int kb = 0; kb < 2; ++kb) {
                // small products first, the hi x hi product last
                mma_bf16_16816(d[mb], w.lo[mb][kb], bh[kb][0], bh[kb][1]);
                mma_bf16_16816(d[mb], w.hi[mb][kb], bl[kb][0], bl[kb][1]);
                mma_bf16_16816(d[mb], w.hi[mb][kb], bh[kb][0], bh[kb][1]);
            }
        // this lane holds outputs k in {g, g+8} of butterflies n in {2t, 2t+1}
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int k = g + ((e & 2) ? 8 : 0);
            int ol, oq;
            tc_butterfly<NB, LPT, GROUP_LINES>(grp, 2 * t + (e & 1), ol, oq);
            const int base = (NS == 1) ? oq * 16 : (oq / NS) * NS * 16 + (oq % NS);
            dst(ol, base + k * NS, make_float2(d[0][e], d[1][e]));
        }
    }
}

// The same stage on a position-major tile of 16 columns (value of position j,
// column c at p[j * 16 + c]), a warp taking the 16 butterflies of one q at a
// time.  A lane reads two adjacent columns, 2g and 2g + 1, of its four inputs r
// with 16-byte loads, so a warp's load covers whole 128-byte rows (the eight
// columns of one MMA alone put its four rows on the same banks: two wavefronts
// for one); the even columns form one MMA's N side, the odd ones another's, and
// their outputs land as four adjacent columns 4t .. 4t + 3 per lane, stored with
// 16-byte stores (the two halves in opposite order in odd rows, so that eight
// lanes cover all banks).  `src` and `dst` may be the same tile where a
// butterfly's outputs take its inputs' places (NS * 16 == N): a warp has read
// its inputs when its products run.
template <int N, int NS>
__device__ __forceinline__ void tc_stage16_cols16(const float2 *src, float2 *dst, bool conj, const float2 *tw,
                                                  const TcW &w, int warp, int nwarps)
{
    constexpr int NB = N / 16;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const float sg = conj ? -1.f : 1.f;
    for (int q = warp; q < NB; q += nwarps) {
        float2 v[2][4]; // [column 2g + h][input]
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int r = 2 * t + (e & 1) + ((e & 2) ? 8 : 0);
            const float4 x = *reinterpret_cast<const float4 *>(src + (q + r * NB) * 16 + 2 * g);
            v[0][e] = make_float2(x.x, sg * x.y);
            v[1][e] = make_float2(x.z, sg * x.w);
            if constexpr (NS > 1) {
                if (r > 0) {
                    const float2 c = tw[(r - 1) * NS + (q % NS)];
                    v[0][e] = cmul(v[0][e], c);
                    v[1][e] = cmul(v[1][e], c);
                }
            }
        }
        float d[2][2][4] = {}; // [h][yr | yi][fragment]
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t bh[2][2], bl[2][2]; // [xr|xi][register]
            split_pair(v[h][0].x, v[h][1].x, bh[0][0], bl[0][0]);
            split_pair(v[h][2].x, v[h][3].x, bh[0][1], bl[0][1]);
            split_pair(v[h][0].y, v[h][1].y, bh[1][0], bl[1][0]);
            split_pair(v[h][2].y, v[h][3].y, bh[1][1], bl[1][1]);
#pragma unroll
            for (int mb = 0; mb < 2; ++mb)
#pragma unroll
                for (int kb = 0; kb < 2; ++kb) {
                    mma_bf16_16816(d[h][mb], w.lo[mb][kb], bh[kb][0], bh[kb][1]);
                    mma_bf16_16816(d[h][mb], w.hi[mb][kb], bl[kb][0], bl[kb][1]);
                    mma_bf16_16816(d[h][mb], w.hi[mb][kb], bh[kb][0], bh[kb][1]);
                }
        }
        const int base = (NS == 1) ? q * 16 : (q / NS) * NS * 16 + (q % NS);
#pragma unroll
        for (int k8 = 0; k8 < 2; ++k8) {
            float4 *o = reinterpret_cast<float4 *>(dst + (base + (g + 8 * k8) * NS) * 16 + 4 * t);
            const float4 lo = make_float4(d[0][0][2 * k8], d[0][1][2 * k8], d[1][0][2 * k8], d[1][1][2 * k8]);
            const float4 hi = make_float4(d[0][0][2 * k8 + 1], d[0][1][2 * k8 + 1], d[1][0][2 * k8 + 1],
                                          d[1][1][2 * k8 + 1]);
            const bool odd = g & 1;
            o[odd ? 1 : 0] = odd ? hi : lo;
            o[odd ? 0 : 1] = odd ? lo : hi;
        }
    }
}

} // namespace fft3
