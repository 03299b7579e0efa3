// k_pass64.cuh -- complex128 line passes with a compile-time radix list, the
// precision of the paper's experiments (Section 4: complex double): the
// Stockham stages of Section 2.1 (Eq. ct applied repeatedly, fft_engine.cuh),
// one pass per dimension as in the pencil-pencil-pencil definition of Section
// 2.3, computed in 64-bit block fixed point (fix64.cuh).
//   k_pass_j64  contiguous lines (ij == 1, ok == 1), T threads per line, LPT
//               lines per tile, one padded line buffer in shared memory (the
//               first stage reads global memory, the last writes it).
//   k_pass_c64  strided lines (ic == 1, oc == 1), tiles of 8 adjacent
//               columns (128-byte rows), position-major shared layout.
// A tile: every thread loads the inputs of its first butterflies, the line's
// largest magnitudes are reduced in shared memory, the inputs become integers, and
// the stages run as in FP32, the line shifted up to full scale after each, the last
// one rounding to FP64.  A tile with a line
// that the integers do not take (fix_ok) is redone from its input by the FP64
// stages; every thread learns that at the barrier that ends the first stage,
// before anything has been stored.
//
// What bounds it: latency at 16 warps per SM (128 registers: 16 values of four
// words each); the ALU pipe is 57% busy, issue 52%; the FP64 pipe carries only half
// of the final roundings.  256^3: 579 us, 2.8 TB/s per pass, against 2502 us with
// FP64 stages (2 lanes per clock and SM); without the shifts up, which dominated
// lines need, 565.  Tried: radix-8 plans (24 warps, one exchange more) 671 us; up
// to 168 registers (12 warps) 630 us.
// The runtime-radix kernel (k_pass_g64) covers the other lengths.
#pragma once

#include "fix64.cuh"
#include "pass_kernels.cuh"
#include "plans.h"

namespace fft3 {

struct G64Load { // element j at p[j * s]
    const double2 *p;
    int64_t s;
    bool valid, conj;
    __device__ __forceinline__ double2 operator()(int j) const
    {
        const double2 v = valid ? p[(int64_t)j * s] : make_double2(0.0, 0.0);
        return conj ? cconj(v) : v;
    }
};
struct G64Store {
    double2 *p;
    int64_t s;
    bool valid, conj;
    __device__ __forceinline__ void operator()(int k, double2 v) const
    {
        if (valid)
            p[(int64_t)k * s] = conj ? cconj(v) : v;
    }
};
template <class C, int SH>
struct Smem64Line { // line-major, position p at p + (p >> SH), SH = 0: p
    C *p;
    __device__ __forceinline__ static int pos(int j)
    {
        if constexpr (SH > 0)
            return j + (j >> SH);
        else
            return j;
    }
    __device__ __forceinline__ C operator()(int j) const { return p[pos(j)]; }
    __device__ __forceinline__ void operator()(int k, C v) const { p[pos(k)] = v; }
};
template <class C, int LPT>
struct Smem64Col { // element j of column l at p[j*LPT] (p = buffer + l)
    C *p;
    __device__ __forceinline__ C operator()(int j) const { return p[j * LPT]; }
    __device__ __forceinline__ void operator()(int k, C v) const { p[k * LPT] = v; }
};
struct FixStore { // rounds to FP64 and stores
    G64Store g;
    int sh;
    __device__ __forceinline__ void operator()(int k, fix2 v) const
    {
        // one component on the integer pipe, one on the FP64 pipe: 256^3 in 594 us, both on the
        // FP64 pipe 596, both on the integer pipe 639 (512-point lines: 451, 474, 449 us)
        g(k, make_double2(from_fix_int(v.x, sh), from_fix(v.y, sh)));
    }
};

__device__ __forceinline__ unsigned char *smem64()
{
    extern __shared__ __align__(16) unsigned char s64_raw[];
    return s64_raw;
}

// Powers of two the integer stages of a radix list scale down by, and the least of their fix_exact_bits.
template <class Rad>
struct FixScale;
template <int R>
struct FixScale<Radices<R>> {
    static constexpr int value = BflyFix<R, false>::scale;
    static constexpr int exact = fix_exact_bits(BflyFix<R, false>::scale);
};
template <int R, int R2, int... Rest>
struct FixScale<Radices<R, R2, Rest...>> {
    using Later = FixScale<Radices<R2, Rest...>>;
    static constexpr int value = BflyFix<R, false>::scale + 2 + Later::value;
    static constexpr int exact = fix_exact_bits(BflyFix<R, false>::scale) < Later::exact ? fix_exact_bits(BflyFix<R, false>::scale)
                                                                                  : Later::exact;
};

// OR of a line's normalisation words over the adjacent lanes that hold it, into
// the line's shared slot.
template <int SEG>
__device__ __forceinline__ void norm_out(unsigned acc, unsigned *slot)
{
#pragma unroll
    for (int o = 1; o < SEG; o <<= 1)
        acc |= __shfl_xor_sync(0xffffffffu, acc, o);
    if (SEG == 1 || (threadIdx.x & (SEG - 1)) == 0)
        atomicOr(slot, acc);
}

// Stages after the first: shared buffer to shared buffer, the last to `dst`.
// `nrm` is the slot the stage before left its normalisation word in, the next
// stage's is NSTEP words on.
template <int N, int T, int NS, class Rad, int SEG, int NSTEP, bool RN>
struct FixRest;
template <int N, int T, int NS, int R, int... Rest, int SEG, int NSTEP, bool RN>
struct FixRest<N, T, NS, Radices<R, Rest...>, SEG, NSTEP, RN> {
    static constexpr bool LAST = sizeof...(Rest) == 0;
    template <class Sm>
    __device__ __forceinline__ static void run(int t, const Sm &sm, FixStore dst, const root62 *tw, unsigned *nrm)
    {
        constexpr int NB = N / R, BPT = (NB + T - 1) / T;
        constexpr bool FULL = NB % T == 0;
        const int up = norm_shift(*nrm);
        dst.sh -= up;
        fix2 v[BPT][R];
        unsigned acc = 0;
#pragma unroll
        for (int b = 0; b < BPT; ++b) {
            const int q = t + b * T;
            if (FULL || q < NB) {
#pragma unroll
                for (int r = 0; r < R; ++r)
                    v[b][r] = sm(q + r * NB);
            }
        }
        if constexpr (!LAST)
            __syncthreads();
#pragma unroll
        for (int b = 0; b < BPT; ++b) {
            const int q = t + b * T;
            if (FULL || q < NB) {
                const int k = q % NS;
                if (up > 0) {
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        v[b][r] = shl(v[b][r], up);
                }
                v[b][0] = quarter<RN>(v[b][0]);
#pragma unroll
                for (int r = 1; r < R; ++r)
                    v[b][r] = cmul62(v[b][r], tw[(r - 1) * NS + k]);
                BflyFix<R, RN>::run(v[b]);
                const int base = (q / NS) * NS * R + k;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if constexpr (LAST) {
                        dst(base + r * NS, v[b][r]);
                    } else {
                        sm(base + r * NS, v[b][r]);
                        acc |= norm_word(v[b][r].x) | norm_word(v[b][r].y);
                    }
                }
            }
        }
        if constexpr (!LAST) {
            norm_out<SEG>(acc, nrm + NSTEP);
            __syncthreads();
            FixRest<N, T, NS * R, Radices<Rest...>, SEG, NSTEP, RN>::run(t, sm, dst, tw + (R - 1) * NS, nrm + NSTEP);
        }
    }
};

// The FP64 stages of one tile (twiddles read from global memory).
template <int N, int T, class Rad, class Sm>
__device__ __noinline__ void tile_fp64(int t, G64Load src, Sm sm, G64Store dst, const double2 *tw)
{
    __syncthreads();
    EngineFixed<N, T, 1, Rad>::template run<true, false>(t, src, sm, dst, tw);
}

// One tile's line of this thread: `slot` is the line's first shared word (largest
// magnitude words of the real and the imaginary parts, then a normalisation word
// per stage but the last; zero on entry), the following ones NSTEP words apart;
// SEG > 1 the adjacent lanes of a warp that hold one line.
template <int N, int T, class Rad, int SEG, int NSTEP>
struct FixTile;
template <int N, int T, int R, int... Rest, int SEG, int NSTEP>
struct FixTile<N, T, Radices<R, Rest...>, SEG, NSTEP> {
    using Rad = Radices<R, Rest...>;
    template <class SmF, class SmD>
    __device__ __forceinline__ static void run(int t, const G64Load &src, const SmF &sm, const SmD &smd,
                                               const G64Store &dst, const root62 *tw, const double2 *twd,
                                               unsigned *slot)
    {
        constexpr int NB = N / R, BPT = (NB + T - 1) / T;
        constexpr bool FULL = NB % T == 0, ONE = sizeof...(Rest) == 0;
        constexpr bool RN = fix_rounds(BflyFix<R, false>::scale);
        static_assert(!ONE || T == 1, "a line of one stage belongs to one thread");
        double2 x[BPT][R];
        FixScan scan;
        scan.zeros = ONE;
        FixMag &line = scan.line;
#pragma unroll
        for (int b = 0; b < BPT; ++b) {
            const int q = t + b * T;
            if (FULL || q < NB) {
#pragma unroll
                for (int r = 0; r < R; ++r)
                    x[b][r] = src(q + r * NB);
                FixMag m{0u, 0u};
#pragma unroll
                for (int r = 0; r < R; ++r)
                    mag_max(m, x[b][r]);
                scan.add(m);
            }
        }
        if constexpr (!ONE) {
#pragma unroll
            for (int o = 1; o < SEG; o <<= 1) {
                line.re = max(line.re, __shfl_xor_sync(0xffffffffu, line.re, o));
                line.im = max(line.im, __shfl_xor_sync(0xffffffffu, line.im, o));
            }
            if (SEG == 1 || (threadIdx.x & (SEG - 1)) == 0) {
                atomicMax(slot, line.re);
                atomicMax(slot + NSTEP, line.im);
            }
            __syncthreads();
            line.re = slot[0];
            line.im = slot[NSTEP];
        }
        const bool ok = fix_ok(scan, fix_strict(N, R), FixScale<Rad>::exact);
        const int emax = fix_emax(mag_all(line));
        // 2 and 4 points are additions alone, exact in FP64 more often than not
        if (ONE && (R == 2 || R == 4 || !ok)) {
            Bfly<R>::run(x[0]);
#pragma unroll
            for (int r = 0; r < R; ++r)
                dst(r, x[0][r]);
            return;
        }
        unsigned acc = 0;
        const FixStore out{dst, emax - 1081 + FixScale<Rad>::value};
#pragma unroll
        for (int b = 0; b < BPT; ++b) {
            const int q = t + b * T;
            if (FULL || q < NB) {
                fix2 v[R];
#pragma unroll
                for (int r = 0; r < R; ++r)
                    v[r] = fix2{to_fix<false>(x[b][r].x, emax), to_fix<false>(x[b][r].y, emax)};
                BflyFix<R, RN>::run(v);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    if constexpr (ONE) {
                        out(r, v[r]);
                    } else {
                        sm(q * R + r, v[r]);
                        acc |= norm_word(v[r].x) | norm_word(v[r].y);
                    }
                }
            }
        }
        if constexpr (!ONE) {
            norm_out<SEG>(acc, slot + 2 * NSTEP);
            if (__syncthreads_or(!ok)) {
                tile_fp64<N, T, Rad>(t, src, smd, dst, twd);
                return;
            }
            FixRest<N, T, R, Radices<Rest...>, SEG, NSTEP, RN>::run(t, sm, out, tw + (R - 1), slot + 2 * NSTEP);
        }
    }
};

// The tile loop of both kernels; LINES: contiguous lines, else columns, G tiles
// side by side in a block (one barrier domain).
template <int N, int T, class Rad, int LPT, int G, bool LINES, int SH = 4, int PITCH = line_pitch(N)>
__device__ __forceinline__ void pass64(const PassArgs &a)
{
    constexpr int GT = T * LPT, NT = GT * G;
    constexpr int WORDS = 1 + Rad::count; // FixTile's words of a line
    __shared__ unsigned slots[2][WORDS][G * LPT]; // [tile parity][word][line]
    root62 *tw = reinterpret_cast<root62 *>(smem64());
    unsigned char *buf = smem64() + (size_t)tw_slots(a.tw_len) * 16;
    const root62 *twg = reinterpret_cast<const root62 *>(a.tw_fix);
    for (int i = threadIdx.x; i < a.tw_len; i += NT)
        tw[i] = twg[i];
    pdl_wait();
    const double2 *twd = reinterpret_cast<const double2 *>(a.tw);
    const double2 *in = reinterpret_cast<const double2 *>(a.in);
    double2 *out = reinterpret_cast<double2 *>(a.out);
    const int g = G > 1 ? threadIdx.x / GT : 0, gt = G > 1 ? threadIdx.x % GT : threadIdx.x;
    const int t = LINES ? gt % T : gt / LPT;
    const int l = LINES ? gt / T : gt % LPT;
    // lanes of a line that are adjacent in a warp (whole warps only)
    constexpr int SEG = LINES && NT % 32 == 0 && (T & (T - 1)) == 0 ? (T < 32 ? T : 32) : 1;
    const bool conj = a.conj != 0;
    int par = 0;
    for (int64_t tile0 = (int64_t)blockIdx.x * G; tile0 < a.ntiles; tile0 += (int64_t)gridDim.x * G, par ^= 1) {
        for (int i = threadIdx.x; i < WORDS * G * LPT; i += NT)
            slots[par][i / (G * LPT)][i % (G * LPT)] = 0;
        __syncthreads();
        const bool live = G == 1 || tile0 + g < a.ntiles;
        const TileId id = decode_tile(live ? tile0 + g : tile0, a.tiles_c, a.g.A, LPT);
        const int64_t c = id.c0 + l;
        const bool valid = live && c < a.g.C;
        const G64Load src{in + c * a.g.ic + id.a * a.g.ia + id.b * a.g.ib, LINES ? 1 : a.g.ij, valid, conj};
        const G64Store dst{out + c * a.g.oc + id.a * a.g.oa + id.b * a.g.ob, LINES ? 1 : a.g.ok, valid, conj};
        unsigned *slot = &slots[par][0][g * LPT + l];
        if constexpr (LINES) {
            const Smem64Line<fix2, SH> sm{reinterpret_cast<fix2 *>(buf) + l * PITCH};
            const Smem64Line<double2, SH> smd{reinterpret_cast<double2 *>(buf) + l * PITCH};
            FixTile<N, T, Rad, SEG, G * LPT>::run(t, src, sm, smd, dst, tw, twd, slot);
        } else {
            const Smem64Col<fix2, LPT> sm{reinterpret_cast<fix2 *>(buf) + g * (LPT * N) + l};
            const Smem64Col<double2, LPT> smd{reinterpret_cast<double2 *>(buf) + g * (LPT * N) + l};
            FixTile<N, T, Rad, SEG, G * LPT>::run(t, src, sm, smd, dst, tw, twd, slot);
        }
    }
}

// at most 128 registers a thread: 16 warps per SM
constexpr int fix_min_blocks(int threads) { return threads >= 512 ? 1 : 512 / threads; }

template <int N, int T, class Rad, int LPT, int SH = 4, int PITCH = line_pitch(N)>
__global__ void __launch_bounds__(T *LPT, fix_min_blocks(T *LPT)) k_pass_j64(PassArgs a)
{
    pass64<N, T, Rad, LPT, 1, true, SH, PITCH>(a);
}

template <int N, int T, class Rad, int LPT, int G>
__global__ void __launch_bounds__(T *LPT *G, fix_min_blocks(T *LPT *G)) k_pass_c64(PassArgs a)
{
    pass64<N, T, Rad, LPT, G, false>(a);
}

} // namespace fft3
