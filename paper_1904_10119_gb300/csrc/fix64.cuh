// fix64.cuh -- complex128 line transforms in 64-bit block fixed point.
//
// GB300 issues 2 FP64 operations per clock and SM against 64 integer adds and
// 64 wide integer multiply-adds, so an FP64 butterfly is bound by the FP64
// pipe at a few per cent of the memory bandwidth.  Here a line's values are
// converted once to 64-bit integers with one exponent per line, the Stockham
// stages run on integers, and the result is rounded once to FP64.
//
// Format: a component is an integer V, its value V * 2^(unit exponent).  Moduli
// stay below 2^62: every radix-4 layer takes moduli below 2^60 (a butterfly of
// four grows them at most fourfold) and the multiplication before it scales by
// 1/4, so the unit exponent rises by two per layer (see cmul62).  Radix 2, 3
// and 8 = 4 * 2 layers fit the same rule; radix 5 takes one more halving.
//
// Error: products are rounded to the unit, shifts down truncate, so a layer adds
// about one unit to a value.  After every stage but the last the line is shifted up
// to full scale (block floating point), so scale that a line does not grow by is not
// lost, and the result is rounded once to FP64.  Lists that lose more to their first
// stage's scale (radix 10, 15, 32) round the shifts as well, and lists of run-time
// length the conversion of the input too (256^3: 1.5% for the shifts, 10% for the
// conversions).
// Which lines take them: those in which no part is small enough to lose what
// FP64 would keep.  Components share the largest one's exponent, so one that is
// 2^-d of it keeps 59 - d bits.  Next to the largest values FP64 rounds to 53 bits
// as well; what it keeps apart are real and imaginary parts, where no twiddle mixes
// them.  So the largest real and the largest imaginary part must be within 2^5 of
// each other, or one of them all zeros; and in a line that may be a single value
// (a first-stage butterfly of zeros, or one stage in all), which FP64 carries
// through the first element's additions as it is, so close that no stage shifts a
// bit of it out (fix_exact_bits).  Lists that lose more of the scale, in a radix-32
// first stage or over more than 2048 points from radix 5 on, are too coarse for
// spikes over a background: there every first-stage butterfly must hold a value of
// 2^-4 of the largest (fix_strict).
// What is given up: results that are small because larger values cancel exactly are
// good to about 2^-57 of the line's largest value, where FP64 may hold more bits of them.
// Measured on the host over every radix list of the plans (relative 2-norm per line
// against long double; flat, real, tones, bumps, spectra, constants and spikes over
// a background of 10^-1 to 10^-12): on the lines taken at most the error of the same
// stages in FP64: flat lines 0.5e-16 against 2.9e-16, the hardest (4096 points, a
// spike over 10^-12) 2.1e-16 against 2.4e-16.  A shift up after the first stage of
// lines from 512 points on alone left a spike over 1e-3 with 1.1e-15 at 256 points
// as 8 x 8 x 4.
// Other lines, and those with an infinity, a NaN or values so large or small
// that their exponent cannot be carried (below 2^-895, above 2^1007), take the
// FP64 stages.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#ifndef FFT3_HD
#define FFT3_HD __host__ __device__ __forceinline__
#endif

namespace fft3 {

struct __align__(16) fix2 {
    long long x, y;
};

FFT3_HD fix2 cadd(fix2 a, fix2 b) { return fix2{a.x + b.x, a.y + b.y}; }
FFT3_HD fix2 csub(fix2 a, fix2 b) { return fix2{a.x - b.x, a.y - b.y}; }
FFT3_HD fix2 mul_mi(fix2 a) { return fix2{a.y, -a.x}; }
// Shifts down, rounded (RN) or not: rounding costs two instructions a component.
template <bool RN>
FFT3_HD fix2 quarter(fix2 a)
{
    constexpr int h = RN ? 2 : 0;
    return fix2{(a.x + h) >> 2, (a.y + h) >> 2};
}
template <bool RN>
FFT3_HD fix2 half(fix2 a)
{
    constexpr int h = RN ? 1 : 0;
    return fix2{(a.x + h) >> 1, (a.y + h) >> 1};
}
FFT3_HD fix2 shl(fix2 a, int s)
{
    return fix2{(long long)((unsigned long long)a.x << s), (long long)((unsigned long long)a.y << s)};
}

FFT3_HD long long mad_wide(int a, int b, long long c) { return (long long)a * b + c; }

// V = h * 2^32 + l with l in [-2^31, 2^31).
FFT3_HD int bal_lo(long long v) { return (int)(unsigned)v; }
FFT3_HD int bal_hi(long long v) { return (int)(v >> 32) + (int)((unsigned)v >> 31); }

// A root of unity times 2^62, each component as balanced 32-bit halves, the low
// halves in (-2^31, 2^31) so that they can be negated.
struct __align__(16) root62 {
    int rh, rl, ih, il;
};

// a * w / 4: the product with w * 2^62, shifted down by 64 and rounded.  The
// products of the low halves (below half a unit) are left out.  With moduli
// below 2^62 the middle sum stays below 2^62.6.
FFT3_HD fix2 cmul62(fix2 a, root62 w)
{
    const int ah = bal_hi(a.x), al = bal_lo(a.x), bh = bal_hi(a.y), bl = bal_lo(a.y);
    const int nih = -w.ih, nil = -w.il;
    long long m = mad_wide(ah, w.rl, 1ll << 31);
    m = mad_wide(al, w.rh, m);
    m = mad_wide(bh, nil, m);
    m = mad_wide(bl, nih, m);
    long long r = mad_wide(ah, w.rh, (int)(m >> 32));
    r = mad_wide(bh, nih, r);
    m = mad_wide(ah, w.il, 1ll << 31);
    m = mad_wide(al, w.ih, m);
    m = mad_wide(bh, w.rl, m);
    m = mad_wide(bl, w.rh, m);
    long long i = mad_wide(ah, w.ih, (int)(m >> 32));
    i = mad_wide(bh, w.rh, i);
    return fix2{r, i};
}

// a * c / 4 for a real constant c * 2^62 in the same halves.
FFT3_HD long long rmul62(long long a, int ch, int cl)
{
    const int ah = bal_hi(a), al = bal_lo(a);
    long long m = mad_wide(ah, cl, 1ll << 31);
    m = mad_wide(al, ch, m);
    return mad_wide(ah, ch, (int)(m >> 32));
}

// cos(k pi / 16) * 2^62 for k = 0..8, from which every power of w_32 follows.
constexpr long long kFxC32[9] = {4611686018427387904ll, 4523073764714963030ll, 4260642322793532497ll,
                                 3834476785802888710ll, 3260954456333195553ll, 2562115475870945497ll,
                                 1764815834521887442ll, 899695310372275547ll, 0ll};
FFT3_HD constexpr int const_hi(long long v) { return (int)((v + (1ll << 31)) >> 32); }
FFT3_HD constexpr int const_lo(long long v) { return (int)(v - ((long long)const_hi(v) << 32)); }
FFT3_HD constexpr long long fx_cos32(int m)
{
    m &= 31;
    return m <= 8 ? kFxC32[m] : m < 16 ? -kFxC32[16 - m] : m < 24 ? -fx_cos32(m - 16) : kFxC32[32 - m];
}

// a * w_32^M / 4, M known at compile time.
template <int M, bool RN>
FFT3_HD fix2 mul_w32_4(fix2 a)
{
    if constexpr (M == 0) {
        return quarter<RN>(a);
    } else if constexpr (M == 8) {
        return quarter<RN>(mul_mi(a));
    } else {
        constexpr long long c = fx_cos32(M), s = fx_cos32(M - 8); // w = c - i s
        return cmul62(a, root62{const_hi(c), const_lo(c), const_hi(-s), const_lo(-s)});
    }
}

// In-register DFT_R of values with moduli below 2^60 (2^59 for R = 5); results
// below 2^62.  scale: powers of two the result is scaled down by; RN: shifts down
// are rounded.
template <int R, bool RN>
struct BflyFix;

template <bool RN>
struct BflyFix<2, RN> {
    static constexpr int scale = 0;
    FFT3_HD static void run(fix2 *v)
    {
        const fix2 a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    }
};

template <bool RN>
struct BflyFix<4, RN> {
    static constexpr int scale = 0;
    FFT3_HD static void run(fix2 *v)
    {
        const fix2 t0 = cadd(v[0], v[2]), t1 = csub(v[0], v[2]);
        const fix2 t2 = cadd(v[1], v[3]), t3 = mul_mi(csub(v[1], v[3]));
        v[0] = cadd(t0, t2);
        v[2] = csub(t0, t2);
        v[1] = cadd(t1, t3);
        v[3] = csub(t1, t3);
    }
};

// 8 = 2 * 4 and 16 = 4 * 4 by Eq. ct, as the floating-point butterflies, the
// inner twiddles scaling by 1/4.
template <bool RN>
struct BflyFix<8, RN> {
    static constexpr int scale = 2;
    FFT3_HD static void run(fix2 *v)
    {
        fix2 e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
        BflyFix<4, RN>::run(e);
        BflyFix<4, RN>::run(o);
        o[0] = mul_w32_4<0, RN>(o[0]);
        o[1] = mul_w32_4<4, RN>(o[1]);
        o[2] = mul_w32_4<8, RN>(o[2]);
        o[3] = mul_w32_4<12, RN>(o[3]);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const fix2 q = quarter<RN>(e[k]);
            v[k] = cadd(q, o[k]);
            v[k + 4] = csub(q, o[k]);
        }
    }
};

template <bool RN>
struct BflyFix<16, RN> {
    static constexpr int scale = 2;
    FFT3_HD static void run(fix2 *v)
    {
        fix2 t[4][4];
#pragma unroll
        for (int i0 = 0; i0 < 4; ++i0) {
#pragma unroll
            for (int i1 = 0; i1 < 4; ++i1)
                t[i0][i1] = v[i0 + 4 * i1];
            BflyFix<4, RN>::run(t[i0]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            t[0][k] = quarter<RN>(t[0][k]);
        t[1][0] = quarter<RN>(t[1][0]);
        t[1][1] = mul_w32_4<2, RN>(t[1][1]);
        t[1][2] = mul_w32_4<4, RN>(t[1][2]);
        t[1][3] = mul_w32_4<6, RN>(t[1][3]);
        t[2][0] = quarter<RN>(t[2][0]);
        t[2][1] = mul_w32_4<4, RN>(t[2][1]);
        t[2][2] = mul_w32_4<8, RN>(t[2][2]);
        t[2][3] = mul_w32_4<12, RN>(t[2][3]);
        t[3][0] = quarter<RN>(t[3][0]);
        t[3][1] = mul_w32_4<6, RN>(t[3][1]);
        t[3][2] = mul_w32_4<12, RN>(t[3][2]);
        t[3][3] = mul_w32_4<18, RN>(t[3][3]);
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            fix2 c[4] = {t[0][k1], t[1][k1], t[2][k1], t[3][k1]};
            BflyFix<4, RN>::run(c);
#pragma unroll
            for (int k0 = 0; k0 < 4; ++k0)
                v[k1 + 4 * k0] = c[k0];
        }
    }
};

// 32 = 2 * 16 (the radix-32 plan of 1024 points).
template <int K, bool RN>
struct Tw32Fix {
    FFT3_HD static void run(fix2 *o)
    {
        o[K] = mul_w32_4<K, RN>(o[K]);
        if constexpr (K + 1 < 16)
            Tw32Fix<K + 1, RN>::run(o);
    }
};

template <bool RN>
struct BflyFix<32, RN> {
    static constexpr int scale = 4;
    FFT3_HD static void run(fix2 *v)
    {
        fix2 e[16], o[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            e[i] = v[2 * i];
            o[i] = v[2 * i + 1];
        }
        BflyFix<16, RN>::run(e);
        BflyFix<16, RN>::run(o);
        Tw32Fix<0, RN>::run(o);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const fix2 q = quarter<RN>(e[k]);
            v[k] = cadd(q, o[k]);
            v[k + 16] = csub(q, o[k]);
        }
    }
};

// Constants of DFT_3 and DFT_5 times 2^64, as the parts below 1/2 that a signed
// 64-bit word holds: sin(2 pi/3) = 1 - f etc., so a product keeps every unit.
constexpr long long kFx1mS3 = 2471395088767036514ll;  // 1 - sin(2 pi / 3)
constexpr long long kFxC51 = 5700357409661599243ll;   // cos(2 pi / 5)
constexpr long long kFx1pC52 = 3523014627193176565ll; // 1 + cos(4 pi / 5)
constexpr long long kFx1mS51 = 902847917979075853ll;  // 1 - sin(2 pi / 5)
constexpr long long kFx1mS52 = 7604019954369499282ll; // 1 - sin(4 pi / 5)

// a * f for f * 2^64 = c (|f| < 1/2, |a| < 2^62), rounded to the unit.
FFT3_HD long long fmulc(long long a, long long c) { return rmul62(a, const_hi(c), const_lo(c)); }

// DFT_3 and DFT_5 in the forms of the floating-point butterflies.
template <bool RN>
struct BflyFix<3, RN> {
    static constexpr int scale = 0;
    FFT3_HD static void run(fix2 *v)
    {
        const fix2 s = cadd(v[1], v[2]), d = csub(v[1], v[2]);
        const fix2 a = csub(v[0], half<RN>(s));
        const fix2 b = fix2{d.x - fmulc(d.x, kFx1mS3), d.y - fmulc(d.y, kFx1mS3)};
        v[0] = cadd(v[0], s);
        v[1] = fix2{a.x + b.y, a.y - b.x};
        v[2] = fix2{a.x - b.y, a.y + b.x};
    }
};

template <bool RN>
struct BflyFix<5, RN> {
    static constexpr int scale = 1; // halves its inputs first
    // a1 = x0 + cos(2 pi/5) sa + cos(4 pi/5) sb, a2 the same with sa and sb swapped
    FFT3_HD static long long even(long long x0, long long sa, long long sb)
    {
        return x0 - sb + fmulc(sa, kFxC51) + fmulc(sb, kFx1pC52);
    }
    FFT3_HD static void run(fix2 *v)
    {
        const fix2 x0 = half<RN>(v[0]);
        const fix2 p1 = half<RN>(v[1]), p2 = half<RN>(v[2]), p3 = half<RN>(v[3]), p4 = half<RN>(v[4]);
        const fix2 sa = cadd(p1, p4), da = csub(p1, p4), sb = cadd(p2, p3), db = csub(p2, p3);
        const fix2 a1 = fix2{even(x0.x, sa.x, sb.x), even(x0.y, sa.y, sb.y)};
        const fix2 a2 = fix2{even(x0.x, sb.x, sa.x), even(x0.y, sb.y, sa.y)};
        // b1 = s1 da + s2 db, b2 = s2 da - s1 db
        const fix2 b1 = fix2{da.x + db.x - fmulc(da.x, kFx1mS51) - fmulc(db.x, kFx1mS52),
                             da.y + db.y - fmulc(da.y, kFx1mS51) - fmulc(db.y, kFx1mS52)};
        const fix2 b2 = fix2{da.x - db.x - fmulc(da.x, kFx1mS52) + fmulc(db.x, kFx1mS51),
                             da.y - db.y - fmulc(da.y, kFx1mS52) + fmulc(db.y, kFx1mS51)};
        v[0] = cadd(x0, cadd(sa, sb));
        v[1] = fix2{a1.x + b1.y, a1.y - b1.x};
        v[4] = fix2{a1.x - b1.y, a1.y + b1.x};
        v[2] = fix2{a2.x + b2.y, a2.y - b2.x};
        v[3] = fix2{a2.x - b2.y, a2.y + b2.x};
    }
};

// cos and sin of 2 pi m / N times 2^62 for m <= N/2: the inner twiddles of the
// composite butterflies.
constexpr long long kFxCos9[5] = {
    4611686018427387904ll, 3532756447825785444ll, 800810873071977681ll, -2305843009213693952ll,
    -4333567320897763126ll};
constexpr long long kFxSin9[5] = {
    0ll, 2964334632409774423ll, 4541624145405292212ll, 3993837246235628775ll,
    1577289512995517789ll};
constexpr long long kFxCos10[6] = {
    4611686018427387904ll, 3730932361629093763ll, 1425089352415399811ll, -1425089352415399811ll,
    -3730932361629093763ll, -4611686018427387904ll};
constexpr long long kFxSin10[6] = {
    0ll, 2710681029835013083ll, 4385974038932618941ll, 4385974038932618941ll,
    2710681029835013083ll, 0ll};
constexpr long long kFxCos12[7] = {
    4611686018427387904ll, 3993837246235628775ll, 2305843009213693952ll, 0ll,
    -2305843009213693952ll, -3993837246235628775ll, -4611686018427387904ll};
constexpr long long kFxSin12[7] = {
    0ll, 2305843009213693952ll, 3993837246235628775ll, 4611686018427387904ll,
    3993837246235628775ll, 2305843009213693952ll, 0ll};
constexpr long long kFxCos15[8] = {
    4611686018427387904ll, 4212984814208232069ll, 3085820261846986643ll, 1425089352415399811ll,
    -482052452579138307ll, -2305843009213693952ll, -3730932361629093763ll, -4510909614262386453ll};
constexpr long long kFxSin15[8] = {
    0ll, 1875741690054758654ll, 3427150601320760278ll, 4385974038932618941ll,
    4586422719889771737ll, 3993837246235628775ll, 2710681029835013083ll, 958823437611858663ll};
template <int N>
FFT3_HD constexpr long long fx_cos_n(int m)
{
    const int k = m <= N / 2 ? m : N - m;
    return N == 9 ? kFxCos9[k < 5 ? k : 0] : N == 10 ? kFxCos10[k < 6 ? k : 0] : N == 12 ? kFxCos12[k < 7 ? k : 0]
         : kFxCos15[k < 8 ? k : 0];
}
template <int N>
FFT3_HD constexpr long long fx_sin_n(int m)
{
    const int k = m <= N / 2 ? m : N - m;
    const long long v = N == 9 ? kFxSin9[k < 5 ? k : 0] : N == 10 ? kFxSin10[k < 6 ? k : 0]
                      : N == 12 ? kFxSin12[k < 7 ? k : 0] : kFxSin15[k < 8 ? k : 0];
    return m <= N / 2 ? v : -v;
}

// DFT_{A B} by Eq. ct (DFT_B, inner twiddles w_{AB}^{i0 k1} / 4, DFT_A); NT is
// the table the twiddles come from (AB or a multiple).
template <int A, int B, int NT, int I, bool RN>
struct CtFixTw {
    FFT3_HD static void run(fix2 (*t)[B])
    {
        if constexpr (I < A * B) {
            constexpr int m = (I / B) * (I % B) * (NT / (A * B)) % NT;
            fix2 &v = t[I / B][I % B];
            if constexpr (m == 0) {
                v = quarter<RN>(v);
            } else {
                constexpr long long c = fx_cos_n<NT>(m), s = fx_sin_n<NT>(m);
                v = cmul62(v, root62{const_hi(c), const_lo(c), const_hi(-s), const_lo(-s)});
            }
            CtFixTw<A, B, NT, I + 1, RN>::run(t);
        }
    }
};

template <int A, int B, int NT, bool RN>
struct BflyFixCt {
    static constexpr int scale = BflyFix<B, RN>::scale + 2 + BflyFix<A, RN>::scale;
    FFT3_HD static void run(fix2 *v)
    {
        fix2 t[A][B];
#pragma unroll
        for (int i0 = 0; i0 < A; ++i0) {
#pragma unroll
            for (int i1 = 0; i1 < B; ++i1)
                t[i0][i1] = v[i0 + A * i1];
            BflyFix<B, RN>::run(t[i0]);
        }
        CtFixTw<A, B, NT, 0, RN>::run(t);
#pragma unroll
        for (int k1 = 0; k1 < B; ++k1) {
            fix2 c[A];
#pragma unroll
            for (int i0 = 0; i0 < A; ++i0)
                c[i0] = t[i0][k1];
            BflyFix<A, RN>::run(c);
#pragma unroll
            for (int k0 = 0; k0 < A; ++k0)
                v[k1 + B * k0] = c[k0];
        }
    }
};
template <bool RN>
struct BflyFix<6, RN> : BflyFixCt<2, 3, 12, RN> {};
template <bool RN>
struct BflyFix<9, RN> : BflyFixCt<3, 3, 9, RN> {};
template <bool RN>
struct BflyFix<10, RN> : BflyFixCt<2, 5, 10, RN> {};
template <bool RN>
struct BflyFix<12, RN> : BflyFixCt<4, 3, 12, RN> {};
template <bool RN>
struct BflyFix<15, RN> : BflyFixCt<3, 5, 15, RN> {};

// Normalisation between stages: `acc` is the OR of norm_word over the
// components of a line; the line is shifted up by norm_shift(acc), which keeps
// components below 2^61 (a line within one bit of that stays as it is).
FFT3_HD unsigned norm_word(long long v)
{
    const int h = (int)(v >> 32);
    return (unsigned)(h ^ (h >> 31));
}
FFT3_HD int clz32(unsigned v)
{
#ifdef __CUDA_ARCH__
    return __clz((int)v);
#else
    return v ? __builtin_clz(v) : 32;
#endif
}
FFT3_HD int norm_shift(unsigned acc)
{
    const int l = clz32(acc) - 3;
    return l > 1 ? l : 0;
}

// ------------------------------------------------------- conversions ---- //
// Exponent field range of a line's largest component that the integer stages
// take; zero lines (field 0, all bits zero) are taken too.
constexpr int kFixMinExp = 128, kFixMaxExp = 2030;

// Magnitude word of one component for the line maximum: its high word without
// the sign, or 1 for a subnormal whose high word is zero.
FFT3_HD unsigned mag_word(double v)
{
    unsigned long long b;
    memcpy(&b, &v, 8);
    const unsigned h = (unsigned)(b >> 32) & 0x7fffffffu;
    return h ? h : ((unsigned)b != 0u ? 1u : 0u);
}
// Largest magnitude words of the real and of the imaginary parts of some values.
struct FixMag {
    unsigned re, im;
};
FFT3_HD void mag_max(FixMag &m, double2 v)
{
    const unsigned a = mag_word(v.x), b = mag_word(v.y);
    m.re = a > m.re ? a : m.re;
    m.im = b > m.im ? b : m.im;
}
FFT3_HD unsigned mag_all(FixMag m) { return m.re > m.im ? m.re : m.im; }

// What decides over a line, gathered over its first-stage butterflies.
struct FixScan {
    FixMag line{0u, 0u}; // the line's largest
    unsigned least = ~0u; // the least of the butterflies' largest, those of zeros left out
    bool zeros = false;  // whether there is a butterfly of zeros
    FFT3_HD void add(FixMag m)
    {
        line.re = m.re > line.re ? m.re : line.re;
        line.im = m.im > line.im ? m.im : line.im;
        const unsigned all = mag_all(m);
        zeros = zeros || all == 0u;
        least = all != 0u && all < least ? all : least;
    }
};

// How far (2^-bits) below the largest component another may lie without a stage of
// radix scale `scale` shifting a bit of it out: a first stage has six bits to spare
// and loses the butterfly's scale, a later one has eight (from the shift up) and
// loses two more.
FFT3_HD constexpr int fix_exact_bits(int scale) { return 6 - scale; }

// Whether a list whose first stage has this scale rounds its shifts down.
FFT3_HD constexpr bool fix_rounds(int scale) { return scale > 2; }

// Whether a list of n points that starts with radix R takes only lines with a large
// value in every first-stage butterfly.
FFT3_HD constexpr bool fix_strict(int n, int R) { return R == 32 || (R == 5 && n > 2048); }

// Whether a line takes the integer stages; exact: the least fix_exact_bits of its
// stages.  Holds for a line when it holds for every part of its butterflies (least,
// zeros) with the whole line's `line`.
FFT3_HD bool fix_ok(const FixScan &s, bool strict, int exact)
{
    const unsigned m = mag_all(s.line), e = m >> 20;
    if (m == 0u)
        return true;
    if (e < (unsigned)kFixMinExp || e > (unsigned)kFixMaxExp || (strict && s.least < m - (4u << 20)))
        return false;
    const unsigned low = m - ((s.zeros && exact < 5 ? (unsigned)exact : 5u) << 20);
    return (s.line.re == 0u || s.line.re >= low) && (s.line.im == 0u || s.line.im >= low);
}

// Exponent field the line's values are scaled by (any of the range for a zero
// line: a zero's mantissa is then shifted out).
FFT3_HD int fix_emax(unsigned m) { return m ? (int)(m >> 20) : 1023; }

// v in units of 2^(emax - 1023 - 58), rounded (RN) or truncated: components below 2^59, moduli below 2^60
// (emax: exponent field of the line's largest component).
template <bool RN>
FFT3_HD long long to_fix(double v, int emax)
{
    unsigned long long b;
    memcpy(&b, &v, 8);
    const unsigned hi = (unsigned)(b >> 32);
    const int e = (int)((hi >> 20) & 0x7ffu);
    unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | (unsigned)b;
    const int d = emax - e;
    m <<= 6;
    if (RN)
        m += (1ull << (d < 62 ? d : 62)) >> 1;
    m >>= d < 63 ? d : 63;
    return (int)hi < 0 ? -(long long)m : (long long)m;
}

// V * 2^sh, rounded once (to the nearest): sh shifts the exponent field of
// (double)V.  from_fix_int is the same conversion on the integer pipe: the
// hardware's runs at 2 lanes per clock and SM on the FP64 pipe.
FFT3_HD double from_fix(long long v, int sh)
{
    const double d = (double)v;
    unsigned long long b;
    memcpy(&b, &d, 8);
    b += (unsigned long long)(long long)sh << 52;
    double r;
    memcpy(&r, &b, 8);
    return v ? r : 0.0;
}
FFT3_HD double from_fix_int(long long v, int sh)
{
    const unsigned sign = (unsigned)((unsigned long long)v >> 32) & 0x80000000u;
    unsigned long long u = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const unsigned h = (unsigned)(u >> 32);
    const int z = h ? clz32(h) : 32 + clz32((unsigned)u);
    // leading bit to bit 62, rounded to 53 bits (ties to even) and to bit 52,
    // where it adds one to the exponent field (a carry past it one more)
    u <<= z - 1;
    u += 0x1ffu + ((unsigned)(u >> 10) & 1u);
    u >>= 10;
    const unsigned hi = (unsigned)(u >> 32) + ((unsigned)(1023 + 62 - z + sh) << 20);
    const unsigned long long b = ((unsigned long long)(hi | sign) << 32) | (unsigned)u;
    double r;
    memcpy(&r, &b, 8);
    return v ? r : 0.0;
}

// ---------------------------------------------------------- roots ------- //
// sin and cos of theta / 2^64 (theta < pi/4 * 2^64) as Q62, by their Taylor
// series in 64-bit fixed point.
FFT3_HD unsigned long long mulhi64(unsigned long long a, unsigned long long b)
{
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (unsigned long long)(((unsigned __int128)a * b) >> 64);
#endif
}
FFT3_HD void sincos_q64(unsigned long long th, long long *s, long long *c)
{
    const unsigned long long t2 = mulhi64(th, th);
    // terms theta^k / k! for k = 2, 3, ...; cos = 1 - T2 + T4 - ..., sin = T1 - T3 + ...
    unsigned long long tc = t2 >> 1, ts = mulhi64(th, t2) / 6;
    long long cs = 0;                        // cos - 1, Q64 (|cos - 1| < 0.3)
    long long ss = (long long)(th >> 1);     // sin, Q63
    cs -= (long long)tc;
    ss -= (long long)(ts >> 1);
    for (int k = 2; k < 12; ++k) {
        tc = mulhi64(tc, t2) / (unsigned)((2 * k) * (2 * k - 1));
        ts = mulhi64(ts, t2) / (unsigned)((2 * k + 1) * (2 * k));
        if (k & 1) {
            cs -= (long long)tc;
            ss -= (long long)(ts >> 1);
        } else {
            cs += (long long)tc;
            ss += (long long)(ts >> 1);
        }
    }
    *c = (1ll << 62) + ((cs + 2) >> 2);
    *s = (ss + 1) >> 1;
}

// w_n^m = exp(-2 pi i m / n) times 2^62, m reduced mod n and to an octant in
// integers: 8m = o n + rem, theta = 2 pi rem / (8n) or its complement to pi/4.
FFT3_HD root62 root_fix(int64_t m, int n)
{
    int64_t mm = m % n;
    if (mm < 0)
        mm += n;
    const int64_t o = 8 * mm / n;
    int64_t rem = 8 * mm - o * n; // in [0, n)
    if (o & 1)
        rem = n - rem;            // odd octants run backwards, in (0, n]
    long long s, c;
    if (rem == n) {
        constexpr long long h = fx_cos32(4); // sqrt(1/2)
        s = c = h;
    } else {
        // rem / n as Q64 times pi / 4 as Q64
        const unsigned long long q = (((unsigned long long)rem << 32) / (unsigned)n) << 32;
        const unsigned long long r2 = ((unsigned long long)rem << 32) % (unsigned)n;
        const unsigned long long frac = q | ((r2 << 32) / (unsigned)n);
        sincos_q64(mulhi64(frac, 0xc90fdaa22168c235ull), &s, &c);
    }
    long long re, im; // exp(+i angle)
    switch (o & 7) {
    case 0: re = c; im = s; break;
    case 1: re = s; im = c; break;
    case 2: re = -s; im = c; break;
    case 3: re = -c; im = s; break;
    case 4: re = -c; im = -s; break;
    case 5: re = -s; im = -c; break;
    case 6: re = s; im = -c; break;
    default: re = c; im = -s; break;
    }
    im = -im;
    root62 w;
    if ((unsigned)re == 0x80000000u)
        --re;
    if ((unsigned)im == 0x80000000u)
        --im;
    w.rh = bal_hi(re);
    w.rl = bal_lo(re);
    w.ih = bal_hi(im);
    w.il = bal_lo(im);
    return w;
}

} // namespace fft3
