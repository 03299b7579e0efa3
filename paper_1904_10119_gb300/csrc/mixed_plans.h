// mixed_plans.h -- compile-time line plans of the 2*3*5-smooth lengths up to
// 1024 that are not powers of two (those have their own list, plans.h).
//
// Each row: line length N, threads per line T, radix list (first stage first).
// The rows come from one rule, a search over every list of the radices 2, 3, 4,
// 5, 6, 8, 9, 10, 12, 15 and 16 with product N and every T up to 64: least
// instructions per value, counted as the butterfly's arithmetic, one shared
// memory exchange per stage and the twiddles of the later stages, times the
// share of butterfly slots that a stage with N/R butterflies leaves idle on T
// threads, with at most 16 values per thread and stage (up to 24 where that
// saves more than 7%).  It gives two stages up to 240 points and three up to
// 1024 for nearly every length, where the runtime-radix kernel, whose lists
// hold only 16, 8, 4, 2, 5 and 3, runs up to six.
// The list is split over four translation units that compile in parallel.
#pragma once

#define FFT3_MIXED_PLANS_A(X)                                       \
    X(3, 1, 3) X(10, 1, 10) X(20, 2, 10, 2)                         \
    X(30, 2, 15, 2) X(48, 4, 12, 4) X(72, 6, 12, 6)                 \
    X(90, 10, 10, 9) X(120, 8, 15, 8) X(150, 15, 15, 10)            \
    X(192, 16, 16, 12) X(240, 16, 16, 15) X(288, 24, 12, 12, 2)     \
    X(360, 24, 15, 8, 3) X(405, 45, 9, 9, 5) X(486, 27, 9, 9, 6)    \
    X(600, 40, 15, 8, 5) X(675, 45, 15, 15, 3) X(768, 32, 12, 8, 8) \
    X(900, 60, 15, 15, 4)

#define FFT3_MIXED_PLANS_B(X)                                          \
    X(5, 1, 5) X(12, 1, 12) X(24, 2, 12, 2)                            \
    X(36, 3, 12, 3) X(50, 5, 10, 5) X(75, 5, 15, 5)                    \
    X(96, 4, 12, 8) X(125, 13, 5, 5, 5) X(160, 10, 16, 10)             \
    X(200, 20, 10, 10, 2) X(243, 27, 9, 9, 3) X(300, 20, 15, 5, 4)     \
    X(375, 25, 15, 5, 5) X(432, 36, 12, 12, 3) X(500, 50, 10, 10, 5)   \
    X(625, 42, 5, 5, 5, 5) X(720, 48, 16, 15, 3) X(800, 40, 10, 10, 8) \
    X(960, 64, 15, 8, 8)

#define FFT3_MIXED_PLANS_C(X)                                       \
    X(6, 1, 6) X(15, 1, 15) X(25, 2, 5, 5)                          \
    X(40, 2, 10, 4) X(54, 3, 9, 6) X(80, 10, 10, 8)                 \
    X(100, 10, 10, 10) X(135, 9, 15, 9) X(162, 18, 9, 9, 2)         \
    X(216, 18, 12, 6, 3) X(250, 25, 10, 5, 5) X(320, 22, 8, 8, 5)   \
    X(384, 16, 12, 8, 4) X(450, 30, 15, 15, 2) X(540, 30, 10, 9, 6) \
    X(640, 43, 16, 8, 5) X(729, 41, 9, 9, 9) X(810, 45, 10, 9, 9)   \
    X(972, 54, 12, 9, 9)

#define FFT3_MIXED_PLANS_D(X)                                             \
    X(9, 1, 9) X(18, 3, 6, 3) X(27, 3, 9, 3)                              \
    X(45, 3, 15, 3) X(60, 4, 15, 4) X(81, 9, 9, 9)                        \
    X(108, 12, 12, 9) X(144, 12, 12, 12) X(180, 15, 15, 12)               \
    X(225, 15, 15, 15) X(270, 30, 10, 9, 3) X(324, 18, 9, 6, 6)           \
    X(400, 27, 16, 5, 5) X(480, 32, 15, 8, 4) X(576, 48, 12, 12, 4)       \
    X(648, 54, 12, 6, 3, 3) X(750, 50, 15, 5, 5, 2) X(864, 36, 12, 12, 6) \
    X(1000, 50, 10, 10, 10)

#define FFT3_MIXED_PLANS(X) \
    FFT3_MIXED_PLANS_A(X) FFT3_MIXED_PLANS_B(X) FFT3_MIXED_PLANS_C(X) FFT3_MIXED_PLANS_D(X)

namespace fft3 {

struct MixedPlanMeta {
    int n, T;
    int rad[8];
};

// Passes compiled for one mixed plan: contiguous lines (256 / T lines per
// tile), strided columns (mixed_lpt_c columns per tile).
struct MixedKernels {
    int n;
    const void *j;
    const void *c;
};
const MixedKernels *mixed_kernels(int n); // nullptr: no plan of that length

// Columns per strided tile: 16 (128-byte rows) while two tiles fit an SM's
// shared memory and a tile's block has at most 512 threads, else 8.
constexpr int mixed_lpt_c(int n, int T) { return n <= 640 && T * 16 <= 512 ? 16 : 8; }

} // namespace fft3
