// mixed_plans.h -- compile-time line plans of the 2*3*5-smooth lengths up to
// 1024 that are not powers of two (those have their own list, plans.h).
//
// Contiguous lines (J): length N, threads per line T, lines per tile, blocks
// per SM the launch bounds ask for, layout of a line in shared memory (position
// p at p + (p >> SH), SH = 0: p; lines PITCH values apart), radix list (first
// stage first).  Strided columns (C): N, T, columns per tile, blocks per SM,
// radix list.
//
// Every row was picked by measurement among candidates made by one rule: lists
// of the radices 2, 3, 4, 5, 6, 8, 9, 10, 12, 15 and 16 with product N in every
// order that starts with a large one, T that leaves few of the N / R butterflies
// of a stage without a thread (at most 30 values per thread), blocks of 512,
// 768 or 1024 threads per SM as far as 32 resident blocks allow (one thread a
// column makes blocks of 16: half a warp each, 512 threads per SM), the six best
// by instructions per value and bank conflicts; SH and PITCH are those with the fewest conflicts over all stages,
// counted from the addresses of each warp.  The padding of the power-of-two
// plans (SH = 4) costs odd radices 3 to 5 times the accesses: 375 points ran
// at 2.8 TB/s with it, at 4.9 without.  Rates of the rows below on 268 MB (one
// read and one write per value), contiguous / strided, TB/s: 4.4-6.1 / 5.1-6.4 at
// 18-100 points, 4.6-6.2 / 5.4-6.2 at 108-240, 4.5-5.5 / 4.4-5.8 at 243-500, 3.9-5.5 / 3.7-5.2 at
// 540-1000.
// The lists are split over four translation units that compile in parallel.
#pragma once

#define FFT3_MIXED_J_A(X)                                                   \
    X(3, 1, 256, 4, 0, 0, 3) X(10, 1, 256, 4, 0, 0, 10)                     \
    X(20, 4, 64, 4, 2, 28, 4, 5) X(30, 6, 42, 4, 2, 37, 6, 5)               \
    X(48, 8, 32, 3, 3, 56, 8, 6) X(72, 9, 28, 5, 0, 72, 9, 8)               \
    X(90, 10, 25, 5, 0, 90, 9, 10) X(120, 8, 32, 4, 3, 136, 8, 15)          \
    X(150, 15, 17, 5, 0, 150, 15, 10) X(192, 16, 16, 2, 4, 203, 16, 12)     \
    X(240, 18, 14, 3, 4, 256, 16, 15) X(288, 24, 10, 4, 5, 296, 12, 12, 2)  \
    X(360, 24, 10, 3, 0, 360, 15, 8, 3) X(405, 45, 5, 5, 0, 413, 5, 9, 9)   \
    X(486, 27, 9, 4, 0, 491, 6, 9, 9) X(600, 40, 6, 3, 0, 600, 15, 8, 5)    \
    X(675, 45, 5, 4, 0, 685, 15, 15, 3) X(768, 64, 4, 4, 4, 815, 16, 12, 4) \
    X(900, 60, 4, 4, 0, 908, 15, 4, 15)

#define FFT3_MIXED_C_A(X)                                                               \
    X(3, 1, 16, 32, 3) X(10, 1, 16, 32, 10) X(20, 2, 16, 24, 10, 2)                     \
    X(30, 2, 16, 24, 15, 2) X(48, 4, 16, 12, 12, 4) X(72, 6, 16, 8, 12, 6)              \
    X(90, 10, 16, 7, 10, 9) X(120, 12, 16, 6, 12, 10) X(150, 15, 16, 5, 15, 10)         \
    X(192, 16, 16, 4, 16, 12) X(240, 18, 16, 4, 16, 15) X(288, 24, 16, 3, 12, 6, 4)     \
    X(360, 12, 16, 4, 10, 6, 6) X(405, 45, 16, 2, 9, 9, 5) X(486, 27, 16, 2, 9, 9, 6)   \
    X(600, 20, 16, 2, 10, 10, 6) X(675, 45, 8, 2, 15, 15, 3) X(768, 48, 8, 2, 16, 8, 6) \
    X(900, 60, 8, 2, 15, 15, 4)

#define FFT3_MIXED_J_B(X)                                                     \
    X(5, 1, 256, 4, 0, 0, 5) X(12, 1, 256, 2, 0, 0, 12)                       \
    X(24, 4, 64, 4, 2, 44, 4, 6) X(36, 6, 42, 5, 2, 45, 6, 6)                 \
    X(50, 5, 51, 3, 0, 53, 10, 5) X(75, 8, 32, 4, 0, 87, 15, 5)               \
    X(96, 8, 32, 4, 4, 104, 16, 6) X(125, 13, 19, 4, 0, 125, 5, 5, 5)         \
    X(160, 16, 16, 4, 4, 169, 16, 10) X(200, 20, 12, 5, 0, 212, 10, 10, 2)    \
    X(243, 27, 9, 5, 0, 251, 9, 3, 9) X(300, 20, 12, 3, 0, 308, 15, 4, 5)     \
    X(375, 25, 10, 4, 0, 377, 15, 5, 5) X(432, 36, 7, 5, 0, 436, 6, 12, 6)    \
    X(500, 52, 4, 5, 0, 500, 10, 5, 10) X(625, 25, 10, 3, 0, 633, 5, 5, 5, 5) \
    X(720, 48, 5, 3, 4, 764, 16, 15, 3) X(800, 40, 6, 3, 0, 808, 10, 5, 4, 4) \
    X(960, 64, 4, 3, 4, 1019, 16, 15, 4)

#define FFT3_MIXED_C_B(X)                                                                   \
    X(5, 1, 16, 32, 5) X(12, 1, 16, 32, 12) X(24, 2, 16, 24, 12, 2)                         \
    X(36, 3, 16, 16, 12, 3) X(50, 5, 16, 13, 10, 5) X(75, 5, 16, 10, 15, 5)                 \
    X(96, 4, 16, 12, 12, 8) X(125, 5, 16, 7, 5, 5, 5) X(160, 16, 16, 4, 16, 10)             \
    X(200, 10, 16, 5, 10, 5, 4) X(243, 9, 16, 4, 9, 9, 3) X(300, 10, 16, 4, 10, 6, 5)       \
    X(375, 25, 8, 4, 15, 5, 5) X(432, 18, 16, 3, 12, 12, 3) X(500, 25, 16, 2, 10, 10, 5)    \
    X(625, 25, 16, 2, 5, 5, 5, 5) X(720, 48, 8, 2, 16, 15, 3) X(800, 40, 8, 2, 10, 5, 4, 4) \
    X(960, 64, 8, 2, 16, 15, 4)

#define FFT3_MIXED_J_C(X)                                                  \
    X(6, 1, 256, 2, 0, 0, 6) X(15, 1, 256, 3, 0, 0, 15)                    \
    X(25, 3, 85, 5, 0, 35, 5, 5) X(40, 5, 51, 5, 0, 41, 5, 8)              \
    X(54, 9, 28, 5, 0, 54, 9, 6) X(80, 10, 25, 5, 3, 90, 8, 10)            \
    X(100, 10, 25, 3, 5, 106, 10, 10) X(135, 9, 28, 3, 0, 135, 15, 9)      \
    X(162, 18, 14, 5, 0, 162, 9, 6, 3) X(216, 36, 7, 3, 0, 217, 6, 6, 6)   \
    X(250, 25, 10, 5, 0, 265, 5, 5, 10) X(320, 40, 6, 5, 0, 328, 10, 8, 4) \
    X(384, 16, 16, 3, 4, 407, 8, 6, 8) X(450, 50, 5, 4, 0, 450, 9, 10, 5)  \
    X(540, 45, 8, 3, 0, 541, 15, 12, 3) X(640, 40, 6, 4, 0, 648, 10, 8, 8) \
    X(729, 27, 9, 3, 0, 731, 9, 9, 9) X(810, 45, 5, 3, 0, 813, 10, 9, 9)   \
    X(972, 54, 4, 4, 0, 982, 9, 12, 9)

#define FFT3_MIXED_C_C(X)                                                               \
    X(6, 1, 16, 32, 6) X(15, 1, 16, 32, 15) X(25, 1, 16, 32, 5, 5)                      \
    X(40, 2, 16, 16, 10, 4) X(54, 6, 16, 11, 9, 6) X(80, 10, 16, 7, 10, 8)              \
    X(100, 10, 16, 7, 10, 10) X(135, 9, 16, 6, 15, 3, 3) X(162, 9, 16, 6, 9, 6, 3)      \
    X(216, 18, 16, 4, 6, 6, 6) X(250, 25, 16, 3, 10, 5, 5) X(320, 40, 8, 4, 10, 8, 4)   \
    X(384, 16, 16, 3, 12, 8, 4) X(450, 30, 16, 2, 15, 15, 2) X(540, 45, 8, 3, 15, 6, 6) \
    X(640, 40, 8, 2, 16, 8, 5) X(729, 27, 16, 2, 9, 9, 9) X(810, 45, 16, 1, 10, 9, 9)   \
    X(972, 54, 8, 2, 9, 9, 6, 2)

#define FFT3_MIXED_J_D(X)                                                   \
    X(9, 1, 256, 2, 0, 0, 9) X(18, 3, 85, 4, 4, 25, 3, 6)                   \
    X(27, 3, 85, 4, 0, 27, 9, 3) X(45, 5, 51, 5, 0, 57, 5, 9)               \
    X(60, 6, 42, 4, 2, 74, 12, 5) X(81, 9, 28, 3, 0, 81, 9, 9)              \
    X(108, 12, 21, 5, 0, 108, 9, 12) X(144, 12, 21, 4, 2, 180, 12, 12)      \
    X(180, 15, 17, 3, 0, 180, 15, 12) X(225, 17, 15, 3, 0, 225, 15, 15)     \
    X(270, 30, 8, 4, 0, 270, 9, 10, 3) X(324, 36, 7, 4, 0, 324, 9, 12, 3)   \
    X(400, 20, 12, 3, 0, 404, 10, 10, 4) X(480, 32, 8, 3, 0, 480, 15, 8, 4) \
    X(576, 36, 7, 4, 0, 580, 9, 8, 8) X(648, 36, 7, 3, 0, 660, 9, 12, 6)    \
    X(750, 50, 5, 3, 0, 754, 15, 10, 5) X(864, 36, 7, 3, 0, 868, 9, 8, 12)  \
    X(1000, 50, 5, 3, 0, 1001, 10, 10, 10)

#define FFT3_MIXED_C_D(X)                                                                 \
    X(9, 1, 16, 32, 9) X(18, 2, 16, 24, 9, 2) X(27, 3, 16, 22, 9, 3)                      \
    X(45, 3, 16, 16, 15, 3) X(60, 6, 16, 11, 12, 5) X(81, 9, 16, 8, 9, 9)                 \
    X(108, 12, 16, 6, 12, 9) X(144, 14, 16, 5, 12, 12) X(180, 15, 16, 5, 15, 12)          \
    X(225, 17, 16, 4, 15, 15) X(270, 30, 16, 3, 10, 9, 3) X(324, 18, 16, 3, 9, 6, 6)      \
    X(400, 20, 16, 3, 10, 10, 4) X(480, 32, 16, 2, 16, 15, 2) X(576, 24, 16, 2, 12, 8, 6) \
    X(648, 36, 8, 2, 9, 9, 8) X(750, 25, 8, 3, 15, 10, 5) X(864, 36, 8, 2, 12, 12, 6)     \
    X(1000, 50, 8, 2, 10, 10, 10)

#define FFT3_MIXED_J(X) FFT3_MIXED_J_A(X) FFT3_MIXED_J_B(X) FFT3_MIXED_J_C(X) FFT3_MIXED_J_D(X)
#define FFT3_MIXED_C(X) FFT3_MIXED_C_A(X) FFT3_MIXED_C_B(X) FFT3_MIXED_C_C(X) FFT3_MIXED_C_D(X)

namespace fft3 {

struct MixedPlanMeta {
    int n, T, lpt;
    int pitch; // contiguous lines: values of shared memory per line
    int rad[8];
};

struct MixedKernels {
    int n;
    const void *func;
};
// The pass compiled for lines of n points (contiguous or strided columns), nullptr if none is.
const void *mixed_kernel(int n, bool contiguous);

} // namespace fft3
