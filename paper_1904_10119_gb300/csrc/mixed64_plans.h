// mixed64_plans.h -- complex128 plans of the 2*3*5-smooth lengths up to 512 that
// are not powers of two.
//
// Row: line length N, threads per line T, contiguous lines per tile, shared layout
// of a contiguous line (position p at p + (p >> SH), SH = 0: p; lines PITCH values
// apart), radix list (first stage first).  Strided columns use T and the radices,
// 8 columns per tile.  The rows come from one rule: the list of the radices 2, 3,
// 4, 5, 6, 8, 9, 10, 12, 15 and 16 and the T up to 64 with the fewest integer
// instructions per value at no more than 16 values a thread (128 registers), then
// the stage order, SH and PITCH with the fewest bank conflicts of 16-byte
// accesses.  The runtime lists (16, 8, 4, 2, 5, 3) of the other lengths take a
// third of the rate: 240^3 in 1810 us against 656.  The list ends at 512 points;
// longer mixed lengths (540 to 1000 points) keep the runtime lists, no compiled plan
// of theirs was measured.
#pragma once

#define FFT3_MIXED64_A(X)                                            \
    X(3, 1, 128, 0, 0, 3) X(15, 1, 128, 0, 0, 15)                    \
    X(30, 2, 64, 0, 30, 15, 2) X(54, 6, 21, 0, 54, 9, 6)             \
    X(90, 10, 12, 0, 90, 9, 10) X(135, 9, 14, 0, 137, 15, 3, 3)      \
    X(192, 16, 8, 4, 203, 16, 12) X(250, 25, 5, 0, 257, 10, 5, 5)    \
    X(360, 24, 5, 3, 404, 8, 3, 15) X(450, 30, 4, 0, 454, 15, 2, 15)

#define FFT3_MIXED64_B(X)                                           \
    X(5, 1, 128, 0, 0, 5) X(18, 3, 42, 0, 19, 6, 3)                 \
    X(36, 3, 42, 2, 45, 12, 3) X(60, 4, 32, 0, 60, 15, 4)           \
    X(96, 8, 16, 3, 107, 8, 12) X(144, 12, 10, 2, 180, 12, 12)      \
    X(200, 14, 9, 0, 206, 5, 5, 8) X(270, 30, 4, 0, 270, 9, 10, 3)  \
    X(375, 25, 5, 0, 377, 15, 5, 5) X(480, 32, 4, 3, 539, 8, 4, 15)

#define FFT3_MIXED64_C(X)                                           \
    X(6, 1, 128, 0, 0, 6) X(20, 2, 64, 3, 22, 10, 2)                \
    X(40, 4, 32, 3, 44, 10, 4) X(72, 6, 21, 2, 90, 12, 6)           \
    X(100, 10, 12, 5, 106, 10, 10) X(150, 15, 8, 0, 151, 15, 10)    \
    X(216, 18, 7, 0, 218, 6, 3, 12) X(288, 24, 5, 4, 305, 12, 6, 4) \
    X(384, 32, 4, 3, 431, 8, 4, 12) X(486, 54, 2, 0, 486, 9, 9, 6)

#define FFT3_MIXED64_D(X)                                             \
    X(9, 1, 128, 0, 0, 9) X(24, 2, 64, 2, 30, 4, 6)                   \
    X(45, 3, 42, 3, 51, 15, 3) X(75, 5, 25, 0, 75, 15, 5)             \
    X(108, 12, 10, 0, 108, 9, 12) X(160, 16, 8, 4, 169, 16, 10)       \
    X(225, 15, 8, 0, 225, 15, 15) X(300, 20, 6, 0, 300, 15, 4, 5)     \
    X(400, 40, 3, 0, 400, 10, 4, 10) X(500, 50, 2, 0, 506, 10, 5, 10)

#define FFT3_MIXED64_E(X)                                         \
    X(10, 1, 128, 0, 0, 10) X(25, 2, 64, 0, 26, 5, 5)             \
    X(48, 4, 32, 2, 60, 12, 4) X(80, 10, 12, 3, 90, 8, 10)        \
    X(120, 8, 16, 0, 120, 15, 8) X(162, 18, 7, 0, 162, 9, 9, 2)   \
    X(240, 16, 8, 4, 254, 16, 15) X(320, 40, 3, 3, 359, 8, 4, 10) \
    X(405, 45, 2, 0, 405, 9, 9, 5)

#define FFT3_MIXED64_F(X)                                         \
    X(12, 1, 128, 0, 0, 12) X(27, 3, 42, 0, 27, 9, 3)             \
    X(50, 5, 25, 0, 53, 10, 5) X(81, 9, 14, 0, 81, 9, 9)          \
    X(125, 13, 9, 0, 125, 5, 5, 5) X(180, 15, 8, 0, 180, 15, 12)  \
    X(243, 27, 4, 0, 243, 9, 9, 3) X(324, 41, 3, 0, 329, 9, 9, 4) \
    X(432, 36, 3, 5, 445, 12, 12, 3)

#define FFT3_MIXED64(X) \
    FFT3_MIXED64_A(X) FFT3_MIXED64_B(X) FFT3_MIXED64_C(X) FFT3_MIXED64_D(X) FFT3_MIXED64_E(X) FFT3_MIXED64_F(X)

namespace fft3 {

struct Mixed64Meta {
    int n, T, lpt;
    int pitch; // contiguous lines: values of shared memory per line
    int rad[8];
};
struct Mixed64Kernels {
    int n;
    const void *j, *c; // contiguous lines; strided columns
};
const Mixed64Kernels *mixed64_kernels(int n); // nullptr if none is compiled

} // namespace fft3
