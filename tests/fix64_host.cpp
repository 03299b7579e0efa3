// Host model of the complex128 line passes: reads lists "c n R R ..." (a line length
// and its radix list, first stage first) and prints, per kind of line, the relative
// 2-norm error (rms over the lines) of the integer stages where fix_ok takes the
// line and of the FP64 stages on the same lines, both against long double, and how
// many lines were taken.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>

#include <algorithm>
#include <complex>
#include <iostream>
#include <random>
#include <sstream>
#include <string>
#include <type_traits>
#include <vector>

static inline void __syncthreads() {}
#include "fft_engine.cuh"
#include "fix64.cuh"

using namespace fft3;
typedef std::complex<double> Cd;
typedef std::complex<long double> Cl;

static Cl root(int64_t m, int n)
{
    m = 8 * (m % n);
    int o = (int)(m / n);
    int64_t rem = m - (int64_t)o * n;
    if (o & 1)
        rem = n - rem;
    const long double a = acosl(-1.0L) / 4 * rem / n, c = cosl(a), s = sinl(a);
    const long double re[8] = {c, s, -s, -c, -c, -s, s, c}, im[8] = {s, c, c, s, -s, -c, -c, -s};
    return Cl(re[o], -im[o]);
}

template <class F>
static void with_radix(int R, const F &f)
{
    switch (R) {
#define CASE(r) case r: f(std::integral_constant<int, r>()); break;
    CASE(2) CASE(3) CASE(4) CASE(5) CASE(6) CASE(8) CASE(9) CASE(10) CASE(12) CASE(15) CASE(16) CASE(32)
    default: fprintf(stderr, "radix %d\n", R); exit(1);
    }
}

// DFT of the line by its own list in long double (direct sums per butterfly).
static std::vector<Cl> exact(const std::vector<Cd> &x, const std::vector<int> &rad, const std::vector<Cl> &w)
{
    const int n = (int)x.size();
    std::vector<Cl> a(n), b(n);
    for (int i = 0; i < n; ++i)
        a[i] = Cl(x[i].real(), x[i].imag());
    int NS = 1;
    for (int R : rad) {
        for (int q = 0; q < n / R; ++q)
            for (int r = 0; r < R; ++r) {
                Cl s = 0;
                for (int i = 0; i < R; ++i)
                    s += a[q + i * (n / R)] * w[((int64_t)i * (q % NS) * (n / (NS * R)) + (int64_t)i * r % R * (n / R)) % n];
                b[(q / NS) * NS * R + q % NS + r * NS] = s;
            }
        std::swap(a, b);
        NS *= R;
    }
    return a;
}

template <class C, class Stage>
static void stages(std::vector<C> &a, const std::vector<int> &rad, const Stage &stage)
{
    const int n = (int)a.size();
    std::vector<C> b(n);
    int NS = 1;
    for (size_t s = 0; s < rad.size(); ++s) {
        with_radix(rad[s], [&](auto rc) {
            constexpr int R = decltype(rc)::value;
            for (int q = 0; q < n / R; ++q) {
                C v[R];
                const int k = q % NS;
                for (int r = 0; r < R; ++r)
                    v[r] = a[q + r * (n / R)];
                stage(rc, s, v, [&](int r) { return (int64_t)r * k * (n / (NS * R)) % n; });
                for (int r = 0; r < R; ++r)
                    b[(q / NS) * NS * R + k + r * NS] = v[r];
            }
        });
        std::swap(a, b);
        NS *= rad[s];
    }
}

// Kinds: d... a constant, s... a spike, i... a real line, over a background of 10^-number (spike-999: of zeros).
static std::vector<Cd> line(const std::string &kind, int n, std::mt19937_64 &g)
{
    auto u = [&] { return 2.0 * (double)(g() >> 11) * 0x1p-53 - 1.0; };
    auto c = [&] { const double a = u(); return Cd(a, u()); };
    std::vector<Cd> x(n);
    const double bg = kind.find('-') == std::string::npos ? 0.0 : pow(10.0, -atof(kind.c_str() + kind.find('-') + 1));
    for (int i = 0; i < n; ++i) {
        const int f = std::min(i, n - i);
        x[i] = kind == "uniform" ? c()
             : kind == "real" ? Cd(u(), 0)
             : kind == "decades" ? std::polar(pow(10.0, 12 * u()), 3.14 * u())
             : kind == "spectrum" ? c() / ((1.0 + f) * (1.0 + f))
             : kind == "bump" ? Cd(exp(-0.5 * pow((i - 0.4 * n) / (0.05 * n), 2)), 0)
             : kind[0] == 'd' ? Cd(1.01, 0.7) + bg * c() // dc-...
             : kind[0] == 'i' ? Cd(u(), bg * u())        // im-...
                              : bg * c();                 // spike-...
    }
    if (kind.rfind("spike", 0) == 0)
        x[g() % n] = Cd(1.01, 0.3);
    return x;
}

int main()
{
    const char *kinds[] = {"uniform", "real", "decades", "spectrum", "bump", "dc-1", "dc-3", "dc-12",
                           "im-1", "im-12", "spike-1", "spike-1.4", "spike-999", "spike-3", "spike-12"};
    std::string row;
    while (std::getline(std::cin, row)) {
        std::istringstream is(row);
        int n, R;
        std::vector<int> rad;
        std::string kernel;
        is >> kernel >> n;
        const bool runtime = kernel == "g";
        while (is >> R)
            rad.push_back(R);
        std::vector<Cl> w(n);
        for (int m = 0; m < n; ++m)
            w[m] = root(m, n);
        int exact_bits = 6;
        bool rounds = runtime;
        with_radix(rad[0], [&](auto rc) { rounds = rounds || fix_rounds(BflyFix<decltype(rc)::value, false>::scale); });
        for (int r : rad)
            with_radix(r, [&](auto rc) { exact_bits = std::min(exact_bits, fix_exact_bits(BflyFix<decltype(rc)::value, false>::scale)); });
        for (const char *kind : kinds) {
            std::mt19937_64 g(n);
            double efix = 0, e64 = 0;
            int taken = 0;
            const int lines = 16;
            for (int i = 0; i < lines; ++i) {
                const std::vector<Cd> x = line(kind, n, g);
                FixScan scan;
                scan.zeros = rad.size() == 1;
                const FixMag &lm = scan.line;
                for (int q = 0; q < n / rad[0]; ++q) {
                    FixMag m{0u, 0u};
                    for (int r = 0; r < rad[0]; ++r) {
                        const Cd v = x[q + r * (n / rad[0])];
                        mag_max(m, make_double2(v.real(), v.imag()));
                    }
                    scan.add(m);
                }
                if (!fix_ok(scan, fix_strict(n, rad[0]), exact_bits))
                    continue;
                ++taken;
                const std::vector<Cl> e = exact(x, rad, w);
                std::vector<double2> d(n);
                for (int j = 0; j < n; ++j)
                    d[j] = make_double2(x[j].real(), x[j].imag());
                stages(d, rad, [&](auto rc, size_t s, double2 *v, const auto &m) {
                    for (int r = 1; s && r < rc; ++r)
                        v[r] = cmul(v[r], make_double2((double)w[m(r)].real(), (double)w[m(r)].imag()));
                    Bfly<decltype(rc)::value>::run(v);
                });
                const int emax = fix_emax(mag_all(lm));
                std::vector<fix2> a(n);
                for (int j = 0; j < n; ++j)
                    a[j] = runtime ? fix2{to_fix<true>(x[j].real(), emax), to_fix<true>(x[j].imag(), emax)}
                                   : fix2{to_fix<false>(x[j].real(), emax), to_fix<false>(x[j].imag(), emax)};
                unsigned acc[12] = {};
                int sh = emax - 1081;
                for (size_t s = 0; s < rad.size(); ++s)
                    with_radix(rad[s], [&](auto rc) { sh += BflyFix<decltype(rc)::value, false>::scale + (s ? 2 : 0); });
                stages(a, rad, [&](auto rc, size_t s, fix2 *v, const auto &m) {
                    constexpr int RR = decltype(rc)::value;
                    for (int r = 0; s && r < RR; ++r) {
                        v[r] = shl(v[r], norm_shift(acc[s - 1]));
                        v[r] = r ? cmul62(v[r], root_fix(m(r), n)) : rounds ? quarter<true>(v[r]) : quarter<false>(v[r]);
                    }
                    rounds ? BflyFix<RR, true>::run(v) : BflyFix<RR, false>::run(v);
                    for (int r = 0; r < RR; ++r)
                        acc[s] |= norm_word(v[r].x) | norm_word(v[r].y);
                });
                for (size_t s = 0; s + 1 < rad.size(); ++s)
                    sh -= norm_shift(acc[s]);
                long double nn = 0, df = 0, dd = 0;
                for (int j = 0; j < n; ++j) {
                    nn += std::norm(e[j]);
                    df += std::norm(e[j] - Cl(from_fix(a[j].x, sh), from_fix_int(a[j].y, sh)));
                    dd += std::norm(e[j] - Cl(d[j].x, d[j].y));
                }
                efix += (double)(df / nn);
                e64 += (double)(dd / nn);
            }
            printf("%d %s %d %.4e %.4e\n", n, kind, taken, sqrt(efix / std::max(1, taken)), sqrt(e64 / std::max(1, taken)));
        }
    }
}
