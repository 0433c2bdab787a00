// Twiddle tables of the two-factor FFT kernels (host).
#pragma once
#include <cmath>
#include <vector>

namespace pp {

struct Twiddle {
    float x, y;
};

// Mean of |w|^2 - 1 that the FP32 constants of a register DFT leave in its output
// energy (pp_fft.cuh, pp_fft4.cuh, pp_fftgen.cuh): the radix kernels' own
// constants, and the inner twiddles of a composite A * B.
inline double reg_dft_gain(int N) {
    const double pi = 3.14159265358979323846;
    auto sq = [](double v) { const double f = (float)v; return f * f; };
    if (N <= 2 || N == 4) return 0.0;
    if (N == 3) return (3.0 + 2.0 * (1.0 + 2.0 * (0.25 + sq(std::sqrt(3.0) / 2.0)))) / 9.0 - 1.0;
    if (N == 5) {
        double e = 0.0;
        for (int q = 1; q <= 2; ++q) e += sq(std::cos(2.0 * pi * q / 5.0)) + sq(std::sin(2.0 * pi * q / 5.0));
        return (5.0 + 4.0 * (1.0 + 2.0 * e)) / 25.0 - 1.0;
    }
    if (N == 8) return 0.25 * (2.0 * sq(std::sqrt(0.5)) - 1.0);   // two of the eight inner products
    static const int ab[][2] = {{3, 2}, {3, 3}, {5, 2}, {4, 3}, {5, 3}, {4, 4}, {9, 2}, {4, 5}, {8, 3}, {5, 5}, {9, 3}, {10, 3}, {8, 4}};
    for (const auto& f : ab) {
        const int A = f[0], B = f[1];
        if (A * B != N) continue;
        double g = 0.0;
        for (int b = 0; b < B; ++b)
            for (int k = 0; k < A; ++k)
                g += sq(std::cos(2.0 * pi * b * k / N)) + sq(std::sin(2.0 * pi * b * k / N)) - 1.0;
        return reg_dft_gain(A) + reg_dft_gain(B) + g / N;
    }
    return 0.0;
}

// exp(-2 pi i t / n), t < n = n1 n2, of the kernels that multiply by W_n^(m k),
// m < n2, k < n1.  Rounding them and the register DFTs' constants to FP32 changes the
// transform's mean output energy by some 5e-8, always the same way, so that it adds
// up over the transforms of a solve where rounding does not.  The table is scaled by
// the largest factor that leaves the mean at 1 or below, so that a normalised operator
// stays one and FISTA's unit step stays safe (bisection: entries round one by one, so
// the mean falls short of 1 by less than one entry's step: 2e-8 at 16 and 32 points,
// 8e-9 at 80, 5e-9 at 256, mostly below 2e-9).  Coefficient gradients of a 3-iteration
// unrolled solve, differences of large sums, against 64 bits, mean of four data sets:
// 8 slices of 256 x 256 2.0e-6 with the plain table, 3.5e-7 so; 2 slices of 128 x 128
// with d = 2 2.5e-6 and 1.2e-6; of 384 x 384 with d = 1 3.0e-6 and 6.6e-7.
inline std::vector<Twiddle> balanced_twiddles(int n1, int n2) {
    const int n = n1 * n2;
    const double reg = reg_dft_gain(n1) + reg_dft_gain(n2);
    std::vector<double> c(n), s(n);
    std::vector<int> used(n, 0);   // products that take entry t
    for (int t = 0; t < n; ++t) {
        const double a = -2.0 * 3.14159265358979323846 * (double)t / (double)n;
        c[t] = std::cos(a);
        s[t] = std::sin(a);
    }
    for (int m = 0; m < n2; ++m)
        for (int k = 0; k < n1; ++k) ++used[m * k];
    auto table = [&](double scale) {
        std::vector<Twiddle> tw(n);
        for (int t = 0; t < n; ++t) tw[t] = {(float)(scale * c[t]), (float)(scale * s[t])};
        tw[0] = {1.f, 0.f};
        return tw;
    };
    auto gain = [&](const std::vector<Twiddle>& tw) {
        double e = 0.0;
        for (int t = 0; t < n; ++t)
            e += used[t] * ((double)tw[t].x * tw[t].x + (double)tw[t].y * tw[t].y - 1.0);
        return reg + e / n;
    };
    double lo = 1.0 - 5e-7, hi = 1.0 + 5e-7;
    for (int it = 0; it < 20; ++it) {
        const double mid = 0.5 * (lo + hi);
        (gain(table(mid)) > 0.0 ? hi : lo) = mid;
    }
    return table(lo);
}

}  // namespace pp
