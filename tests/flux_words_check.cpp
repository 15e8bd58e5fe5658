// Host check of the three-word residual (flux_words.h) against quadruple
// precision, over cells of n per side: smooth and rough neighbours, boundary
// faces, faces over many decades, residuals near the rounding of the values.
// For every cell, beyond the rounding of the differences themselves, the error
// is at most 2^-62 of c sum |k d| (third words only are rounded) plus 2^-46 of
// the residual (which goes on as an FP32 number and into a sum of squares); over
// a family of cells the mean square of the error beyond that last rounding is at
// most that of the FP64 form. Prints "ok" or the first excess.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "flux_words.h"

#ifdef __SIZEOF_FLOAT128__
typedef __float128 quad;
#else
typedef long double quad;  // 113 bits where there is no __float128
#endif

static double size(quad x) { return static_cast<double>(x < 0 ? -x : x); }

int main()
{
    using namespace mlqmc_words;
    std::mt19937_64 g(1806);
    std::uniform_real_distribution<double> U(-1.0, 1.0);
    std::normal_distribution<double> N(0.0, 1.0);
    for (const int n : {32, 36, 96, 128, 320, 1024, 4096})
        for (int family = 0; family < 6; ++family) {
            const float c = static_cast<float>(n) * static_cast<float>(n);
            double ss_words = 0.0, ss_fp64 = 0.0;
            for (int cell = 0; cell < 20000; ++cell) {
                // 0 smooth, 1 beside a corner, 2 unrelated neighbours, 3 faces over 2^+-40,
                // 4 and 5: a solved equation (k = 1; rough k), u off by its rounding alone
                double up = 0.04 * (1.1 + U(g)), nb[4];
                float k[4];
                for (int j = 0; j < 4; ++j) {
                    k[j] = family == 4 ? 1.0f : static_cast<float>(std::exp(N(g) * (family == 3 ? 9.0 : 1.0)));
                    nb[j] = family == 2 ? 0.04 * (1.1 + U(g)) : up * (1.0 + 4.0 * U(g) / n);
                }
                if (family == 1) nb[0] = nb[2] = 0.0;
                if (family >= 4) {
                    const double part = k[0] * (up - nb[0]) + k[1] * (up - nb[1]) + k[2] * (up - nb[2]);
                    nb[3] = up - (1.0 / c - part) / k[3];
                }
                quad sum = 0, sum_d = 0;
                double mag = 0.0;
                for (int j = 0; j < 4; ++j) {
                    const quad d = static_cast<quad>(up) - static_cast<quad>(nb[j]);
                    sum += static_cast<quad>(k[j]) * d;
                    sum_d += static_cast<quad>(k[j]) * static_cast<quad>(up - nb[j]);
                    mag += size(static_cast<quad>(c) * static_cast<quad>(k[j]) * d);
                }
                float b, rem;
                residual(c, flux(k[0], up, nb[0]), flux(k[1], nb[1], up), flux(k[2], up, nb[2]), flux(k[3], nb[3], up), b, rem);
                const quad r = static_cast<quad>(b) + static_cast<quad>(rem);
                const double excess = size(r - (1 - static_cast<quad>(c) * sum_d));
                if (!(excess <= 0x1p-62 * mag + 0x1p-46 * size(r))) {
                    std::printf("n %d family %d cell %d: off by 2^%.1f of the fluxes\n", n, family, cell, std::log2(excess / mag));
                    return 1;
                }
                double acc = static_cast<double>(k[0]) * (up - nb[0]);
                for (int j = 1; j < 4; ++j) acc = std::fma(static_cast<double>(k[j]), up - nb[j], acc);
                const double r64 = std::fma(-static_cast<double>(c), acc, 1.0);
                const quad exact = 1 - static_cast<quad>(c) * sum;
                const double ew = std::fmax(0.0, size(r - exact) - 0x1p-46 * size(r)) / mag, ef = size(static_cast<quad>(r64) - exact) / mag;
                ss_words += ew * ew;
                ss_fp64 += ef * ef;
            }
            if (!(ss_words <= ss_fp64)) {
                std::printf("n %d family %d: mean square %.3e against FP64's %.3e\n", n, family, ss_words, ss_fp64);
                return 1;
            }
        }
    // the parts of a difference: exact for 53 bits at every exponent the bit operations take, at both ends
    // of the range, and to 2^-72 or the smallest FP32 number beyond it
    for (int e = -180; e <= 127; ++e)
        for (int rep = 0; rep < 200; ++rep) {
            const double d = std::ldexp(rep == 0 ? 2.0 - 0x1p-52 : 1.0 + std::fabs(U(g)) * (1.0 - 0x1p-52), e) * (rep & 1 ? -1.0 : 1.0);
            const Words w = split(d);
            const quad s = static_cast<quad>(w.h) + static_cast<quad>(w.m) + static_cast<quad>(w.l);
            if (w.h - w.h != 0.0f) {
                if (e == 127 && rep < 200) continue;  // rounds up to infinity: the caller sees it and takes FP64
                std::printf("split(%a) overflows\n", d);
                return 1;
            }
            if (size(s - static_cast<quad>(d)) > (e >= -74 ? 0.0 : 0x1p-149)) {
                std::printf("split(%a): %a %a %a\n", d, w.h, w.m, w.l);
                return 1;
            }
        }
    for (const double d : {0.0, -0.0}) {
        const Words w = split(d);
        if (w.h != 0.0f || w.m != 0.0f || w.l != 0.0f) return 1;
    }
    std::printf("ok\n");
    return 0;
}
