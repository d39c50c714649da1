// Host check of the acceptance criterion of csrc/oz_digits.h: dot products of
// vectors whose exponents spread over a number of bits (x rising where y falls,
// in random order), through the digits where oz_accept takes them and by FMAs
// elsewhere, as the kernel does it.  Errors are relative to sum |x y|, in units of
// 2^-53.  Prints one "name value" line per quantity; "rms K spread ppm": the rms
// error over that of the FMA chain.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>

#include "oz_digits.h"

using namespace gkba;

static uint64_t bits(double x) {
    uint64_t u;
    std::memcpy(&u, &x, 8);
    return u;
}
static double dbl(uint64_t u) {
    double x;
    std::memcpy(&x, &u, 8);
    return x;
}
// value of the FP16 magnitude of an element whose leading digit is d0
static double mag(int d0, double x) {
    const uint32_t nz = oz_nonzero((uint32_t)(bits(x) >> 32), (uint32_t)bits(x));
    const int d = std::abs(d0);
    int e = 0;
    while (d >> (e + 1)) ++e;
    const uint32_t h = oz_magnitude(d == 0 ? 0x8000u : 0x8000u | (uint32_t)((15 + e) << 10) | (uint32_t)((d << (10 - e)) & 0x3FF), nz);
    if (h < 0x400u) return std::ldexp((double)h, -24);
    return std::ldexp(1024.0 + (h & 0x3FF), (int)(h >> 10) - 25);
}

struct Dot {
    double value;
    bool accepted;
};
static Dot dot(const double* x, const double* y, int K, double* fma_value) {
    uint32_t ea = kOzExpMin, eb = kOzExpMin;
    int a[kOzLevels] = {0};
    for (int k = 0; k < K; ++k) {
        ea = std::max(ea, (uint32_t)(bits(x[k]) >> 32) & kOzExpMask);
        eb = std::max(eb, (uint32_t)(bits(y[k]) >> 32) & kOzExpMask);
    }
    double M = 0.0, sx = 0.0, sy = 0.0, f = 0.0;
    for (int k = 0; k < K; ++k) {
        const uint64_t s = oz_digits((uint32_t)(bits(x[k]) >> 32), (uint32_t)bits(x[k]), ea);
        const uint64_t t = oz_digits((uint32_t)(bits(y[k]) >> 32), (uint32_t)bits(y[k]), eb);
        for (int i = 0; i < kOzSlices; ++i)
            for (int j = 0; j < kOzSlices && i + j < kOzLevels; ++j) a[i + j] += oz_digit(s, i) * oz_digit(t, j);
        const int dx = oz_digit(s, 0), dy = oz_digit(t, 0);
        M += mag(dx, x[k]) * mag(dy, y[k]);
        sx += dx * dx / 4096.0;
        sy += dy * dy / 4096.0;
        f = std::fma(x[k], y[k], f);
    }
    *fma_value = f;
    float fa[kOzLevels];
    for (int l = 0; l < kOzLevels; ++l) fa[l] = (float)a[l];
    const int Es = oz_exponent(ea) + oz_exponent(eb) - 1014;
    uint32_t hi, lo, ha, e1;
    oz_sum(fa, kOzMul, hi, lo);
    const double z = dbl(oz_pack(hi, lo, Es, kOzMul, ha, e1));
    const bool ok = oz_packed(ha, e1) && ea > kOzExpMin && eb > kOzExpMin &&
                    oz_accept((float)M, kOzAccept * (float)sx + kOzAccept * (float)sy);
    if (ok) return {z, true};
    return {M == 0.0 && Es < kOzNonFinite / 2 ? 0.0 : f, false};
}

int main() {
    std::mt19937_64 r(7);
    std::normal_distribution<double> n;
    long long over = 0;
    for (int K : {4, 8, 10, 20, 33, 48, 66, 96})
        for (int spread : {0, 4, 8, 12, 16, 24, 36, 48}) {
            double e2 = 0.0, f2 = 0.0;
            long long taken = 0;
            const int reps = 4000;
            for (int rep = 0; rep < reps; ++rep) {
                double x[96], y[96], hi = 0.0, lo = 0.0, S = 0.0, f;
                for (int k = 0; k < K; ++k) {
                    x[k] = std::ldexp(n(r), (int)(r() % (spread + 1)));
                    y[k] = std::ldexp(n(r), -(int)(r() % (spread + 1)));
                    const double p = x[k] * y[k], pe = std::fma(x[k], y[k], -p);
                    const double s = hi + p, b = s - hi;
                    lo += ((hi - (s - b)) + (p - b)) + pe;
                    hi = s;
                    S += std::fabs(p);
                }
                const Dot d = dot(x, y, K, &f);
                const double e = std::fabs((d.value - hi) - lo) / S * 0x1p53, ef = std::fabs((f - hi) - lo) / S * 0x1p53;
                // worst case of an accepted result: 2^-55 (sum x / X + sum y / Y) of the largest
                // product, by Cauchy and Schwarz and the criterion; digits are rounded to 1 / 64
                over += d.accepted && e > 1.1 * 1024.0 * std::sqrt(2.0 * K / kOzAccept) + 2.0;
                taken += d.accepted;
                e2 += e * e;
                f2 += ef * ef;
            }
            std::printf("rms_%d_%d %lld\ntaken_%d_%d %lld\n", K, spread, (long long)(1e6 * std::sqrt(e2 / f2)), K, spread,
                        (long long)(1e6 * taken / reps));
        }
    std::printf("over_bound %lld\n", over);
    // small elements that meet zeros or small ones, zeros, the ends of the range
    struct Case {
        double x[3], y[3], value;
    };
    const double inf = INFINITY;
    const Case cases[] = {
        {{1.0, 1e-17, 0.0}, {0.0, 1.0, 0.0}, 1e-17},
        {{1.0, 1e-12, 3e-12}, {0.0, 0.75, 0.25}, std::fma(3e-12, 0.25, 1e-12 * 0.75)},
        {{1.3, 0x1.1p-60, 0.0}, {0x1.3p-60, 1.7, 0.0}, std::fma(0x1.1p-60, 1.7, 1.3 * 0x1.3p-60)},
        {{1.0, 0x1p-1074, 0.0}, {0.0, 2.0, 0.0}, 0x1p-1073},
        {{1.0, 0.0, 2.0}, {0.0, 5.0, 0.0}, 0.0},
        {{0x1p-600, 0.0, 0.0}, {0x1p-460, 0.0, 0.0}, 0x1p-1060},
        {{0x1p-1000, 0.0, 0.0}, {0x1.8p500, 0.0, 0.0}, 0x1.8p-500},
        {{inf, 0.0, 0.0}, {2.0, 0.0, 0.0}, inf},
        {{0x1p1000, 0.0, 0.0}, {-0x1p100, 0.0, 0.0}, -inf},
    };
    long long wrong = 0;
    double f;
    for (const Case& c : cases) wrong += dot(c.x, c.y, 3, &f).value != c.value;
    const double ni[3] = {inf, 1.0, 0.0}, zero[3] = {0.0, 1.0, 0.0};
    wrong += !std::isnan(dot(ni, zero, 3, &f).value);  // infinity times zero
    std::printf("wrong %lld\n", wrong);
    return 0;
}
