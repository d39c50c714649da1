// Host check of csrc/oz_digits.h: dot products of FP64 vectors through the
// 8-bit digits, as the FP16 tensor-core GEMM forms them, against double-double
// sums.  Prints one "name value" line per quantity.
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

// sum_k x_k y_k through the digits; *big: a digit or a level sum out of range
static double oz_dot(const double* x, const double* y, int K, bool* big) {
    uint32_t ea = kOzExpMin, eb = kOzExpMin;
    int a[kOzLevels] = {0};
    for (int k = 0; k < K; ++k) {
        ea = std::max(ea, (uint32_t)(bits(x[k]) >> 32) & kOzExpMask);
        eb = std::max(eb, (uint32_t)(bits(y[k]) >> 32) & kOzExpMask);
    }
    for (int k = 0; k < K; ++k) {
        const uint64_t s = oz_digits((uint32_t)(bits(x[k]) >> 32), (uint32_t)bits(x[k]), ea);
        const uint64_t t = oz_digits((uint32_t)(bits(y[k]) >> 32), (uint32_t)bits(y[k]), eb);
        for (int i = 0; i < kOzSlices; ++i)
            for (int j = 0; j < kOzSlices && i + j < kOzLevels; ++j) {
                if (std::abs(oz_digit(s, i)) > 128) *big = true;
                a[i + j] += oz_digit(s, i) * oz_digit(t, j);
            }
    }
    float f[kOzLevels];
    for (int l = 0; l < kOzLevels; ++l) {
        if (std::abs(a[l]) >= (l < 3 ? 1 << 22 : 1 << 24)) *big = true;
        f[l] = (float)a[l];
    }
    const int Es = oz_exponent(ea) + oz_exponent(eb) - 1014;
    uint32_t hi, lo, ha, e1;
    oz_sum(f, kOzMul, hi, lo);
    const uint64_t r = oz_pack_any(hi, lo, Es), fast = oz_pack(hi, lo, Es, kOzMul, ha, e1);
    if (oz_packed(ha, e1) && fast != r) *big = true;  // the two packings agree
    return dbl(r);
}

int main() {
    std::mt19937_64 r(1);
    std::normal_distribution<double> n;
    long long over_bound = 0, level_overflow = 0;
    double e_oz = 0.0, e_fma = 0.0;  // rms errors over the largest products, K >= 16
    const int Ks[] = {1, 2, 7, 16, 33, 48, 96};
    for (int K : Ks)
        for (int rep = 0; rep < 20000; ++rep) {
            double x[96], y[96], mx = 0.0, my = 0.0;
            const int spread = (rep % 4) * 12;  // exponents within a vector: 1, 12, 24, 36 bits
            for (int k = 0; k < K; ++k) {
                x[k] = std::ldexp(n(r), (int)(r() % (spread + 1)));
                y[k] = std::ldexp(n(r), -(int)(r() % (spread + 1)));
                if (rep % 97 == 0) x[k] = std::ldexp(1.0, rep % 3) * (r() & 1 ? 1 : -1) * (2.0 - 0x1p-52);  // all at the top
                if (rep % 97 == 0) y[k] = 2.0 - 0x1p-52;
                mx = std::max(mx, std::fabs(x[k]));
                my = std::max(my, std::fabs(y[k]));
            }
            double hi = 0.0, lo = 0.0, f = 0.0;  // double-double sum (two-sum, two-product)
            for (int k = 0; k < K; ++k) {
                const double p = x[k] * y[k], pe = std::fma(x[k], y[k], -p);
                const double s = hi + p, b = s - hi;
                lo += ((hi - (s - b)) + (p - b)) + pe;
                hi = s;
                f = std::fma(x[k], y[k], f);
            }
            bool big = false;
            const double z = oz_dot(x, y, K, &big);
            level_overflow += big;
            const double err = std::fabs((z - hi) - lo);
            // two rounded operands per product, the cut of the 64-bit sum, the final rounding
            const double bound = (K * (0x1.02p-53 + 0x1p-57) + 0x1p-53) * mx * my + 0x1p-53 * std::fabs(hi);
            over_bound += err > bound;
            if (K >= 16) {
                e_oz += err * err / (mx * mx * my * my * K);
                const double ef = std::fabs((f - hi) - lo);
                e_fma += ef * ef / (mx * mx * my * my * K);
            }
        }
    std::printf("over_bound %lld\nlevel_overflow %lld\nerror_ratio_ppm %lld\n", over_bound, level_overflow,
                (long long)(1e6 * std::sqrt(e_oz / e_fma)));
    // products of two numbers are rounded correctly, with any exponents
    long long one_bad = 0;
    for (int i = 0; i < 200000; ++i) {
        const double x = std::ldexp(n(r), (int)(r() % 900) - 450), y = std::ldexp(n(r), (int)(r() % 900) - 450);
        bool big = false;
        const double z = oz_dot(&x, &y, 1, &big);
        one_bad += big || std::fabs(z - x * y) > 0x1p-52 * std::fabs(x * y);
    }
    std::printf("one_bad %lld\n", one_bad);
    const double zero = 0.0, one = 1.0, inf = INFINITY, nan = NAN, mone = -1.0, tiny = 0x1p-1074, half = 0.5;
    const double huge = 0x1p1000;
    bool b = false;
    int special = 0;
    special += oz_dot(&zero, &one, 1, &b) == 0.0;
    special += oz_dot(&one, &mone, 1, &b) == -1.0;
    special += std::isnan(oz_dot(&inf, &one, 1, &b));
    special += std::isnan(oz_dot(&one, &nan, 1, &b));
    special += oz_dot(&tiny, &half, 1, &b) == 0.0;          // below the normal range
    special += std::isinf(oz_dot(&huge, &huge, 1, &b));
    special += oz_dot(&tiny, &huge, 1, &b) == 0.0;          // below the floor of the window exponent
    std::printf("special %d\n", special);
    return 0;
}
