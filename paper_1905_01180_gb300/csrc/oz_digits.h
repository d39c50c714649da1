// oz_digits.h - FP64 values as sums of 8-bit digits, and back: the arithmetic
// of the FP64 contraction on FP16 tensor cores (oz_gemm.cu), shared by the
// device code and a host-side test.
//
// The error-free splitting is that of Ozaki, Ogita, Oishi and Rump (Numer.
// Algorithms 59, 2012), with integer digits and one scale per row and K window.
// With E the largest biased exponent of the row's window, x = X 2^(E - 1076),
// |X| < 2^54, and X = sum_{i=0..6} d_i 2^(8 (6 - i)) with d_i in [-128, 127]
// (|d_0| <= 64): every digit is an FP16 integer.  The products of two windows
// are grouped by level l = i + j, weight 2^(96 - 8 l); a level's sum over a
// window of at most 96 K is an integer below 7 96 2^14 < 2^24, exact in the
// tensor core's FP32 accumulator.  Levels 0 .. 7 are kept (34 of the 49 digit
// products); the dropped ones are below 2^-60 of the window's largest product,
// less than the rounding of X (2^-55 of the row's largest element).
#pragma once

#include <cstdint>

#if defined(__CUDACC__)
#define GKBA_OZ_HD __host__ __device__ __forceinline__
#else
#define GKBA_OZ_HD inline
#endif

namespace gkba {

constexpr int kOzSlices = 7;   // digits of an element
constexpr int kOzLevels = 8;   // digit-product levels kept
constexpr int kOzMaxKw = 96;   // longest K window (exact level sums, see above)

// Biased exponent of an FP64 bit pattern's high word; subnormals count as 1.
GKBA_OZ_HD int oz_exponent(uint32_t hi) {
    const int e = (int)((hi >> 20) & 0x7FFu);
    return e > 1 ? e : 1;
}

// Digits of the FP64 bit pattern u at the window exponent E >= its own: byte
// 7 - i of the result is d_i + 128 (byte 0 is the dropped fraction; the added
// 0x80 in it rounds to nearest).  Negative values are complemented, not
// negated: off by 2^-8 of the last digit's unit.
GKBA_OZ_HD uint64_t oz_digits(uint64_t u, int E) {
    const uint32_t hi = (uint32_t)(u >> 32);
    const uint32_t ef = (hi >> 20) & 0x7FFu;
    const uint64_t m = ((uint64_t)((hi & 0xFFFFFu) | (ef ? 0x100000u : 0u)) << 32) | (uint32_t)u;
    const int s = E - (int)(ef > 1u ? ef : 1u);
    uint64_t t = s < 64 ? (m << 9) >> s : 0ull;
    const uint64_t neg = (uint64_t)((int64_t)u >> 63);
    t ^= neg;
    return t + 0x8080808080808080ull;
}

// Digit i (0 = leading) of an oz_digits word.
GKBA_OZ_HD int oz_digit(uint64_t t, int i) { return (int)((t >> (8 * (7 - i))) & 0xFF) - 128; }

// Round-to-nearest FP64 bit pattern of sum_l a_l 2^(96 - 8 l) 2^(Ea + Eb - 2152)
// for level sums a_0 .. a_7 of a window of at most 96 K.  Integer arithmetic
// only (the GPU's FP64 rate is 1/64 of its FP32 rate): the sum is formed as a
// 64-bit integer in units of 2^-44 of level 0, |W| < 2^62.6, and normalised.
// Ea or Eb = 0x7FF (a non-finite operand) gives NaN; results below the normal
// range give zero.
GKBA_OZ_HD int oz_clz64(uint64_t w) {
#if defined(__CUDA_ARCH__)
    return __clzll((long long)w);
#else
    return w ? __builtin_clzll(w) : 64;
#endif
}
GKBA_OZ_HD uint64_t oz_combine(const int (&a)[kOzLevels], int Ea, int Eb) {
    const int c = a[5] * 16 + ((a[6] + (a[7] >> 8)) >> 4);
    const int b3 = a[3] * 256 + a[4];
    const int b1 = a[1] * 256 + a[2];
    int64_t W = (int64_t)c + (int64_t)b3 * 4096 + (int64_t)b1 * (1 << 28);
    W = (int64_t)((uint64_t)W + ((uint64_t)(uint32_t)(a[0] * 4096) << 32));
    const uint64_t neg = (uint64_t)(W >> 63);
    uint64_t w = (uint64_t)W ^ neg;
    const int z = oz_clz64(w);
    w <<= z & 63;
    const int Er = Ea + Eb - z - 1014;
    uint64_t r = (w >> 11) + ((w >> 10) & 1u) + ((uint64_t)(uint32_t)(Er - 1) << 52);
    if (Er < 1 || z == 64) r = 0;
    if (Er > 2046 && z != 64) r = 0x7FF0000000000000ull;
    r |= neg & 0x8000000000000000ull;
    if (Ea == 0x7FF || Eb == 0x7FF) r = 0x7FF8000000000000ull;
    return r;
}

}  // namespace gkba
