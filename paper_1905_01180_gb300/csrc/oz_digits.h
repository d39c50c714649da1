// oz_digits.h - FP64 values as sums of 8-bit digits, and back: the arithmetic
// of the FP64 contraction on FP16 tensor cores (oz_gemm.cu), shared by the
// device code and a host-side test.
//
// The error-free splitting is that of Ozaki, Ogita, Oishi and Rump (Numer.
// Algorithms 59, 2012), with integer digits and one scale per row and K window.
// With E the largest biased exponent of the row's window (at least 64),
// x = X 2^(E - 1076), |X| < 2^54, and X = sum_{i=0..6} d_i 2^(8 (6 - i)) with
// d_i in [-128, 127] (|d_0| <= 64): every digit is an FP16 integer.  The products
// of two windows are grouped by level l = i + j, weight 2^(96 - 8 l); a level's
// sum over a window of at most 96 K is an integer below 7 96 2^14 < 2^24, exact
// in the tensor core's FP32 accumulator.  Levels 0 .. 7 are kept (34 of the 49
// digit products); the dropped ones sum to at most 2^-57.6 of the window's largest
// product a term (five digit products of up to 2^14 at level 8, of 2^108), less
// than the rounding of X (2^-55 of the row's largest element).
//
// That error is normwise: 2^-55 of the largest elements times the other operand,
// whatever the elements that meet.  Where small elements meet large ones, or zeros,
// it can exceed the rounding of an FMA chain, which is relative to sum |x y|, by any
// factor.  So every window result carries M = sum |d_0(x)| |d_0(y)| (one more MMA)
// and is taken only if its error is small against M (oz_accept); the others are
// summed again by FMAs.  Results that leave the normal range and rows with Inf, NaN
// or nothing above 2^-958 go the same way.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#if defined(__CUDACC__)
#define GKBA_OZ_HD __host__ __device__ __forceinline__
#else
#define GKBA_OZ_HD inline
#endif

namespace gkba {

constexpr int kOzSlices = 7;   // digits of an element
constexpr int kOzLevels = 8;   // digit-product levels kept
constexpr int kOzMaxKw = 96;   // longest K window (exact level sums, see above)

constexpr uint32_t kOzExpMask = 0x7FF00000u;
constexpr uint32_t kOzExpMin = 64u << 20;     // floor of E: zeros need a shift of 64
constexpr int kOzNonFinite = 0x10000;         // window exponent of a row with Inf or NaN

// Window exponent E from the largest exponent field (high word, masked) of a row.
GKBA_OZ_HD int oz_exponent(uint32_t emax) { return emax == kOzExpMask ? kOzNonFinite : (int)(emax >> 20); }

// Digits of the FP64 value (hi, lo) for a row whose largest exponent field is
// emax >= kOzExpMin: byte 7 - i of the result is d_i + 128 (byte 0 is the
// dropped fraction; the 0x80 added to it rounds to nearest).  Negative values
// are complemented, not negated: off by 2^-8 of the last digit's unit.
GKBA_OZ_HD uint64_t oz_digits(uint32_t hi, uint32_t lo, uint32_t emax) {
    const uint32_t s = (emax >> 20) - ((hi << 1) >> 21);
    const uint32_t m = (hi & 0xFFFFFu) | 0x100000u;
    uint64_t t = ((uint64_t)((m << 9) | (lo >> 23)) << 32) | (uint32_t)(lo << 9);
#if defined(__CUDA_ARCH__)
    asm("shr.u64 %0, %1, %2;" : "=l"(t) : "l"(t), "r"(s));  // 0 for s >= 64
#else
    t = s < 64 ? t >> s : 0ull;
#endif
    const uint64_t neg = (uint64_t)((int64_t)((uint64_t)hi << 32) >> 63);
    return (t ^ neg) + 0x8080808080808080ull;
}

// Magnitude of an element for M, as FP16 bits: |d_0|, its last bit set for every
// element but zero, so that M = 0 means that no two nonzero elements meet.  d0: the
// FP16 bits of d_0.
GKBA_OZ_HD uint32_t oz_nonzero(uint32_t hi, uint32_t lo) {
    const uint32_t any = (hi & 0x7FFFFFFFu) | lo;
    return any < 1u ? any : 1u;
}
GKBA_OZ_HD uint32_t oz_magnitude(uint32_t d0, uint32_t nonzero) { return (d0 & 0x7FFFu) | nonzero; }

// Acceptance of a window result.  With unit errors of 2^-55 / sqrt(3) an element its
// error is e = 2^-55 / sqrt(3) sqrt(sx + sy) of the largest product, sx = sum (d_0(x) / 64)^2,
// and |x|.|y| is M / 64^2 of it: M^2 >= c (sx + sy) bounds e by 2^-53 590 / sqrt(c) of
// sum |x y|, 3.3 2^-53 here (an FMA chain's rms error is 0.5 to 2 2^-53 of it).  Well
// scaled operands stay far below the bound (0.2 to 0.5) and nearly all of their results
// are taken: of random ones at N = 10, 24 and 33 all but 6e-4, 2e-6 and 4e-7 in stage S1
// and 2e-4, 0 and 0 in S2 (twice the constant: 4e-3, 5e-5 and 1e-5; 3e-3, 0 and 0).
constexpr float kOzAccept = 32768.0f;
GKBA_OZ_HD bool oz_accept(float M, float cs) { return M * M >= cs; }  // cs = c (sx + sy)

// Digit i (0 = leading) of an oz_digits word.
GKBA_OZ_HD int oz_digit(uint64_t t, int i) { return (int)((t >> (8 * (7 - i))) & 0xFF) - 128; }

// Powers of two as run-time values.  The multiply-adds by them then stay on the
// FMA pipe; as constants they become shifts and adds on the integer pipe, which
// has half the rate and bounds the kernels that use this header.
struct OzMul {
    int m4, m8, m12, m20, m28, one;
};
constexpr OzMul kOzMul = {1 << 4, 1 << 8, 1 << 12, 1 << 20, 1 << 28, 1};

#if defined(__CUDA_ARCH__)
__device__ __forceinline__ uint32_t oz_mad(uint32_t a, int b, uint32_t c) {
    uint32_t d;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
__device__ __forceinline__ int64_t oz_mad_wide(int a, int b, int64_t c) {
    int64_t d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}
GKBA_OZ_HD uint32_t oz_bits(float x) { return __float_as_uint(x); }
GKBA_OZ_HD int oz_int(float x) { return __float2int_rn(x); }
GKBA_OZ_HD int oz_clz(uint32_t x) { return __clz((int)x); }
GKBA_OZ_HD float oz_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
#else
inline uint32_t oz_mad(uint32_t a, int b, uint32_t c) { return a * (uint32_t)b + c; }
inline int64_t oz_mad_wide(int a, int b, int64_t c) { return (int64_t)a * b + c; }
inline uint32_t oz_bits(float x) {
    uint32_t u;
    std::memcpy(&u, &x, 4);
    return u;
}
inline int oz_int(float x) { return (int)std::lrintf(x); }
inline int oz_clz(uint32_t x) { return x ? __builtin_clz(x) : 32; }
inline float oz_fma(float a, float b, float c) { return std::fmaf(a, b, c); }
#endif

// FP64 bit pattern (round to nearest) of sum_l a_l 2^(96 - 8 l) 2^(Ea + Eb - 2152)
// for the level sums a_0 .. a_7 of a window of at most 96 K; Es = Ea + Eb - 1014.
// Integer and FP32 arithmetic only (the FP64 rate is 1/64 of the FP32 rate).
//
// oz_sum: the sum as a 64-bit integer W = (hi, lo) in units of 2^-44 of level 0
// (|W| < 2^62.6).  The sums of levels 0 - 2 are below 2^22 and become integers
// by adding 1.5 2^23 (the conversion instruction runs at an eighth of the FP32
// rate; the constant's bits 0x4B400000 vanish modulo 2^32 when shifted by 12);
// levels 6 and 7 are rounded to W's unit together.
GKBA_OZ_HD void oz_sum(const float (&a)[kOzLevels], const OzMul& k, uint32_t& hi, uint32_t& lo) {
    const float kMagic = 12582912.0f;
    const uint32_t m0 = oz_bits(a[0] + kMagic), m1 = oz_bits(a[1] + kMagic), m2 = oz_bits(a[2] + kMagic);
    const int c = (int)oz_mad((uint32_t)oz_int(a[5]), k.m4,
                              (uint32_t)oz_int(oz_fma(a[7], 1.0f / 4096.0f, a[6] * 0.0625f)));
    const int b3 = (int)oz_mad((uint32_t)oz_int(a[3]), k.m8, (uint32_t)oz_int(a[4]));
    const int b1 = (int)oz_mad(m1, k.m8, m2 - 257u * 0x4B400000u);
    const int64_t W = oz_mad_wide(b1, k.m28, oz_mad_wide(b3, k.m12, (int64_t)c));
    hi = oz_mad(m0, k.m12, (uint32_t)((uint64_t)W >> 32));
    lo = (uint32_t)W;
}
// W as FP64 when its absolute value's high word ha is not zero and the biased
// exponent e1 + 1 is in 1 .. 2046 (the caller checks both).
GKBA_OZ_HD uint64_t oz_pack(uint32_t hi, uint32_t lo, int Es, const OzMul& k, uint32_t& ha, uint32_t& e1) {
    const uint32_t neg = (uint32_t)((int32_t)hi >> 31);
    ha = hi ^ neg;
    // leading bit to bit 62, half a unit of the last place added, exponent in place
    const int z = oz_clz(ha);
    uint64_t w = ((uint64_t)ha << 32) | (lo ^ neg);
    w = (uint64_t)oz_mad_wide(0x200, k.one, (int64_t)(w << (z - 1))) >> 10;
    e1 = (uint32_t)(Es - 1 - z);
    const uint32_t rh = oz_mad(e1, k.m20, (uint32_t)(w >> 32)) | (neg & 0x80000000u);
    return ((uint64_t)rh << 32) | (uint32_t)w;
}
GKBA_OZ_HD bool oz_packed(uint32_t ha, uint32_t e1) { return ha != 0u && e1 <= 2045u; }
// W as FP64 in every case, to check the packing above against: Es >= kOzNonFinite / 2
// (a non-finite operand) gives NaN, results below the normal range zero.
GKBA_OZ_HD uint64_t oz_pack_any(uint32_t hi, uint32_t lo, int Es) {
    const uint32_t neg = (uint32_t)((int32_t)hi >> 31);
    hi ^= neg;
    lo ^= neg;
    int z = oz_clz(hi);
    if (hi == 0) z = 32 + oz_clz(lo);
    uint64_t w = ((uint64_t)hi << 32) | lo;
    w = ((w << ((z - 1) & 63)) + 0x200u) >> 10;
    const int Er = (hi | lo) == 0 ? Es - 4096 : Es - z;
    uint32_t rh = (uint32_t)(w >> 32) + ((uint32_t)(Er - 1) << 20), rl = (uint32_t)w;
    if ((uint32_t)(Er - 1) > 2045u) {
        rh = Es >= kOzNonFinite / 2 ? 0x7FF80000u : Er > 2046 ? 0x7FF00000u : 0u;
        rl = 0u;
    }
    return ((uint64_t)(rh | (neg & 0x80000000u)) << 32) | rl;
}

}  // namespace gkba
