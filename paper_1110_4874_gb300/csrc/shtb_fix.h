// Stored elements of the butterfly operator (interpolation blocks T and
// residual blocks R) as self-describing 64-bit fixed-point words, in the
// place of the doubles they are built from.
//
// A column of a block (the k elements that make one dense output) shares one
// exponent E, 2^{E-1} <= max |t| < 2^E, and each element is
//   t = X 2^{E - 58},  |X| <= 2^58, X a multiple of 16: 54 bits and a sign,
// rounded to nearest, so an element as large as its column's largest is
// exact and the others are off by at most 2^{E-55}, a quarter of the last
// place of the largest element.  X is kept as six signed digits of radix
// 2^10, X = sum_i D_i 2^{10 (5 - i)} (|D_0| <= 256, the others in -512 ..
// 511, D_5 a multiple of 16), each biased by 512 to f_i in 0 .. 1023: the
// digits are what the tensor cores multiply (see shtb_bf_fix.cuh), and the
// bit places are chosen so that the digits of two elements are brought to
// the halves of a register by a byte permutation and a mask:
//   low word   f_0 at 0, f_2's low 6 bits at 10, f_1 at 16, f_2's high 4
//              bits at 26, the low 2 bits of E + kFixExpBias at 30;
//   high word  f_3 at 0, f_5 / 16 at 10, f_4 at 16, the high 6 bits of
//              E + kFixExpBias at 26.
// Plan files hold the doubles (fix_unpack on the way out, the pack kernel on
// the way in); packing an unpacked block gives the same words.
#pragma once

#include <cstdint>
#include <cstring>

namespace shtb {

constexpr int kFixExpBias = 191;      // 8 bits hold E = -191 .. 64
constexpr int kFixExpMax = 255 - kFixExpBias;
constexpr uint64_t kFixDigitBias = 512ULL * (1ULL + (1ULL << 10) + (1ULL << 20) + (1ULL << 30) + (1ULL << 40) +
                                             (1ULL << 50));

#ifdef __CUDACC__
#define SHTB_HD __host__ __device__
#else
#define SHTB_HD
#endif

// the word of X (a multiple of 16) and e8 = E + kFixExpBias
SHTB_HD inline uint64_t fix_word(int64_t X, int e8)
{
    const uint64_t y = (uint64_t)X + kFixDigitBias;
    const uint32_t f0 = (uint32_t)(y >> 50) & 1023, f1 = (uint32_t)(y >> 40) & 1023, f2 = (uint32_t)(y >> 30) & 1023;
    const uint32_t f3 = (uint32_t)(y >> 20) & 1023, f4 = (uint32_t)(y >> 10) & 1023, f5 = (uint32_t)y & 1023;
    const uint32_t lo = f0 | (f2 & 63) << 10 | f1 << 16 | (f2 >> 6) << 26 | ((uint32_t)e8 & 3) << 30;
    const uint32_t hi = f3 | (f5 >> 4) << 10 | f4 << 16 | ((uint32_t)e8 >> 2) << 26;
    return (uint64_t)hi << 32 | lo;
}

SHTB_HD inline int fix_word_exp(uint32_t lo, uint32_t hi)
{
    return (int)((hi >> 26) << 2 | lo >> 30) - kFixExpBias;
}

// X of a word
SHTB_HD inline int64_t fix_word_int(uint32_t lo, uint32_t hi)
{
    const uint64_t f0 = lo & 1023, f1 = (lo >> 16) & 1023, f2 = ((lo >> 10) & 63) | ((lo >> 26) & 15) << 6;
    const uint64_t f3 = hi & 1023, f4 = (hi >> 16) & 1023, f5 = ((hi >> 10) & 63) << 4;
    return (int64_t)((f0 << 50) + (f1 << 40) + (f2 << 30) + (f3 << 20) + (f4 << 10) + f5 - kFixDigitBias);
}

// 2^n, -1022 <= n <= 1023
SHTB_HD inline double pow2(int n)
{
    const uint64_t b = (uint64_t)(n + 1023) << 52;
    double d;
    memcpy(&d, &b, sizeof d);
    return d;
}

// the double a word stands for (exact: X / 16 has at most 54 bits and is a
// multiple of 2 above 2^53)
SHTB_HD inline double fix_unpack(uint64_t w)
{
    const uint32_t lo = (uint32_t)w, hi = (uint32_t)(w >> 32);
    return (double)(fix_word_int(lo, hi) / 16) * pow2(fix_word_exp(lo, hi) - 54);
}

}  // namespace shtb
