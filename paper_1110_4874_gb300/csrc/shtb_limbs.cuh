// FP64 sums of products as 64-bit integer ones, for factors that a thread
// makes itself (the recurrence kernels of shtb_legendre.cu): numbers of a
// common exponent as two signed limbs of radix 2^28, a product as three
// 32 x 32 + 64-bit multiply-adds (P += ah bh, M += ah bl + al bh, value
// P 2^56 + M 2^28; the product of the low limbs is below the cut).  A
// multiply-add takes a warp half a clock of an SM, a DFMA 16.
#pragma once

#include <cuda_runtime.h>

#include "shtb_bf_fix.cuh"

namespace shtb_dev {

// (P 2^28 + M) 2^q rounded to nearest, be0 = q + 28 + 1054, for results in the normal range
__device__ __forceinline__ double limbs_to_double(long long P, long long M, int be0)
{
    const long long top = P + (M >> 28);
    int hi = (int)(top >> 32);
    unsigned mid = (unsigned)top, low = (unsigned)M << 4;
    int pos = bfind_s32(hi);                        // the leading bit is bit pos of the upper word
    if (pos < 0) {                                  // upper word empty: |top| < 2^32
        hi = (int)__funnelshift_l(mid, (unsigned)hi, 31);
        mid = __funnelshift_l(low, mid, 31);
        low <<= 31;
        be0 -= 31;
        pos = bfind_s32(hi);
        if (pos < 0) return 0.0;
    }
    const int sm = hi >> 31, n = 30 - pos;
    const unsigned zh = __funnelshift_l(mid, (unsigned)hi, n) ^ (unsigned)sm;
    const unsigned zl = __funnelshift_l(low, mid, n) ^ (unsigned)sm;
    const unsigned long long z = ((unsigned long long)zh << 32 | zl) + 0x200u;    // bit 62 leads; keep 53 bits
    const unsigned rl = (unsigned)(z >> 10), rh = (unsigned)(z >> 42);
    return __hiloint2double((int)((rh + ((unsigned)(be0 + pos) << 20)) | ((unsigned)sm & 0x80000000u)), (int)rl);
}

// v as limbs of a whole number: its 53 bits at the top of 64, less sh (PTX
// clamps shifts above 63 to an empty result: zeros and subnormals, whose
// exponent field is 0, under a scale that is not)
__device__ __forceinline__ int2 to_limbs(double v, int sh)
{
    const int hi = __double2hiint(v), lo = __double2loint(v);
    const unsigned mh = __funnelshift_l((unsigned)lo, (unsigned)hi, 11) | 0x80000000u;
    unsigned long long a;
    asm("shr.u64 %0, %1, %2;" : "=l"(a) : "l"((unsigned long long)mh << 32 | ((unsigned)lo << 11)), "r"(sh));
    const long long s = (long long)(hi >> 31);
    const long long X = (long long)(a ^ (unsigned long long)s) - s;
    return make_int2((int)((unsigned)X << 4) >> 4, (int)((X + (1 << 27)) >> 28));
}

__device__ __forceinline__ long long mad_wide(int a, int b, long long c)
{
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

__device__ __forceinline__ int exp_bits(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

}  // namespace shtb_dev
