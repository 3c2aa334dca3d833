// The ring stage's tables (roots of unity, Bluestein filters, Rader kernels,
// fold weights) as fixed-point complex numbers, in the place of the doubles
// they are built from: {low, high} balanced halves of the real and of the
// imaginary part, v = (high 2^32 + low) 2^-62 with low signed (-2^31 left out,
// so that a sign flip is one negation a half); the fold weights, of modulus up
// to 2, in units of 2^-61.  Plan files hold the doubles.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

struct shtb_plan_s;

namespace shtb {

constexpr int kRootBits = 62, kFoldBits = 61;

inline double ring_half_unpack(int lo, int hi, int bits)
{
    return (double)((int64_t)hi * 4294967296LL + lo) / (double)(1ULL << bits);
}

}  // namespace shtb

#ifdef __CUDACC__
namespace shtb_dev {

__device__ __forceinline__ int2 ring_half_pack(double v, int bits)
{
    long long q = __double2ll_rn(v * (double)(1ULL << bits));
    if ((int)q == (int)0x80000000) ++q;
    const int lo = (int)q;
    return make_int2(lo, (int)((q - lo) >> 32));
}

__device__ __forceinline__ const int4 *ring_table(const double2 *p) { return reinterpret_cast<const int4 *>(p); }

}  // namespace shtb_dev
#endif
