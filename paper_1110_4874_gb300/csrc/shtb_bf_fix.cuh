// Block products of the butterfly, out[n][c] = sum_k T[k][n] v[k][c], on the
// tensor cores, to the last place of FP64: both factors are fixed-point
// numbers cut into six signed digits of radix 2^10, the digit products run as
// f16 MMAs whose FP32 sums are whole numbers, exact up to 2^24 (see below), and
// the sums are put together in integer arithmetic and rounded to double once.
//
// Why: the FP64 pipe does 2 FMAs a clock on an SM (a warp's DFMA occupies it
// for 16 clocks), the legacy f16 MMA 1024.  21 digit products of 10 bits a
// side replace an FP64 product, and what surrounds them is 32-bit integer
// work at 64 to 128 lanes a clock.  The MMA form is mma.sync and not tcgen05
// because the blocks are small and ragged (about 24 x 20 elements, each with
// its own input vector): a 128-row tcgen05 tile would be mostly padding, and
// its operands would have to be expanded to 12 bytes an element in shared
// memory, while here the 8-byte words go from global memory to registers.
//
// T: words of shtb_fix.h (58 bits, 54 stored, exponent E per column).
// v: X = v 2^{1079 - e} cut to a whole number, |X| < 2^57, e the largest
// biased exponent of the component over a chunk of at most 32 entries k.
// With digits t_i, u_j, pairs with i + j <= 5 are kept: the sum of diagonal
// d = i + j carries 2^{10 (10 - d)}.  The dropped diagonals are below 2^-57
// of max|T| max|v| per product (rms), the cuts of T and v below 2^-55 and
// 2^-56; an FP64 FMA chain over 24 entries rounds to 2^-53 of its partial
// sums 24 times.  On the compressed Legendre blocks of Nside = 256, L = 512
// the relative rms error is 0.9e-16 with the words' 54 bits, against 1.6e-16
// of the FMA chain.
// FP32 sums over 32 entries: |t_0| <= 256, |u_0| <= 128, the other digits at
// most 512, so diagonals 0, 1, 2 stay below 2^20, 2^22.6 and 2^23.9 and are
// exact.  Diagonals 3, 4 and 5 have 2^24.5, 2^24.9 and 2^25.2 as their largest
// and pass 2^24, from where a sum is rounded to even, at 73, 53 and 42 % of it:
// only if digits that large meet with one sign in all entries and pairs.  A unit
// of diagonal 3, 4 or 5 is 2^-45, 2^-55 or 2^-65 of max|T| max|v|.  Digits of T
// (interpolation weights and Legendre functions) are as good as random, ten
// standard deviations away from that; where they repeat along a sum (the
// constant l = 0 function, over a block's rings) the worst vector brings
// diagonals 3 and 4 to 76 and 95 % of 2^24, and diagonal 5 past it.
//
// Measured (GB300, Nside = 512, L = 1024, eps = 1e-10; residual blocks plus
// levels, FP64 FMA kernels before): 8 maps 5.31 -> 1.50 ms, 4 maps 2.79 ->
// 1.23, 2 maps 1.69 -> 0.95, 1 map 0.93 -> 0.79; at 8 maps the adjoint's
// levels and residual blocks 5.75 -> 1.83 ms.  What bounds them now is the
// latency of loads and of the integer chains at 16 warps an SM (issue slots
// 41-52 % used, tensor pipe 17-29 %, FP64 pipe 1 %).
//
// Results do not depend on the other components, on how maps are grouped or
// on the lane layout: the sums are exact (but for the vectors just named), and
// chunks of 32 are added in FP64 in order.  The digits of -x are not those of x
// negated, so a negated input gives the negated result up to its last place.
// A component whose chunk holds an infinity or a NaN gives NaN.
#pragma once

#include <cuda_runtime.h>

#include "shtb_fix.h"

namespace shtb_dev {

constexpr int kFixChunk = 32;              // contraction entries per exponent and accumulator pass

// d = a b + c; c = zero for a sum's first product
__device__ __forceinline__ void mma_k16(float (&d)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3,
                                        unsigned b0, unsigned b1, bool first)
{
    if (first)
        asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%10,%10,%10,%10};"
            : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
            : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
    else
        asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},{%0,%1,%2,%3};"
            : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
            : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void mma_k8(float (&d)[4], unsigned a0, unsigned a1, unsigned b0, bool first)
{
    if (first)
        asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5},{%6},{%7,%7,%7,%7};"
            : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
            : "r"(a0), "r"(a1), "r"(b0), "f"(0.f));
    else
        asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5},{%6},{%0,%1,%2,%3};"
            : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
            : "r"(a0), "r"(a1), "r"(b0));
}

// Two digits as f16: the 10-bit fields at bits 0 and 16 of x become 1024 + f
// by setting the exponent bits, less 1024 + 512 is the signed digit (exact).
constexpr unsigned kF16Magic = 0x64006400u, kF16Bias = 0x66006600u, kF16Field = 0x03ff03ffu;

__device__ __forceinline__ unsigned f16_digits(unsigned magic_fields)
{
    unsigned h;
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(h) : "r"(magic_fields), "r"(kF16Bias));
    return h;
}

__device__ __forceinline__ unsigned f16_field(unsigned x) { return f16_digits((x & kF16Field) | kF16Magic); }

// the digits of two words of T, a in the low halves
__device__ __forceinline__ void word_digits(uint2 a, uint2 b, unsigned (&h)[6])
{
    const unsigned p0 = __byte_perm(a.x, b.x, 0x5410), q0 = __byte_perm(a.x, b.x, 0x7632);
    const unsigned p1 = __byte_perm(a.y, b.y, 0x5410), q1 = __byte_perm(a.y, b.y, 0x7632);
    h[0] = f16_field(p0);
    h[1] = f16_field(q0);
    h[2] = f16_digits((((q0 >> 4) & 0x03c003c0u) | ((p0 >> 10) & 0x003f003fu)) | kF16Magic);
    h[3] = f16_field(p1);
    h[4] = f16_field(q1);
    h[5] = f16_digits(((p1 >> 6) & 0x03f003f0u) | kF16Magic);
}

// v in units of 2^(emax - 1079), toward zero, plus the digit bias (60 bits):
// the low word and the top 30 bits (digits 5, 4, 3 and 2, 1, 0 at bits 0, 10,
// 20); sh = 7 + emax - (v's exponent).  A zero has exponent field 0 and so,
// in a vector whose emax is in the range below, a shift above 63, which PTX
// clamps to an empty result; the same goes for subnormals.
__device__ __forceinline__ uint2 vec_fix(double v, int sh)
{
    const int hi = __double2hiint(v), lo = __double2loint(v);
    const unsigned mh = __funnelshift_l((unsigned)lo, (unsigned)hi, 11) | 0x80000000u;
    unsigned long long X;
    asm("shr.u64 %0, %1, %2;" : "=l"(X) : "l"((unsigned long long)mh << 32 | ((unsigned)lo << 11)), "r"(sh));
    const long long s = (long long)(hi >> 31);
    const unsigned long long y = (X ^ (unsigned long long)s) + (shtb::kFixDigitBias - (unsigned long long)s);
    return make_uint2((unsigned)y, (unsigned)(y >> 30));
}

__device__ __forceinline__ void vec_digits(uint2 a, uint2 b, unsigned (&h)[6])
{
    h[0] = f16_field(__byte_perm(a.y, b.y, 0x7632) >> 4);
    h[1] = f16_field(__byte_perm(a.y, b.y, 0x6521) >> 2);
    h[2] = f16_field(__byte_perm(a.y, b.y, 0x5410));
    h[3] = f16_field(__byte_perm(a.x, b.x, 0x7632) >> 4);
    h[4] = f16_field(__byte_perm(a.x, b.x, 0x6521) >> 2);
    h[5] = f16_field(__byte_perm(a.x, b.x, 0x5410));
}

// Chunk exponents the digits are made at (effective, biased): results and all
// intermediate shifts then stay in range.  A component of magnitudes below
// 1e-217 or above 1e204 is brought there by 2^+-kFixLift and its outputs
// brought back; one that is not finite gets zero digits and its outputs NaN.
constexpr int kFixExpLo = 300, kFixExpHi = 1700, kFixLift = 600;
// what a component's outputs need (two bits): nothing, 2^-kFixLift, 2^kFixLift, NaN
enum { kFixAsIs = 0, kFixLifted = 1, kFixLowered = 2, kFixNaN = 3 };

__device__ __forceinline__ double fix_after(double v, int what)
{
    if (what == kFixAsIs) return v;
    return v * (what == kFixLifted ? shtb::pow2(-kFixLift) : what == kFixLowered ? shtb::pow2(kFixLift)
                                                                               : __longlong_as_double(0x7ff8000000000000LL));
}

// The sums of the six diagonals, V = sum_d acc_d 2^{10 (5 - d)}, without
// their low 8 bits (2^-62 of the largest possible sum): |V| < 2^71
__device__ __forceinline__ long long fix_combine(float a0, float a1, float a2, float a3, float a4, float a5)
{
    const int i0 = __float2int_rn(a0), i1 = __float2int_rn(a1), i2 = __float2int_rn(a2);
    const int i3 = __float2int_rn(a3), i4 = __float2int_rn(a4), i5 = __float2int_rn(a5);
    const int top = i0 * 1024 + i1 + (i2 >> 10) + (i3 >> 20);
    const unsigned long long low = (unsigned long long)((unsigned)i2 << 22) + ((unsigned)i3 << 12);
    return (long long)(((unsigned long long)(unsigned)top << 32) + low) + (long long)(i4 * 4 + (i5 >> 8));
}

__device__ __forceinline__ int bfind_s32(int x)
{
    int r;
    asm("bfind.s32 %0, %1;" : "=r"(r) : "r"(x));
    return r;
}

// Y 2^q rounded to nearest, be0 = q + 1054, for results in the normal range
__device__ __forceinline__ double fix_to_double(long long Y, int be0)
{
    int pos = bfind_s32((int)(Y >> 32));            // the leading bit is bit pos of the upper word
    if (pos < 0) {                                  // upper word empty: |Y| < 2^32
        Y = (long long)((unsigned long long)Y << 31);
        be0 -= 31;
        pos = bfind_s32((int)(Y >> 32));
        if (pos < 0) return 0.0;                    // 0 or one unit, 2^-62 of the largest possible sum
    }
    const int hi = (int)(Y >> 32), sm = hi >> 31;
    const unsigned lo = (unsigned)Y;
    const int n = 30 - pos;
    const unsigned zh = __funnelshift_l(lo, (unsigned)hi, n) ^ (unsigned)sm, zl = (lo << n) ^ (unsigned)sm;
    const unsigned long long z = ((unsigned long long)zh << 32 | zl) + 0x200u;    // bit 62 leads; keep 53 bits
    const unsigned rl = (unsigned)(z >> 10), rh = (unsigned)(z >> 42);
    return __hiloint2double((int)((rh + ((unsigned)(be0 + pos) << 20)) | ((unsigned)sm & 0x80000000u)), (int)rl);
}

// A vector's chunk is digitised by pairs of entries (2i, 2i + 1), W components
// of each on a lane.  NP pairs a lane: raw values in, 2^20 x the largest
// exponent of each component out; reduce(e) takes the maximum over the lanes
// that share a component.  Components outside the digits' range are brought
// into it and what their outputs need is left in `after`, two bits each.
template <bool EXPN, int NP, int W, class Max>
__device__ __forceinline__ void vec_scale(double (&raw)[NP][2][W], const int (&sh)[NP][2], int (&ev)[W], int &after,
                                          const Max &reduce)
{
    auto largest = [&](int c, int &field) {
        int e = -(1 << 30);
        field = 0;
#pragma unroll
        for (int q = 0; q < NP; ++q)
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const int f = __double2hiint(raw[q][p][c]) & 0x7ff00000;
                e = max(e, EXPN ? f : f + sh[q][p]);
                if (!EXPN) field = max(field, f);
            }
        return reduce(e);
    };
    bool rare = false;
#pragma unroll
    for (int c = 0; c < W; ++c) {
        int field;
        ev[c] = largest(c, field);
        if (!EXPN && reduce(field) == 0x7ff00000) ev[c] = 0x7ff00000;
        rare |= ev[c] < kFixExpLo << 20 || ev[c] > kFixExpHi << 20;
    }
    after = 0;
    if (!__any_sync(0xffffffffu, rare)) return;
#pragma unroll
    for (int c = 0; c < W; ++c) {
        const bool in = ev[c] >= kFixExpLo << 20 && ev[c] <= kFixExpHi << 20, finite = ev[c] != 0x7ff00000;
        const bool low = ev[c] < kFixExpLo << 20;
        const double f = in ? 1.0 : shtb::pow2(low ? kFixLift : -kFixLift);
        int field, e;
#pragma unroll
        for (int q = 0; q < NP; ++q)
#pragma unroll
            for (int p = 0; p < 2; ++p) raw[q][p][c] = finite ? raw[q][p][c] * f : 0.0;
        e = largest(c, field);
        const bool zero = e < kFixExpLo << 20;                       // (a lifted value lies above it)
        if (!in) after |= (!finite ? kFixNaN : zero ? kFixAsIs : low ? kFixLifted : kFixLowered) << 2 * c;
        ev[c] = zero ? kFixExpLo << 20 : e;
    }
}

template <bool EXPN>
__device__ __forceinline__ void vec_pair(double v0, double v1, int sh0, int sh1, int ev, unsigned (&h)[6])
{
    const int e7 = ev + (7 << 20);
    const int f0 = __double2hiint(v0) & 0x7ff00000, f1 = __double2hiint(v1) & 0x7ff00000;
    const uint2 x0 = vec_fix(v0, (EXPN ? e7 - f0 : e7 - f0 - sh0) >> 20);
    const uint2 x1 = vec_fix(v1, (EXPN ? e7 - f1 : e7 - f1 - sh1) >> 20);
    vec_digits(x0, x1, h);
}

// One chunk of kc entries from k0 on, NG = ceil(kc / 8) groups of 8: the
// digits of the vector, then the outputs tile by tile (see fix_product).  NG
// is a template argument so that the loop over the outputs has no branches.
// The words of the first tile are asked for before the vector's digits are
// made, those that follow before the products of the step at hand.
//
// 16 components: they are the 16 rows of the MMA (rows g and g + 8 are
// components 2g and 2g + 1), 8 outputs its columns.
template <int C, bool EXPN, int NG, class Vec, class Out>
__device__ __forceinline__ void fix_chunk_wide(const uint2 *__restrict__ T, int sk, int sn, int k0, int kc, int nn,
                                               const Vec &vec, const Out &out, int lane)
{
    static_assert(C == 16, "one component per MMA row");
    constexpr int NS = (NG + 1) / 2;
    const int g = lane >> 2, t = lane & 3;
    const uint2 *__restrict__ Tk = T + (size_t)(k0 + 2 * t) * sk;
    uint2 w[NG][2];
    auto load_words = [&](int n0) {
        const uint2 *__restrict__ Tn = Tk + (size_t)min(n0 + g, nn - 1) * sn;
#pragma unroll
        for (int q = 0; q < NG; ++q, Tn += 8 * sk) {
            w[q][0] = __ldg(Tn);
            w[q][1] = __ldg(Tn + sk);
        }
    };
    load_words(0);
    unsigned A[NS][6][4];                                            // digit fragments of the k16 (or k8) steps
    int ev[2], after;                                                // chunk exponents, 2^20 e
    {
        double raw[NG][2][2];
        int sh[NG][2];                                               // 2^20 x the entry's own exponent
#pragma unroll
        for (int q = 0; q < NG; ++q)
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const int k = 8 * q + 2 * t + p;
                sh[q][p] = 0;
                raw[q][p][0] = raw[q][p][1] = 0.0;
                if (q < NG - 1 || k < kc) {
                    vec.load(k0 + k, g, raw[q][p]);
                    if (!EXPN) sh[q][p] = vec.shift(k0 + k) << 20;
                }
            }
        vec_scale<EXPN>(raw, sh, ev, after, [](int e) {
            e = max(e, __shfl_xor_sync(0xffffffffu, e, 1));
            return max(e, __shfl_xor_sync(0xffffffffu, e, 2));
        });
#pragma unroll
        for (int q = 0; q < NG; ++q)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                unsigned h[6];
                vec_pair<EXPN>(raw[q][0][c], raw[q][1][c], sh[q][0], sh[q][1], ev[c], h);
#pragma unroll
                for (int j = 0; j < 6; ++j) A[q >> 1][j][(q & 1) * 2 + c] = h[j];
            }
    }
    const bool rare = __any_sync(0xffffffffu, after != 0);
    for (int n0 = 0; n0 < nn; n0 += 8) {
        // where the tile's outputs go is looked up before the products
        int key[2];
#pragma unroll
        for (int x = 0; x < 2; ++x) key[x] = out.key(min(n0 + 2 * t + x, nn - 1));
        float acc[6][4];
        int Eg = 0;
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            constexpr int last = NG - 1;
            const bool k16 = 2 * s + 1 < NG;
            unsigned b0[6], b1[6];
            word_digits(w[2 * s][0], w[2 * s][1], b0);
            if (k16) word_digits(w[k16 ? 2 * s + 1 : last][0], w[k16 ? 2 * s + 1 : last][1], b1);
            if (s == NS - 1) {
                if (EXPN) Eg = shtb::fix_word_exp(w[0][0].x, w[0][0].y);
                load_words(n0 + 8);
            }
#pragma unroll
            for (int j = 0; j < 6; ++j)
#pragma unroll
                for (int i = 0; i + j < 6; ++i) {
                    const unsigned *a = A[s][i];
                    if (k16) mma_k16(acc[i + j], a[0], a[1], a[2], a[3], b0[j], b1[j], s == 0 && j == 0);
                    else mma_k8(acc[i + j], a[0], a[1], b0[j], s == 0 && j == 0);
                }
        }
        // columns 2t and 2t + 1 of the tile; the column's exponent comes
        // from the lane that loaded its words
        int E[2];
#pragma unroll
        for (int x = 0; x < 2; ++x) E[x] = EXPN ? __shfl_sync(0xffffffffu, Eg, (2 * t + x) * 4) : 0;
        auto finish = [&](auto back) {
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                if (n0 + 2 * t + x >= nn) continue;
                double v[2];
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const int f = x + 2 * c;
                    const long long Y = fix_combine(acc[0][f], acc[1][f], acc[2][f], acc[3][f], acc[4][f], acc[5][f]);
                    v[c] = back(fix_to_double(Y, E[x] + (ev[c] >> 20) + (1054 - 1079)), c);
                }
                out.put(key[x], k0 > 0, g, v);
            }
        };
        if (!rare) finish([](double v, int) { return v; });
        else finish([after](double v, int c) { return fix_after(v, after >> 2 * c & 3); });
    }
}

// 2, 4 or 8 components: 16 outputs are the MMA's rows and the components its
// 8 columns (column g is component g mod C), which halves the products per
// word.  The vector's pairs are spread over all lanes and shuffled into the
// fragments, and the repeated columns leave each output with several lanes,
// of which one puts it together: with one map (C = 2) each lane digitises one
// pair and finishes one output per tile, where the wide form would use a
// quarter of the lanes for four of each.
template <int C, bool EXPN, int NG, class Vec, class Out>
__device__ __forceinline__ void fix_chunk_narrow(const uint2 *__restrict__ T, int sk, int sn, int k0, int kc, int nn,
                                                 const Vec &vec, const Out &out, int lane)
{
    static_assert(C == 2 || C == 4 || C == 8, "components per entry");
    constexpr int NS = (NG + 1) / 2, PL = 32 / C, NP = (4 * NG + PL - 1) / PL;   // pairs per pass and passes
    const int g = lane >> 2, t = lane & 3;
    const uint2 *__restrict__ Tk = T + (size_t)(k0 + 2 * t) * sk;
    uint2 w[2][2][2];                                                // [row g, g + 8][half of the k16 step][pair]
    auto load_words = [&](int n0, int s) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const uint2 *__restrict__ Tn = Tk + (size_t)min(n0 + 8 * r + g, nn - 1) * sn + (size_t)(16 * s) * sk;
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (2 * s + h < NG) {
                    w[r][h][0] = __ldg(Tn + (size_t)(8 * h) * sk);
                    w[r][h][1] = __ldg(Tn + (size_t)(8 * h + 1) * sk);
                }
        }
    };
    load_words(0, 0);
    unsigned B[NS][2][6];                                            // digit fragments
    int ev[2], after;
    {
        // pair PL r + lane / C of component lane mod C
        double raw[NP][2][1];
        int sh[NP][2], e[1];
        const int c = lane & (C - 1);
#pragma unroll
        for (int r = 0; r < NP; ++r)
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const int k = 2 * (PL * r + lane / C) + p;
                sh[r][p] = 0;
                raw[r][p][0] = 0.0;
                if (k < kc) {
                    vec.load(k0 + k, c, raw[r][p]);
                    if (!EXPN) sh[r][p] = vec.shift(k0 + k) << 20;
                }
            }
        vec_scale<EXPN>(raw, sh, e, after, [](int x) {
#pragma unroll
            for (int o = C; o < 32; o *= 2) x = max(x, __shfl_xor_sync(0xffffffffu, x, o));
            return x;
        });
        unsigned h[NP][6];
#pragma unroll
        for (int r = 0; r < NP; ++r) vec_pair<EXPN>(raw[r][0][0], raw[r][1][0], sh[r][0], sh[r][1], e[0], h[r]);
        // fragment (s, half): column g takes pair 8 s + 4 half + t
#pragma unroll
        for (int s = 0; s < NS; ++s)
#pragma unroll
            for (int q = 0; q < 2; ++q)
                if (2 * s + q < NG) {
                    const int pr = 8 * s + 4 * q;                    // + t, all in pass pr / PL
                    const int src = (pr % PL + t) * C + (g & (C - 1));
#pragma unroll
                    for (int j = 0; j < 6; ++j) B[s][q][j] = __shfl_sync(0xffffffffu, h[pr / PL][j], src);
                }
        // exponents of the components this lane finishes
        ev[0] = __shfl_sync(0xffffffffu, e[0], C == 2 ? t & 1 : (2 * t) & (C - 1));
        ev[1] = __shfl_sync(0xffffffffu, e[0], C == 2 ? t & 1 : (2 * t + 1) & (C - 1));
        if (__any_sync(0xffffffffu, after != 0)) {
            const int a0 = __shfl_sync(0xffffffffu, after, C == 2 ? t & 1 : (2 * t) & (C - 1));
            const int a1 = __shfl_sync(0xffffffffu, after, C == 2 ? t & 1 : (2 * t + 1) & (C - 1));
            after = a0 | a1 << 2;
        }
    }
    const bool rare = __any_sync(0xffffffffu, after != 0);
    for (int n0 = 0; n0 < nn; n0 += 16) {
        constexpr int NOUT = C == 8 ? 2 : 1;                         // rows this lane finishes
        int key[NOUT];
#pragma unroll
        for (int x = 0; x < NOUT; ++x) key[x] = out.key(min(n0 + g + 8 * (NOUT == 2 ? x : t >> 1), nn - 1));
        float acc[6][4];
        int E[2] = {0, 0};
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const bool k16 = 2 * s + 1 < NG;
            unsigned a[4][6];
            word_digits(w[0][0][0], w[0][0][1], a[0]);
            word_digits(w[1][0][0], w[1][0][1], a[1]);
            if (k16) {
                word_digits(w[0][1][0], w[0][1][1], a[2]);
                word_digits(w[1][1][0], w[1][1][1], a[3]);
            }
            if (EXPN && s == 0)                                      // from lane t = 0, whose entry k0 is in the block
#pragma unroll
                for (int x = 0; x < 2; ++x)
                    E[x] = __shfl_sync(0xffffffffu, shtb::fix_word_exp(w[x][0][0].x, w[x][0][0].y), 4 * g);
            if (s < NS - 1) load_words(n0, s + 1);
            else load_words(n0 + 16, 0);
#pragma unroll
            for (int j = 0; j < 6; ++j)
#pragma unroll
                for (int i = 0; i + j < 6; ++i) {
                    if (k16) mma_k16(acc[i + j], a[0][j], a[1][j], a[2][j], a[3][j], B[s][0][i], B[s][1][i], s == 0 && j == 0);
                    else mma_k8(acc[i + j], a[0][j], a[1][j], B[s][0][i], s == 0 && j == 0);
                }
        }
        // rows g and g + 8, columns 2t and 2t + 1
        auto finish = [&](auto back) {
            if constexpr (C == 2) {
                // both components of both rows on every t: lane t takes row g + 8 (t / 2), component t mod 2
                float f[6];
#pragma unroll
                for (int d = 0; d < 6; ++d) {
                    const float lo = t & 1 ? acc[d][1] : acc[d][0], hi = t & 1 ? acc[d][3] : acc[d][2];
                    f[d] = t & 2 ? hi : lo;
                }
                if (n0 + g + 8 * (t >> 1) < nn) {
                    const double v[1] = {back(fix_to_double(fix_combine(f[0], f[1], f[2], f[3], f[4], f[5]),
                                                            (t & 2 ? E[1] : E[0]) + (ev[0] >> 20) + (1054 - 1079)), 0)};
                    out.put(key[0], k0 > 0, t & 1, v);
                }
            } else if constexpr (C == 4) {
                // lanes t and t + 2 hold components 2 (t mod 2), + 1: one takes row g, the other row g + 8
                if (n0 + g + 8 * (t >> 1) < nn) {
                    double v[2];
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        float f[6];
#pragma unroll
                        for (int d = 0; d < 6; ++d) f[d] = t & 2 ? acc[d][2 + c] : acc[d][c];
                        v[c] = back(fix_to_double(fix_combine(f[0], f[1], f[2], f[3], f[4], f[5]),
                                                  (t & 2 ? E[1] : E[0]) + (ev[c] >> 20) + (1054 - 1079)), c);
                    }
                    out.put(key[0], k0 > 0, t & 1, v);
                }
            } else {
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    if (n0 + g + 8 * x >= nn) continue;
                    double v[2];
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const int f = 2 * x + c;
                        v[c] = back(fix_to_double(fix_combine(acc[0][f], acc[1][f], acc[2][f], acc[3][f], acc[4][f], acc[5][f]),
                                                  E[x] + (ev[c] >> 20) + (1054 - 1079)), c);
                    }
                    out.put(key[x], k0 > 0, t, v);
                }
            }
        };
        if (!rare) finish([](double v, int) { return v; });
        else finish([after](double v, int c) { return fix_after(v, after >> 2 * c & 3); });
    }
}

template <int C, bool EXPN, int NG, class Vec, class Out>
__device__ __forceinline__ void fix_chunk(const uint2 *__restrict__ T, int sk, int sn, int k0, int kc, int nn,
                                          const Vec &vec, const Out &out, int lane)
{
    if constexpr (C == 16) fix_chunk_wide<C, EXPN, NG>(T, sk, sn, k0, kc, nn, vec, out, lane);
    else fix_chunk_narrow<C, EXPN, NG>(T, sk, sn, k0, kc, nn, vec, out, lane);
}

// out.put(out.key(n), add, i, v) for every n < nn and component: v[W] the
// components W i .. W i + W - 1 (W = 1 or 2) of sum_{k < kn} T[k sk + n sn]
// vec[k]; add: v goes on top of an earlier chunk.  EXPN: the words' exponents
// belong to n (a column is contracted over), else to k (vec.shift(k) returns
// them).  vec.load(k, i, x): components W i .. of entry k, called once for
// each entry and component.  All 32 lanes take part.  The words of up to 7 entries past kn are read (and meet zero
// digits): plan arrays are allocated with that slack.
template <int C, bool EXPN, class Vec, class Out>
__device__ __forceinline__ void fix_product(const uint2 *__restrict__ T, int sk, int sn, int kn, int nn, const Vec &vec,
                                            const Out &out, int lane)
{
#pragma unroll 1
    for (int k0 = 0; k0 < kn; k0 += kFixChunk) {
        const int kc = min(kFixChunk, kn - k0);
        if (nn <= 0) {
            // no outputs: the entries are still read (a level child's identity part)
            constexpr int W = C == 16 ? 2 : 1, NC = C / W;
            double x[W];
            for (int i = lane; i < kc * NC; i += 32) vec.load(k0 + i / NC, i % NC, x);
            continue;
        }
        if (kc > 24) fix_chunk<C, EXPN, 4>(T, sk, sn, k0, kc, nn, vec, out, lane);
        else if (kc > 16) fix_chunk<C, EXPN, 3>(T, sk, sn, k0, kc, nn, vec, out, lane);
        else if (kc > 8) fix_chunk<C, EXPN, 2>(T, sk, sn, k0, kc, nn, vec, out, lane);
        else fix_chunk<C, EXPN, 1>(T, sk, sn, k0, kc, nn, vec, out, lane);
    }
}

// Where an entry is read: shared memory (or data the same lane wrote),
// global memory through L1, or through L2 only for data produced earlier in
// the same launch (L1 is not coherent between SMs within one launch).
enum class Ld { kPlain, kGlobal, kL2 };

template <Ld M, class T>
__device__ __forceinline__ T ld_as(const T *p)
{
    if constexpr (M == Ld::kGlobal) return __ldg(p);
    else if constexpr (M == Ld::kL2) return __ldcg(p);
    else return *p;
}

// components W i .. of an entry at p (16-byte aligned)
template <Ld M, int W>
__device__ __forceinline__ void ld_comps(const double *p, int i, double (&x)[W])
{
    if constexpr (W == 2) {
        const double2 y = ld_as<M>(reinterpret_cast<const double2 *>(p) + i);
        x[0] = y.x;
        x[1] = y.y;
    } else {
        x[0] = ld_as<M>(p + i);
    }
}

// ... stored, or added to what is there
template <int W>
__device__ __forceinline__ void st_comps(double *p, int i, const double (&x)[W], bool add)
{
    if constexpr (W == 2) {
        double2 *q = reinterpret_cast<double2 *>(p) + i;
        double2 y = make_double2(x[0], x[1]);
        if (add) {
            const double2 o = *q;
            y.x = o.x + x[0];
            y.y = o.y + x[1];
        }
        *q = y;
    } else {
        p[i] = add ? p[i] + x[0] : x[0];
    }
}

}  // namespace shtb_dev
