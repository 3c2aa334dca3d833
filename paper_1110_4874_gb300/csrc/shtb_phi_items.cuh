// Device bodies of the ring stage (Eq. sh-baseline, Eq. tau): the fold of a
// ring's spectrum, its mixed-radix, Rader or Bluestein FFT in shared memory,
// and the adjoint, used by the ring kernels of shtb_phi.cu and by the
// persistent batch kernel of shtb_batch.cu.
//
// The transforms run in 64-bit fixed point.  An SM does 2 FP64 instructions a
// clock but 56 32 x 32 + 64-bit multiply-adds and 61 64-bit additions, so a
// complex product (12 multiply-adds on balanced 32-bit halves) costs 6 clocks
// a warp where its four FP64 instructions cost 64, and an addition 1 where
// FP64 takes 16.  A ring's points share one power of two: every pass first
// shifts them up so that the largest component has 61 bits (its size is known
// from the pass before: one OR a component, one shared-memory OR a warp) and
// then works without overflow, rounding its results to whole units.  It scales
// down by 2 to 6 bits (pass_bits), so its results keep 55 to 61 bits of the
// largest point.  Relative rms error of a ring (Nside = 256, FP64 transforms ->
// these; white noise, and with one pixel 1e5 times the rest): adjoint 2.5e-16
// -> 1.6e-16 and 2.4e-16 -> 1.7e-16 where K is a power of two, 2.5..2.7e-16 ->
// 1.7..2.0e-16 with a factor 3 to 13, Rader 4.0e-16 -> 3.1e-16 and 3.9e-16 ->
// 3.4e-16, Bluestein 4.8e-16 -> 3.7e-16; synthesis the same to 10 %.
// Measured (Nside = 512, L = 1024, 8 maps; FP64 transforms before): ring
// synthesis 1.80 -> .87 ms, adjoint 2.42 -> .96 ms; Nside = 1024: 7.60 ->
// 3.83 and 9.79 -> 4.05 ms (1.14, 1.16, 3.90 and 4.12 by the change of
// arithmetic alone).  What bounds them now is the issue of integer
// instructions at the direct lengths (65 to 71 % of the slots) and latency
// and instruction fetches at the others (36 to 49 %, 16 warps an SM).
// Rings whose largest value lies outside 1e-217 .. 1e204 are brought into that
// range by a power of two; rings that hold an infinity or a NaN are filled with
// NaN.
#pragma once

#include <cuda_runtime.h>

#include "shtb_bf_fix.cuh"
#include "shtb_internal.h"
#include "shtb_ring_fix.h"

namespace shtb_dev {

__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }

// sign flips as integer operations on the sign bit (no FP64 instruction)
__device__ __forceinline__ double dneg_if(double x, int neg)
{
    return __longlong_as_double(__double_as_longlong(x) ^ ((long long)(neg & 1) << 63));
}
__device__ __forceinline__ double2 cneg_if(double2 a, int neg)
{
    return make_double2(dneg_if(a.x, neg), dneg_if(a.y, neg));
}
__device__ __forceinline__ double2 cconj_i(double2 a) { return make_double2(a.x, dneg_if(a.y, 1)); }

template <bool CG>
__device__ __forceinline__ double2 ldq(const double2 *p)
{
    return CG ? __ldcg(p) : __ldg(p);
}

// G_r = sum over m = r (mod J), |m| <= L, of (-1)^{s t} q_m (m = r + tJ),
// with q_m = conj(q_{-m}) for m < 0.  The first term starts the sum (no add
// to zero) and the signs are flipped bitwise, so every FP64 instruction here
// is one of the sum's additions.
template <class QAt>
__device__ __forceinline__ double2 fold_G(QAt qat, int L, int J, int s, int r)
{
    double2 acc;
    int mp, tt;                         // negative terms m = -mp, mp = tt J - r
    if (r <= L) {
        acc = qat(r);
        int t = 1;
        for (int m = r + J; m <= L; m += J, ++t) acc = cadd(acc, cneg_if(qat(m), s & t));
        mp = J - r;
        tt = 1;
    } else {
        mp = J - r;                     // r in (L, J): only negative terms
        if (mp > L) return make_double2(0.0, 0.0);
        acc = cneg_if(cconj_i(qat(mp)), s);
        mp += J;
        tt = 2;
    }
    for (; mp <= L; mp += J, ++tt) acc = cadd(acc, cneg_if(cconj_i(qat(mp)), s & tt));
    return acc;
}

// The terms of fold_G number part, part + parts, .. of both signs
template <class QAt>
__device__ __forceinline__ double2 fold_part(QAt qat, int L, int J, int s, int r, int part, int parts)
{
    double2 acc = make_double2(0.0, 0.0);
    int t = part;
    for (int m = r + part * J; m <= L; m += parts * J, t += parts) acc = cadd(acc, cneg_if(qat(m), s & t));
    t = part + 1;
    for (int mp = t * J - r; mp <= L; mp += parts * J, t += parts) acc = cadd(acc, cneg_if(cconj_i(qat(mp)), s & t));
    return acc;
}

// ------------------------------------------------ fixed-point complex numbers
typedef longlong2 fx2;

__device__ __forceinline__ fx2 fadd(fx2 a, fx2 b) { return make_longlong2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ fx2 fsub(fx2 a, fx2 b) { return make_longlong2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ fx2 fconj(fx2 a) { return make_longlong2(a.x, -a.y); }
__device__ __forceinline__ fx2 ftimes_i(fx2 a) { return make_longlong2(-a.y, a.x); }
__device__ __forceinline__ fx2 fshl(fx2 a, int s) { return make_longlong2(a.x << s, a.y << s); }

// a / 2^n to nearest (n >= 1)
__device__ __forceinline__ long long rshift(long long a, int n) { return (a + (1LL << (n - 1))) >> n; }
__device__ __forceinline__ fx2 frshift(fx2 a, int n) { return make_longlong2(rshift(a.x, n), rshift(a.y, n)); }

// balanced halves, a = h 2^32 + l with l signed
__device__ __forceinline__ void halves(long long a, int &h, int &l)
{
    l = (int)a;
    h = (int)(a >> 32) - (l >> 31);
}

// table entries: {low, high} balanced halves of the real and the imaginary
// part in units of 2^-62 (fold weights 2^-61; shtb_ring_fix.h)
__device__ __forceinline__ int4 wneg_if(int4 w, bool neg)
{
    return neg ? make_int4(-w.x, -w.y, -w.z, -w.w) : w;
}

// a w / 4 (CONJ: a conj(w) / 4) for |a| < 2^62: the products of the high
// halves, and of high and low halves over 2^32, both exact in 64 bits; those
// of the low halves are below half a unit
template <bool CONJ = false>
__device__ __forceinline__ fx2 fmul(fx2 a, int4 w)
{
    int ah, al, bh, bl;
    halves(a.x, ah, al);
    halves(a.y, bh, bl);
    const int cl = w.x, ch = w.y;
    const int dl = CONJ ? -w.z : w.z, dh = CONJ ? -w.w : w.w, nl = CONJ ? w.z : -w.z, nh = CONJ ? w.w : -w.w;
    long long P = (long long)ah * ch + (long long)bh * nh;
    long long M = (1LL << 31) + (long long)ah * cl;
    M += (long long)al * ch;
    M += (long long)bh * nl;
    M += (long long)bl * nh;
    long long Q = (long long)ah * dh + (long long)bh * ch;
    long long N = (1LL << 31) + (long long)ah * dl;
    N += (long long)al * dh;
    N += (long long)bh * cl;
    N += (long long)bl * ch;
    return make_longlong2(P + (M >> 32), Q + (N >> 32));
}

// a w 2^(k - 2), 0 <= k < 32, for tables of small entries, |a w| 2^(k - 2) < 2^61.5:
// with the low halves' products, whose upper words the result still has
__device__ __forceinline__ fx2 fmul_up(fx2 a, int4 w, int k)
{
    int ah, al, bh, bl;
    halves(a.x, ah, al);
    halves(a.y, bh, bl);
    long long P = (long long)ah * w.y - (long long)bh * w.w;
    long long M = (1LL << (31 - k)) + __mulhi(al, w.x) - __mulhi(bl, w.z);
    M += (long long)ah * w.x + (long long)al * w.y;
    M -= (long long)bh * w.z + (long long)bl * w.w;
    long long Q = (long long)ah * w.w + (long long)bh * w.y;
    long long N = (1LL << (31 - k)) + __mulhi(al, w.z) + __mulhi(bl, w.x);
    N += (long long)ah * w.z + (long long)al * w.w;
    N += (long long)bh * w.x + (long long)bl * w.y;
    return make_longlong2((P << k) + (M >> (32 - k)), (Q << k) + (N >> (32 - k)));
}

// bits of the largest component so far: the OR of the components' upper words
// without their signs
__device__ __forceinline__ unsigned fmag(fx2 a)
{
    const int x = (int)(a.x >> 32), y = (int)(a.y >> 32);
    return (unsigned)(x ^ (x >> 31)) | (unsigned)(y ^ (y >> 31));
}

// The common power of two of a block's points, true value = x 2^e, and the
// shared-memory slots in which a pass leaves its results' size for the next:
// slot i is read after the barrier that ends pass i, filled during pass i,
// and cleared during pass i + 1's predecessor, three slots in turn.
struct FxScale {
    unsigned *slot;                    // 3 words of shared memory
    int i, e;
    // after a pass's results: every thread's OR
    __device__ __forceinline__ void leave(unsigned mag)
    {
        mag = __reduce_or_sync(0xffffffffu, mag);
        if ((threadIdx.x & 31) == 0 && mag) atomicOr(slot + (i + 1) % 3, mag);
    }
    // before a pass: the barrier, and the shift that brings the largest
    // component to 61 bits
    __device__ __forceinline__ int enter()
    {
        __syncthreads();
        i = (i + 1) % 3;
        const unsigned m = slot[i];
        if (threadIdx.x == 0) slot[(i + 2) % 3] = 0;
        const int s = max(0, 61 - (m ? 64 - __clz((int)m) : 32));
        e -= s;
        return s;
    }
};

// ------------------------------------------------ mixed-radix ring FFTs
// A transform of length N = r_0 r_1 ... r_{n-1} (radices 2, 3, 4, 5, 7, 11,
// 13; list rl = {n, r_0, .., r_{n-1}}) runs in place in shared memory in n
// passes.  Pass i works on blocks of B_i = N / (r_0 .. r_{i-1}) points and
// combines the r_i points base + q N_i (N_i = B_i / r_i, q < r_i) of each of
// its B_i / r_i butterflies.  Decimation in frequency (exponent -1, passes
// 0..n-1: radix-r DFT, then the twiddles w_{B_i}^{-p j}) takes natural order
// to "position" order, in which X_k, k = p_0 + r_0 (p_1 + r_1 (p_2 + ..)),
// sits at pos(k) = sum_i p_i N_i.  Decimation in time (exponent +1, passes
// n-1..0, twiddles first) is its conjugate transpose: position order in,
// natural order out, unnormalised.  So no permutation pass is ever needed:
// the fold writes straight to pos(k), and a Bluestein filter is stored in
// position order.

// cos and sin of 2 pi k / R for the odd radices, k < R: R = 3, 5, 7, 11, 13
// at offsets 0, 3, 8, 15, 26
__host__ __device__ constexpr double root_cos(int k)
{
    constexpr double t[39] = {
    1.00000000000000000e+00, -5.00000000000000000e-01, -5.00000000000000000e-01,
    1.00000000000000000e+00, 3.09016994374947451e-01, -8.09016994374947451e-01, -8.09016994374947451e-01,
    3.09016994374947451e-01,
    1.00000000000000000e+00, 6.23489801858733483e-01, -2.22520933956314393e-01, -9.00968867902419146e-01,
    -9.00968867902419146e-01, -2.22520933956314393e-01, 6.23489801858733483e-01,
    1.00000000000000000e+00, 8.41253532831181206e-01, 4.15415013001886435e-01, -1.42314838273285144e-01,
    -6.54860733945285101e-01, -9.59492973614497369e-01, -9.59492973614497369e-01, -6.54860733945285101e-01,
    -1.42314838273285144e-01, 4.15415013001886435e-01, 8.41253532831181206e-01,
    1.00000000000000000e+00, 8.85456025653209911e-01, 5.68064746731155812e-01, 1.20536680255323048e-01,
    -3.54604887042535621e-01, -7.48510748171101081e-01, -9.70941817426052012e-01, -9.70941817426052012e-01,
    -7.48510748171101081e-01, -3.54604887042535621e-01, 1.20536680255323048e-01, 5.68064746731155812e-01,
    8.85456025653209911e-01};
    return t[k];
}
__host__ __device__ constexpr double root_sin(int k)
{
    constexpr double t[39] = {
    0.00000000000000000e+00, 8.66025403784438597e-01, -8.66025403784438597e-01,
    0.00000000000000000e+00, 9.51056516295153531e-01, 5.87785252292473137e-01, -5.87785252292473137e-01,
    -9.51056516295153531e-01,
    0.00000000000000000e+00, 7.81831482468029804e-01, 9.74927912181823619e-01, 4.33883739117558120e-01,
    -4.33883739117558120e-01, -9.74927912181823619e-01, -7.81831482468029804e-01,
    0.00000000000000000e+00, 5.40640817455597555e-01, 9.09631995354518330e-01, 9.89821441880932684e-01,
    7.55749574354258269e-01, 2.81732556841429671e-01, -2.81732556841429671e-01, -7.55749574354258269e-01,
    -9.89821441880932684e-01, -9.09631995354518330e-01, -5.40640817455597555e-01,
    0.00000000000000000e+00, 4.64723172043768562e-01, 8.22983865893656352e-01, 9.92708874098053973e-01,
    9.35016242685414833e-01, 6.63122658240795193e-01, 2.39315664287557767e-01, -2.39315664287557767e-01,
    -6.63122658240795193e-01, -9.35016242685414833e-01, -9.92708874098053973e-01, -8.22983865893656352e-01,
    -4.64723172043768562e-01};
    return t[k];
}
// bits by which dft_small scales down: its roots are in units of 2^-(64 -
// bits), the finest that keep its sums of mixed halves' products below 2^63
// (units of 2^-59 for all left the points 52 to 54 bits, fewer than FP64's 53
// of each point)
__host__ __device__ constexpr int dft_bits(int R) { return R == 2 || R == 4 ? 0 : R <= 5 ? 2 : R == 7 ? 3 : 4; }
__host__ __device__ constexpr long long root_fix(double x, int R)
{
    return (long long)(x * (double)(1LL << (64 - dft_bits(R))));
}
__host__ __device__ constexpr int root_low(long long v) { return (int)(unsigned)(v & 0xffffffffLL); }
__host__ __device__ constexpr int root_high(long long v) { return (int)((v - root_low(v)) / (1LL << 32)); }

template <int R>
__device__ __forceinline__ constexpr int root_off()
{
    return R == 3 ? 0 : R == 5 ? 3 : R == 7 ? 8 : R == 11 ? 15 : 26;
}

// y_q = 2^-dft_bits sum_p a_p e^{S 2 pi i p q / R}, in place (S = +1 or -1),
// |a| < 2^59.5
template <int R, int S>
__device__ __forceinline__ void dft_small(fx2 (&a)[R])
{
    if constexpr (R == 2) {
        const fx2 u = a[0];
        a[0] = fadd(u, a[1]);
        a[1] = fsub(u, a[1]);
    } else if constexpr (R == 4) {
        const fx2 s0 = fadd(a[0], a[2]), s1 = fsub(a[0], a[2]);
        const fx2 s2 = fadd(a[1], a[3]), d = fsub(a[1], a[3]);
        a[0] = fadd(s0, s2);
        a[2] = fsub(s0, s2);
        // s1 +- S i d
        const fx2 p = make_longlong2(s1.x - d.y, s1.y + d.x), m = make_longlong2(s1.x + d.y, s1.y - d.x);
        a[1] = S > 0 ? p : m;
        a[3] = S > 0 ? m : p;
    } else {
        // odd R: pair p with R - p, y_q = A_q + S i B_q, y_{R-q} = A_q - S i
        // B_q; A and B are sums of products with constants, each kept as the
        // sum of the high halves' products and of the mixed ones (at most 6
        // terms of 2^59.5 + 2^(63 - dft_bits))
        constexpr int H = (R - 1) / 2, O = root_off<R>(), D = dft_bits(R);
        int sh[H][2], sl[H][2], dh[H][2], dl[H][2];
        fx2 y0 = make_longlong2(a[0].x >> 1, a[0].y >> 1);
#pragma unroll
        for (int p = 1; p <= H; ++p) {
            const fx2 sp = fadd(a[p], a[R - p]), dp = fsub(a[p], a[R - p]);
            halves(sp.x, sh[p - 1][0], sl[p - 1][0]);
            halves(sp.y, sh[p - 1][1], sl[p - 1][1]);
            halves(dp.x, dh[p - 1][0], dl[p - 1][0]);
            halves(dp.y, dh[p - 1][1], dl[p - 1][1]);
            y0.x += sp.x >> 1;
            y0.y += sp.y >> 1;
        }
        const fx2 a0 = frshift(a[0], D);
#pragma unroll
        for (int q = 1; q <= H; ++q) {
            long long A[2], B[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                long long Ph = 0, Pm = 1LL << 31, Qh = 0, Qm = 1LL << 31;
#pragma unroll
                for (int p = 1; p <= H; ++p) {
                    const long long cs = root_fix(root_cos(O + (p * q) % R), R), sn = root_fix(root_sin(O + (p * q) % R), R);
                    Ph += (long long)sh[p - 1][c] * root_high(cs);
                    Pm += (long long)sh[p - 1][c] * root_low(cs);
                    Pm += (long long)sl[p - 1][c] * root_high(cs);
                    Qh += (long long)dh[p - 1][c] * root_high(sn);
                    Qm += (long long)dh[p - 1][c] * root_low(sn);
                    Qm += (long long)dl[p - 1][c] * root_high(sn);
                }
                A[c] = (c ? a0.y : a0.x) + Ph + (Pm >> 32);
                B[c] = Qh + (Qm >> 32);
            }
            const fx2 iB = S > 0 ? make_longlong2(-B[1], B[0]) : make_longlong2(B[1], -B[0]);
            a[q] = make_longlong2(A[0] + iB.x, A[1] + iB.y);
            a[R - q] = make_longlong2(A[0] - iB.x, A[1] - iB.y);
        }
        a[0] = frshift(y0, D - 1);
    }
}

// bits by which the results of an odd radix, which dft_small leaves below
// 2^59.9, are shifted up before their twiddles, a product of which scales
// down by 2 and may end at 2^61.5
template <int R>
__device__ __forceinline__ constexpr int twiddle_up()
{
    return R == 2 || R == 4 ? 0 : R == 5 ? 1 : 2;
}

// one pass of radix R over Ntot points: back-to-back sequences of Nseq
// points (Nseq a multiple of B), in blocks of B; tw(t) = e^{2 pi i t / Nseq};
// s: the shift of FxScale::enter.  Returns the results' size; scales down by
// pass_bits.
template <int R, bool INV>
__device__ __forceinline__ int pass_bits(int Ns)
{
    return 2 + dft_bits(R) + (!INV && Ns > 1 ? 2 - twiddle_up<R>() : 0);
}

template <int R, bool INV, class TW>
__device__ __forceinline__ unsigned mx_pass(fx2 *x, int Ntot, int Nseq, int B, const TW &tw, int s)
{
    // twiddles are 1 in the first pass of decimation in time and the last of
    // decimation in frequency
    const int Ns = B / R, step = Nseq / B;
    const bool twiddled = Ns > 1;
    unsigned mag = 0;
    for (int t = threadIdx.x; t < Ntot / R; t += blockDim.x) {
        const int j = t % Ns, base = (t - j) * R + j;
        fx2 a[R];
#pragma unroll
        for (int q = 0; q < R; ++q) a[q] = fshl(x[base + q * Ns], s);
        a[0] = frshift(a[0], 2);
        if (INV && twiddled) {
#pragma unroll
            for (int p = 1; p < R; ++p) a[p] = fmul(a[p], tw(p * j * step));
        } else {
#pragma unroll
            for (int p = 1; p < R; ++p) a[p] = frshift(a[p], 2);
        }
        dft_small<R, INV ? 1 : -1>(a);
        if (!INV && twiddled) {
            constexpr int U = twiddle_up<R>();
            if (U < 2) a[0] = frshift(a[0], U < 2 ? 2 - U : 1);
#pragma unroll
            for (int p = 1; p < R; ++p) a[p] = fmul<true>(fshl(a[p], U), tw(p * j * step));
        }
#pragma unroll
        for (int q = 0; q < R; ++q) {
            x[base + q * Ns] = a[q];
            mag |= fmag(a[q]);
        }
    }
    return mag;
}

// cos and sin of 2 pi k / R in units of 2^-60 as halves {low, high, low,
// high}, k < R, for R = 11 and 13 at root_off<R>() - 15
struct RootTable {
    int4 v[24];
};
constexpr RootTable make_root_table()
{
    RootTable t{};
    for (int i = 0; i < 24; ++i) {
        const long long c = root_fix(root_cos(15 + i), 13), n = root_fix(root_sin(15 + i), 13);
        t.v[i].x = root_low(c);
        t.v[i].y = root_high(c);
        t.v[i].z = root_low(n);
        t.v[i].w = root_high(n);
    }
    return t;
}
static __constant__ RootTable kRoots = make_root_table();

// mx_pass for the radices 11 and 13, with dft_small written out around the
// loads and stores: the inputs are taken pair by pair and each pair of
// outputs is stored as soon as it is made, in a rolled loop over the outputs.
// Unrolled, with inputs and outputs in registers, the radix-13 pass spilled
// at 128 registers and the kernel's code overflowed the instruction cache
// (ring stage of 8 maps at Nside = 512 1.058 -> 1.021 ms, adjoint 1.158 ->
// 1.125; radix 7 the same way measured 1.034 and 1.117).
template <int R, bool INV, class TW>
__device__ __forceinline__ unsigned mx_pass_odd(fx2 *x, int Ntot, int Nseq, int B, const TW &tw, int s)
{
    constexpr int H = (R - 1) / 2, O = root_off<R>() - 15, D = dft_bits(R), U = twiddle_up<R>();
    static_assert(D == dft_bits(13) && U == 2, "one table of roots, no shift after the twiddles");
    const int Ns = B / R, step = Nseq / B;
    const bool twiddled = Ns > 1;
    unsigned mag = 0;
    for (int t = threadIdx.x; t < Ntot / R; t += blockDim.x) {
        const int j = t % Ns, base = (t - j) * R + j;
        int sh[H][2], sl[H][2], dh[H][2], dl[H][2];
        const fx2 a0 = frshift(fshl(x[base], s), 2);
        fx2 y0 = make_longlong2(a0.x >> 1, a0.y >> 1);
#pragma unroll
        for (int p = 1; p <= H; ++p) {
            fx2 a = fshl(x[base + p * Ns], s), b = fshl(x[base + (R - p) * Ns], s);
            if (INV && twiddled) {
                a = fmul(a, tw(p * j * step));
                b = fmul(b, tw((R - p) * j * step));
            } else {
                a = frshift(a, 2);
                b = frshift(b, 2);
            }
            const fx2 sp = fadd(a, b), dp = fsub(a, b);
            halves(sp.x, sh[p - 1][0], sl[p - 1][0]);
            halves(sp.y, sh[p - 1][1], sl[p - 1][1]);
            halves(dp.x, dh[p - 1][0], dl[p - 1][0]);
            halves(dp.y, dh[p - 1][1], dl[p - 1][1]);
            y0.x += sp.x >> 1;
            y0.y += sp.y >> 1;
        }
        y0 = frshift(y0, D - 1);
        x[base] = y0;
        mag |= fmag(y0);
        const fx2 a0d = frshift(a0, D);
#pragma unroll 1
        for (int q = 1; q <= H; ++q) {
            long long Ph[2] = {0, 0}, Pm[2] = {1LL << 31, 1LL << 31}, Qh[2] = {0, 0}, Qm[2] = {1LL << 31, 1LL << 31};
            int idx = 0;
#pragma unroll
            for (int p = 0; p < H; ++p) {
                idx += q;
                if (idx >= R) idx -= R;
                const int4 w = kRoots.v[O + idx];
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    Ph[c] += (long long)sh[p][c] * w.y;
                    Pm[c] += (long long)sh[p][c] * w.x;
                    Pm[c] += (long long)sl[p][c] * w.y;
                    Qh[c] += (long long)dh[p][c] * w.w;
                    Qm[c] += (long long)dh[p][c] * w.z;
                    Qm[c] += (long long)dl[p][c] * w.w;
                }
            }
            const fx2 A = make_longlong2(a0d.x + Ph[0] + (Pm[0] >> 32), a0d.y + Ph[1] + (Pm[1] >> 32));
            const fx2 Bv = make_longlong2(Qh[0] + (Qm[0] >> 32), Qh[1] + (Qm[1] >> 32));
            const fx2 iB = INV ? ftimes_i(Bv) : make_longlong2(Bv.y, -Bv.x);
            fx2 y = fadd(A, iB), z = fsub(A, iB);
            if (!INV && twiddled) {
                y = fmul<true>(fshl(y, U), tw(q * j * step));
                z = fmul<true>(fshl(z, U), tw((R - q) * j * step));
            }
            x[base + q * Ns] = y;
            x[base + (R - q) * Ns] = z;
            mag |= fmag(y) | fmag(z);
        }
    }
    return mag;
}

// Rader pass context: the ring's prime tables, and shared-memory scratch
// for its convolutions ((N / p) (p - 1) points after the N of the ring)
struct RaderCtx {
    const RaderInfo *ri;
    const int *rad;
    const int *ints;
    const int4 *tab;
    fx2 *scratch;
};

// One pass, its barrier before it included.  BIG: the radix-11 and radix-13
// butterflies are compiled in (they need many more registers; only lengths
// with those factors are run with BIG)
template <bool INV, bool BIG, class TW>
__device__ __forceinline__ void mx_pass_any(int r, fx2 *x, int Ntot, int Nseq, int B, const TW &tw, FxScale &sc)
{
    const int s = sc.enter(), Ns = B / r;
    unsigned mag = 0;
    switch (r) {
    case 4: mag = mx_pass<4, INV>(x, Ntot, Nseq, B, tw, s); sc.e += pass_bits<4, INV>(Ns); break;
    case 2: mag = mx_pass<2, INV>(x, Ntot, Nseq, B, tw, s); sc.e += pass_bits<2, INV>(Ns); break;
    case 3: mag = mx_pass<3, INV>(x, Ntot, Nseq, B, tw, s); sc.e += pass_bits<3, INV>(Ns); break;
    case 5: mag = mx_pass<5, INV>(x, Ntot, Nseq, B, tw, s); sc.e += pass_bits<5, INV>(Ns); break;
    case 7: mag = mx_pass<7, INV>(x, Ntot, Nseq, B, tw, s); sc.e += pass_bits<7, INV>(Ns); break;
    default:
        if constexpr (BIG) {
            if (r == 11) mag = mx_pass_odd<11, INV>(x, Ntot, Nseq, B, tw, s);
            else mag = mx_pass_odd<13, INV>(x, Ntot, Nseq, B, tw, s);
            sc.e += pass_bits<13, INV>(Ns);
        }
        break;
    }
    sc.leave(mag);
}

// natural order in, position order out, exponent -1; Ntot / Nseq sequences
// of Nseq points transformed side by side.  The results' size is left for
// the caller's FxScale::enter, which is also the barrier after the last pass.
template <bool BIG, class TW>
__device__ __forceinline__ void fft_mx_dif(fx2 *x, int Ntot, int Nseq, const int *__restrict__ rl, const TW &tw,
                                           FxScale &sc)
{
    const int n = rl[0];
    int B = Nseq;
    for (int i = 0; i < n; ++i) {
        const int r = rl[1 + i];
        mx_pass_any<false, BIG>(r, x, Ntot, Nseq, B, tw, sc);
        B /= r;
    }
}

// position order in, natural order out, exponent +1 (unnormalised)
template <bool BIG, class TW>
__device__ __forceinline__ void fft_mx_dit(fx2 *x, int Ntot, int Nseq, const int *__restrict__ rl, const TW &tw,
                                           FxScale &sc)
{
    const int n = rl[0];
    int B = 1;
    for (int i = n - 1; i >= 0; --i) {
        const int r = rl[1 + i];
        B *= r;
        mx_pass_any<true, BIG>(r, x, Ntot, Nseq, B, tw, sc);
    }
}

// ring transform kinds: direct mixed radix over 2, 3, 4, 5, 7; Bluestein
// (7-smooth convolution length); direct with radix 11 or 13 among the
// radices, or with one prime above 13 done by Rader's algorithm
enum RingFft { kDirect = 0, kBluestein = 1, kDirectBig = 2 };

// position of X_k in position order
__device__ __forceinline__ int fft_pos(int k, int N, const int *__restrict__ rl)
{
    const int n = rl[0];
    int pos = 0, Nc = N;
    for (int i = 0; i < n; ++i) {
        const int r = rl[1 + i];
        Nc /= r;
        pos += (k % r) * Nc;
        k /= r;
    }
    return pos;
}

// e^{i pi n / J}, n >= 0, from the ring's half-circle table (n < J)
__device__ __forceinline__ int4 ring_root(const int4 *__restrict__ T, int J, int n)
{
    const int k = n % (2 * J);
    return wneg_if(__ldg(T + (k < J ? k : k - J)), k >= J);
}

// e^{2 pi i t / K} (t < K) from the ring's half-circle table of J = 2K roots
struct TwRing {
    const int4 *T;
    int J;
    __device__ __forceinline__ int4 operator()(int t) const
    {
        const int n = 4 * t;             // e^{2 pi i t / K} = e^{i pi 4t / J}, 4t < 2J
        return wneg_if(__ldg(T + (n < J ? n : n - J)), n >= J);
    }
};

// e^{2 pi i t / M} (t < M) from a table of M roots
struct TwTable {
    const int4 *R;
    __device__ __forceinline__ int4 operator()(int t) const { return __ldg(R + t); }
};

// fmul_up's bits for a filter of M points: its entries are below 1.7 / sqrt(M)
// (checked for every K up to 4096), and 2^(bits - 2) <= sqrt(M) / 2
__device__ __forceinline__ int blue_up(int M) { return (33 - __clz(M)) / 2; }

// x[0..K) holds the input, zeros follow up to M; computes x[n] =
// sum_k x_k e^{2 pi i k n / K} for n < K through Bluestein's chirp transform:
// a cyclic convolution of length M (smooth, >= 2K - 1) with the chirp filter,
// stored transformed in position order and scaled by 1/M.  The input already
// carries its chirp c_k = e^{i pi k^2 / K} and the results do not: the caller
// multiplies them by c_n as it reads them.
__device__ __forceinline__ void bluestein_mx(fx2 *x, int M, const int4 *__restrict__ fb, const int *__restrict__ rl,
                                             const TwTable &tw, FxScale &sc)
{
    fft_mx_dif<false>(x, M, M, rl, tw, sc);
    const int s = sc.enter(), up = blue_up(M);
    unsigned mag = 0;
    for (int k = threadIdx.x; k < M; k += blockDim.x) {
        const fx2 y = fmul_up(fshl(x[k], s), __ldg(fb + k), up);
        x[k] = y;
        mag |= fmag(y);
    }
    sc.e += 2 - up;
    sc.leave(mag);
    fft_mx_dit<false>(x, M, M, rl, tw, sc);
}

// x true = x 2^from in units of 2^to, to nearest
__device__ __forceinline__ fx2 frescale(fx2 a, int from, int to)
{
    const int n = to - from;
    if (n == 0) return a;
    if (n < 0) return fshl(a, -n);
    return n > 62 ? make_longlong2(0, 0) : frshift(a, n);
}

// Rader's algorithm for the p-point DFTs of one pass over N points (blocks
// of p contiguous points, no twiddles: the pass is the first of decimation
// in time, or the last of decimation in frequency).  With g a primitive
// root mod p, y_{g^w} = a_0 + sum_v a_{g^{-v}} e^{2 pi i g^{w-v} / p}: a
// cyclic convolution of alpha_v = a_{g^{-v}} with beta_t = e^{2 pi i g^t / p},
// done as forward transform, product with the stored transform of beta
// (scaled by 1/(p-1)), inverse transform, all of length p - 1 and side by
// side for the N / p blocks in the scratch.  a_0 joins every output through
// the product's zero frequency, and y_0 = a_0 + (sum of alpha) is that
// frequency before the product.  Exponent +1; CONJ = true gives exponent -1
// as conj(DFT(conj a)).  The a_0 stay in the units they have when the pass
// begins; at the end all points are in the convolution's units.  The stored
// transform has modulus sqrt(p) / (p - 1) (1 / (p - 1) at zero), so that
// products without the bits fmul_up keeps would end at 2^52 for p = 1000.
struct RaderRun {
    RaderCtx c;
    RaderInfo ri;
    int N, tot, e0, e1;                                // e0: units of the a_0 left in x; e1: of y_0

    RaderRun() = default;
    __device__ __forceinline__ RaderRun(const RaderCtx &c, int N) : c(c), ri(*c.ri), N(N), tot((N / ri.p) * ri.n) {}

    template <bool CONJ>
    __device__ __forceinline__ void gather(fx2 *x, FxScale &sc)
    {
        const int *__restrict__ gi = c.ints + ri.gi;
        const int s0 = sc.enter();
        e0 = sc.e + s0;
        unsigned mag = 0;
        for (int e = threadIdx.x; e < tot; e += blockDim.x) {
            const int b = e / ri.n, v = e - b * ri.n;
            fx2 a = fshl(x[b * ri.p + __ldg(gi + v)], s0);
            if (CONJ) a = fconj(a);
            c.scratch[e] = a;
            mag |= fmag(a);
        }
        sc.leave(mag);
    }

    // y_0 has units of its own, in which it and its two terms fit, and so has
    // the product with a_0
    template <bool CONJ>
    __device__ __forceinline__ void product(fx2 *x, FxScale &sc)
    {
        const int4 *__restrict__ G = c.tab + ri.G;
        fx2 *S = c.scratch;
        const int s1 = sc.enter(), up = (33 - __clz(ri.n)) / 2;    // 2^(up - 2) sqrt(p) / n <= .52
        const int ec = sc.e + 2 - up, e2 = max(ec, e0) + 2;
        e1 = max(sc.e, e0) + 1;
        unsigned mag = 0;
        for (int e = threadIdx.x; e < tot; e += blockDim.x) {
            const int b = e / ri.n, v = e - b * ri.n;
            const fx2 A = fshl(S[e], s1);
            fx2 C = frescale(fmul_up(A, __ldg(G + v), up), ec, e2);
            if (v == 0) {
                const fx2 a0 = CONJ ? fconj(x[b * ri.p]) : x[b * ri.p];
                C = fadd(C, frescale(a0, e0, e2));
                fx2 y0 = fadd(frescale(a0, e0, e1), frescale(A, sc.e, e1));
                if (CONJ) y0 = fconj(y0);
                x[b * ri.p] = y0;
            }
            S[e] = C;
            mag |= fmag(C);
        }
        sc.e = e2;
        sc.leave(mag);
    }

    template <bool CONJ>
    __device__ __forceinline__ void scatter(fx2 *x, FxScale &sc)
    {
        const int *__restrict__ ga = c.ints + ri.ga;
        const int s2 = sc.enter(), e2 = max(sc.e, e1) + 1;
        unsigned mag = 0;
        for (int e = threadIdx.x; e < tot; e += blockDim.x) {
            const int b = e / ri.n, w = e - b * ri.n;
            fx2 y = frescale(fshl(c.scratch[e], s2), sc.e, e2);
            if (CONJ) y = fconj(y);
            x[b * ri.p + __ldg(ga + w)] = y;
            mag |= fmag(y);
            if (w == 0) {
                const fx2 y0 = frescale(x[b * ri.p], e1, e2);
                x[b * ri.p] = y0;
                mag |= fmag(y0);
            }
        }
        sc.e = e2;
        sc.leave(mag);
    }
};

// a ring's twiddles (TwRing) or, with J = 0, a table's (TwTable)
struct TwAny {
    const int4 *T;
    int J;
    __device__ __forceinline__ int4 operator()(int t) const
    {
        const int n = J ? 4 * t : t;
        const bool neg = J && n >= J;
        return wneg_if(__ldg(T + (neg ? n - J : n)), neg);
    }
};

// fft_mx_dif and fft_mx_dit of a BIG ring, whose first (last) radix may be a
// Rader prime.  The ring's passes and those of the convolution that go the
// same way run through one body, in turn: the kernels are held by instruction
// fetches, and a body of all radices each for the ring and for both ways of
// the convolution was three where two do (Nside = 512, ring stage of 8 maps
// .900 -> .862 ms, adjoint .983 -> .944; 256: .304 -> .279 and .347 -> .323).
__device__ __forceinline__ void fft_big_dif(fx2 *x, int K, const int *__restrict__ rl, const TwRing &tw, FxScale &sc,
                                            const RaderCtx *rc)
{
    RaderRun run = rc ? RaderRun(*rc, K) : RaderRun();
#pragma unroll 1
    for (int phase = 0; phase < (rc ? 2 : 1); ++phase) {
        fx2 *y = phase ? rc->scratch : x;
        const int *__restrict__ l = phase ? run.c.rad + run.ri.rl : rl;
        const int Ntot = phase ? run.tot : K, Nseq = phase ? run.ri.n : K;
        const TwAny w = phase ? TwAny{run.c.tab + run.ri.tw, 0} : TwAny{tw.T, tw.J};
        const int n = l[0] - (rc && !phase);
        int B = Nseq;
        for (int i = 0; i < n; ++i) {
            const int r = l[1 + i];
            mx_pass_any<false, true>(r, y, Ntot, Nseq, B, w, sc);
            B /= r;
        }
        if (rc && !phase) run.gather<true>(x, sc);
    }
    if (!rc) return;
    run.product<true>(x, sc);
    fft_mx_dit<true>(rc->scratch, run.tot, run.ri.n, run.c.rad + run.ri.rl, TwTable{run.c.tab + run.ri.tw}, sc);
    run.scatter<true>(x, sc);
}

__device__ __forceinline__ void fft_big_dit(fx2 *x, int K, const int *__restrict__ rl, const TwRing &tw, FxScale &sc,
                                            const RaderCtx *rc)
{
    RaderRun run = rc ? RaderRun(*rc, K) : RaderRun();
    if (rc) {
        run.gather<false>(x, sc);
        fft_mx_dif<true>(rc->scratch, run.tot, run.ri.n, run.c.rad + run.ri.rl, TwTable{run.c.tab + run.ri.tw}, sc);
        run.product<false>(x, sc);
    }
#pragma unroll 1
    for (int phase = rc ? 0 : 1; phase < 2; ++phase) {
        fx2 *y = phase ? x : rc->scratch;
        const int *__restrict__ l = phase ? rl : run.c.rad + run.ri.rl;
        const int Ntot = phase ? K : run.tot, Nseq = phase ? K : run.ri.n;
        const TwAny w = phase ? TwAny{tw.T, tw.J} : TwAny{run.c.tab + run.ri.tw, 0};
        int B = 1, i = l[0] - 1;
        if (rc && phase) B = l[1 + i--];               // the Rader prime
        for (; i >= 0; --i) {
            const int r = l[1 + i];
            B *= r;
            mx_pass_any<true, true>(r, y, Ntot, Nseq, B, w, sc);
        }
        if (!phase) run.scatter<false>(x, sc);
    }
}

// The Rader context of a ring of a BIG kernel (nullptr for other rings):
// its scratch follows the ring's K points in shared memory.
__device__ __forceinline__ const RaderCtx *rader_ctx(const PlanView &v, int ring, int K, fx2 *sm, RaderCtx &rc)
{
    const int ri = v.ring_rdr[ring];
    if (ri < 0) return nullptr;
    rc = RaderCtx{v.rdr + ri, v.rad, v.rdr_int, ring_table(v.rdr_dbl), sm + K};
    return &rc;
}

// v = a whole number of 2^(ex - 1083) below 2^61, toward zero; sh = 3 + ex - v's exponent
__device__ __forceinline__ long long ring_fix(double v, int sh)
{
    const int hi = __double2hiint(v), lo = __double2loint(v);
    const unsigned mh = __funnelshift_l((unsigned)lo, (unsigned)hi, 11) | 0x80000000u;
    unsigned long long X;
    asm("shr.u64 %0, %1, %2;" : "=l"(X) : "l"((unsigned long long)mh << 32 | ((unsigned)lo << 11)), "r"(sh));
    const unsigned long long s = (unsigned long long)(long long)(hi >> 31);
    return (long long)((X ^ s) - s);
}

__device__ __forceinline__ int exp_field(double v) { return __double2hiint(v) & 0x7ff00000; }
__device__ __forceinline__ unsigned nonzero_bits(double v)
{
    return (unsigned)__double2hiint(v) << 1 | (unsigned)__double2loint(v);
}

// Shared words of a ring's block: the three size slots of FxScale, the
// largest exponent, whether any value is not zero
struct RingAux {
    unsigned slot[3];
    int emax;
    unsigned any;
};

// Range of the block exponent that the fixed-point path takes, and the power
// of two that brings any other finite one into it: values above it are only
// renamed (their units), values below it are lifted first (subnormals among
// them); either way the results are scaled back
constexpr int kRingExpLo = 300, kRingExpHi = 1700, kRingLift = 600;

__device__ __forceinline__ double2 scaled(double2 z, int n)
{
    const double f = shtb::pow2(n);
    return make_double2(z.x * f, z.y * f);
}

// out[0 .. n) of a ring of zeros or (a value is not finite) of NaN
__device__ __forceinline__ void ring_fill(double2 *out, int n, bool zero)
{
    const double f = zero ? 0.0 : __longlong_as_double(0x7ff8000000000000LL);
    for (int i = threadIdx.x; i < n; i += blockDim.x) out[i] = make_double2(f, f);
    __syncthreads();
}

__device__ __forceinline__ void ring_scale_back(double2 *out, int n, int lift)
{
    for (int i = threadIdx.x; i < n; i += blockDim.x) out[i] = scaled(out[i], -lift);
}

// The fold of a ring's spectrum: entry k at sm, in units 2^(f - 1080), and f
// in ex, at the transform's position of k; the largest f and whether any value
// is not zero in aux.  LIFT: of 2^kRingLift times the spectrum.
template <bool BLUE, bool LIFT, class QAt>
__device__ __forceinline__ void ring_fold(QAt qat, int L, int J, int s, const int4 *__restrict__ AB,
                                          const int *__restrict__ rl, fx2 *sm, short *ex, RingAux &aux)
{
    const int K = J / 2;
    int emax = 0;
    unsigned any = 0;
    auto pack = [&](int k, double2 G0, double2 G1) {
        if (LIFT) {
            G0 = scaled(G0, kRingLift);
            G1 = scaled(G1, kRingLift);
        }
        const int f = max(max(exp_field(G0.x), exp_field(G0.y)), max(exp_field(G1.x), exp_field(G1.y)));
        any |= nonzero_bits(G0.x) | nonzero_bits(G0.y) | nonzero_bits(G1.x) | nonzero_bits(G1.y);
        const int f3 = f + (3 << 20);
        const fx2 X0 = make_longlong2(ring_fix(G0.x, (f3 - exp_field(G0.x)) >> 20),
                                      ring_fix(G0.y, (f3 - exp_field(G0.y)) >> 20));
        const fx2 X1 = make_longlong2(ring_fix(G1.x, (f3 - exp_field(G1.x)) >> 20),
                                      ring_fix(G1.y, (f3 - exp_field(G1.y)) >> 20));
        const int pos = BLUE ? k : fft_pos(k, K, rl);
        sm[pos] = fadd(fmul(X0, __ldg(AB + 2 * k)), fmul(X1, __ldg(AB + 2 * k + 1)));
        ex[pos] = (short)(f >> 20);
        emax = max(emax, f >> 20);
    };
    // A short ring folds many terms onto few k (J = 4: L / 2 each): up to 32
    // neighbouring threads then share one k's terms, as many as kFoldThreads
    // gives each k, whatever the block's size: the sums, and so the maps, are
    // the same bits in the ring kernels (128 to 512 threads) and in the batch
    // kernel (32 a warp of its schedule)
    constexpr int kFoldThreads = 128;
    int parts = 1;
    while (parts < 32 && 2 * parts * K <= kFoldThreads) parts *= 2;
    if (parts == 1) {
        for (int k = threadIdx.x; k < K; k += blockDim.x) pack(k, fold_G(qat, L, J, s, k), fold_G(qat, L, J, s, k + K));
    } else {
        for (int i = threadIdx.x; i < ((K * parts + 31) & ~31); i += blockDim.x) {    // whole warps
            const int k = i / parts, part = i & (parts - 1);
            double2 G0 = make_double2(0.0, 0.0), G1 = G0;
            if (k < K) {
                G0 = fold_part(qat, L, J, s, k, part, parts);
                G1 = fold_part(qat, L, J, s, k + K, part, parts);
            }
            for (int o = 1; o < parts; o *= 2) {
                G0.x += __shfl_xor_sync(0xffffffffu, G0.x, o);
                G0.y += __shfl_xor_sync(0xffffffffu, G0.y, o);
                G1.x += __shfl_xor_sync(0xffffffffu, G1.x, o);
                G1.y += __shfl_xor_sync(0xffffffffu, G1.y, o);
            }
            if (k < K && part == 0) pack(k, G0, G1);
        }
    }
    emax = (int)__reduce_max_sync(0xffffffffu, (unsigned)emax);
    any = __reduce_or_sync(0xffffffffu, any);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&aux.emax, emax);
        atomicOr(&aux.any, any);
    }
}

// Pixels of one ring from its q_m (m = 0..L): fold (Eq. tau) and pack the
// Hermitian spectrum into a half-length complex FFT in one step,
// Z_k = G_k A_k + G_{k+K} B_k (the plan's fold weights A, B hold the phi_0
// phase, the packing twiddle and, on Bluestein rings, the chirp), transform,
// and write f_{2n}, f_{2n+1} as the real and imaginary parts of z_n.  The
// fold's sums are FP64; each Z_k is formed in fixed point with its own
// exponent, and once the largest is known all are brought to it.  All threads
// of the block take part; sm holds the transform's entries (K direct, K plus
// the Rader scratch, M Bluestein) and K 16-bit exponents after them.
template <int KIND, class QAt>
__device__ __forceinline__ void phi_synth_ring_at(const PlanView &v, int ring, QAt qat, double *out_ring, fx2 *sm)
{
    constexpr bool BLUE = KIND == kBluestein, BIG = KIND == kDirectBig;
    __shared__ RingAux aux;
    const int L = v.lmax;
    const int J = v.ring_J[ring], K = J / 2, s = v.ring_s[ring];
    const int4 *__restrict__ T = ring_table(v.tw) + v.ring_tw[ring];
    const int4 *__restrict__ AB = ring_table(v.ab) + v.ring_ab[ring];
    const int *__restrict__ rl = v.rad + v.ring_rad[ring];
    RaderCtx rc;
    const RaderCtx *rcp = BIG ? rader_ctx(v, ring, K, sm, rc) : nullptr;
    const int M = BLUE ? v.ring_mx[ring] : 0;
    const int entries = BLUE ? M : BIG && rcp ? K + (K / rcp->ri->p) * rcp->ri->n : K;
    short *ex = reinterpret_cast<short *>(sm + entries);
    if (threadIdx.x == 0) aux = RingAux{{0, 0, 0}, 0, 0};
    __syncthreads();
    ring_fold<BLUE, false>(qat, L, J, s, AB, rl, sm, ex, aux);
    __syncthreads();
    int emax = aux.emax, lift = 0, renamed = 0;
    double2 *out = reinterpret_cast<double2 *>(out_ring);
    if (emax < kRingExpLo || emax > kRingExpHi) {
        if (emax == 0x7ff || !aux.any) {
            ring_fill(out, K, emax != 0x7ff);
            return;
        }
        lift = emax < kRingExpLo ? kRingLift : -kRingLift;
        if (lift < 0) {
            renamed = lift;
        } else {
            __syncthreads();
            if (threadIdx.x == 0) aux.emax = 0;
            __syncthreads();
            // in line: a call costs the ordinary path registers (ring stage of 8
            // maps at Nside = 512 .884 against .875 ms)
            ring_fold<BLUE, true>(qat, L, J, s, AB, rl, sm, ex, aux);
            __syncthreads();
            emax = aux.emax;
        }
    }
    FxScale sc{aux.slot, 0, emax + renamed - 1080};
    unsigned mag = 0;
    for (int p = threadIdx.x; p < (BLUE ? M : K); p += blockDim.x) {
        if (BLUE && p >= K) {
            sm[p] = make_longlong2(0, 0);
            continue;
        }
        const int n = min(63, emax - ex[p]);
        const fx2 z = make_longlong2(sm[p].x >> n, sm[p].y >> n);
        sm[p] = z;
        mag |= fmag(z);
    }
    sc.leave(mag);
    if constexpr (BLUE) bluestein_mx(sm, M, ring_table(v.mfb) + v.ring_mfb[ring], rl, TwTable{ring_table(v.mtw) + v.ring_mtw[ring]}, sc);
    else if constexpr (BIG) fft_big_dit(sm, K, rl, TwRing{T, J}, sc, rcp);
    else fft_mx_dit<false>(sm, K, K, rl, TwRing{T, J}, sc);
    const int sh = sc.enter();
    const int be = sc.e + (BLUE ? 2 : 0) + 1054;
    for (int n = threadIdx.x; n < K; n += blockDim.x) {
        fx2 z = fshl(sm[n], sh);
        if (BLUE) z = fmul(z, ring_root(T, J, 2 * n * n));
        out[n] = make_double2(fix_to_double(z.x, be), fix_to_double(z.y, be));
    }
    if (lift) ring_scale_back(out, K, lift);
    __syncthreads();
}

// ... with q_m read from a ring-major array qr[m]
template <int KIND, bool CG>
__device__ __forceinline__ void phi_synth_ring(const PlanView &v, int ring, const double2 *qr, double *out_ring, fx2 *sm)
{
    phi_synth_ring_at<KIND>(v, ring, [qr](int m) { return ldq<CG>(qr + m); }, out_ring, sm);
}

// ... with q_m formed from the two parity halves of the butterfly output,
// stored as QtView says (qt, lp); north rings (ring < nhalf) take q^0 + q^1, their mirrors q^0 - q^1.
template <int KIND, bool CG>
__device__ __forceinline__ void phi_synth_ring_qt(const PlanView &v, int ring, const double2 *qt, int lp, int b,
                                                  double *out_ring, fx2 *sm)
{
    const int Z = v.nhalf, L = v.lmax;
    const bool north = ring < Z;
    const int r = north ? ring : v.nrings - 1 - ring;
    const double2 *q0 = qt + ((((size_t)((b >> lp) * 2) * Z + r) * (L + 1)) << lp) + (b & ((1 << lp) - 1));
    const double2 *q1 = q0 + ((size_t)Z * (L + 1) << lp);
    auto qat = [=](int m) {
        const double2 x0 = ldq<CG>(q0 + ((size_t)m << lp));
        if (m + 1 > L) return x0;
        return cadd(x0, cneg_if(ldq<CG>(q1 + ((size_t)m << lp)), !north));
    };
    phi_synth_ring_at<KIND>(v, ring, qat, out_ring, sm);
}

// A ring's pixels as points of exponent emax (2^20 times it): z_n in units of
// 2^(emax - 1083), with the chirp on Bluestein rings; returns their size
template <bool BLUE>
__device__ __forceinline__ unsigned ring_load(const double2 *in, int K, int M, const int4 *__restrict__ T, int J,
                                              int emax, int lift, fx2 *sm)
{
    const int e3 = emax + (3 << 20);
    unsigned mag = 0;
    for (int n = threadIdx.x; n < (BLUE ? M : K); n += blockDim.x) {
        if (BLUE && n >= K) {
            sm[n] = make_longlong2(0, 0);
            continue;
        }
        double2 zd = __ldg(in + n);
        if (lift) zd = scaled(zd, lift);
        fx2 z = make_longlong2(ring_fix(zd.x, (e3 - exp_field(zd.x)) >> 20), ring_fix(zd.y, (e3 - exp_field(zd.y)) >> 20));
        if (BLUE) z = fmul(fconj(z), ring_root(T, J, 2 * n * n));    // forward = conj(inverse(conj))
        sm[n] = z;
        mag |= fmag(z);
    }
    return mag;
}

// ... of 2^kRingLift times the pixels, whose largest exponent is left in aux
template <bool BLUE>
__device__ __noinline__ unsigned ring_load_lifted(const double2 *in, int K, int M, const int4 *T, int J, RingAux &aux, fx2 *sm)
{
    __syncthreads();
    if (threadIdx.x == 0) aux.emax = 0;
    __syncthreads();
    int emax = 0;
    for (int n = threadIdx.x; n < K; n += blockDim.x) {
        const double2 z = scaled(in[n], kRingLift);
        emax = max(emax, max(exp_field(z.x), exp_field(z.y)));
    }
    emax = (int)__reduce_max_sync(0xffffffffu, (unsigned)emax);
    if ((threadIdx.x & 31) == 0) atomicMax(&aux.emax, emax);
    __syncthreads();
    return ring_load<BLUE>(in, K, M, T, J, aux.emax, kRingLift, sm);
}

// Adjoint of one ring: q_adj[m] = sum_j f_j e^{-i m phi_j}, m = 0..L, from
// z_n = f_{2n} + i f_{2n+1}, Zf = DFT(z) with exponent -1 (position order, or
// natural order on Bluestein rings), F_r = E'_r + e^{-2 pi i r/J} O'_r with
// E' = (Zf_r + conj Zf_{K-r})/2, O' = (Zf_r - conj Zf_{K-r})/(2i), K-periodic,
// and q_adj[m] = e^{-i pi m s / J} F_{m mod J}.
template <int KIND>
__device__ __forceinline__ void phi_adjoint_ring(const PlanView &v, int ring, const double *f_ring, double2 *outq, fx2 *sm)
{
    constexpr bool BLUE = KIND == kBluestein, BIG = KIND == kDirectBig;
    __shared__ RingAux aux;
    const int L = v.lmax;
    const int J = v.ring_J[ring], K = J / 2, s = v.ring_s[ring];
    const int4 *__restrict__ T = ring_table(v.tw) + v.ring_tw[ring];
    const int *__restrict__ rl = v.rad + v.ring_rad[ring];
    RaderCtx rc;
    const RaderCtx *rcp = BIG ? rader_ctx(v, ring, K, sm, rc) : nullptr;
    const int M = BLUE ? v.ring_mx[ring] : 0;
    if (threadIdx.x == 0) aux = RingAux{{0, 0, 0}, 0, 0};
    __syncthreads();
    const double2 *in = reinterpret_cast<const double2 *>(f_ring);
    int emax = 0, lift = 0;
    unsigned any = 0;
    for (int n = threadIdx.x; n < K; n += blockDim.x) {
        const double2 z = __ldg(in + n);
        emax = max(emax, max(exp_field(z.x), exp_field(z.y)));
        any |= nonzero_bits(z.x) | nonzero_bits(z.y);
    }
    emax = (int)__reduce_max_sync(0xffffffffu, (unsigned)emax);
    any = __reduce_or_sync(0xffffffffu, any);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&aux.emax, emax);
        atomicOr(&aux.any, any);
    }
    __syncthreads();
    emax = aux.emax;
    unsigned mag = 0;
    FxScale sc{aux.slot, 0, 0};
    if (emax < kRingExpLo << 20 || emax > kRingExpHi << 20) {
        if (emax == 0x7ff00000 || !aux.any) {
            ring_fill(outq, L + 1, emax != 0x7ff00000);
            return;
        }
        lift = emax < kRingExpLo << 20 ? kRingLift : -kRingLift;
    }
    if (lift <= 0) {
        sc.e = (emax >> 20) + lift - 1083;
        mag = ring_load<BLUE>(in, K, M, T, J, emax, 0, sm);
    } else {
        mag = ring_load_lifted<BLUE>(in, K, M, T, J, aux, sm);
        sc.e = (aux.emax >> 20) - 1083;
    }
    if (BLUE) sc.e += 2;
    sc.leave(mag);
    if constexpr (BLUE) {
        bluestein_mx(sm, M, ring_table(v.mfb) + v.ring_mfb[ring], rl, TwTable{ring_table(v.mtw) + v.ring_mtw[ring]}, sc);
        const int sh = sc.enter();
        mag = 0;
        for (int n = threadIdx.x; n < K; n += blockDim.x) {
            const fx2 z = fconj(fmul(fshl(sm[n], sh), ring_root(T, J, 2 * n * n)));
            sm[n] = z;
            mag |= fmag(z);
        }
        sc.e += 2;
        sc.leave(mag);
    } else {
        if constexpr (BIG) fft_big_dif(sm, K, rl, TwRing{T, J}, sc, rcp);
        else fft_mx_dif<false>(sm, K, K, rl, TwRing{T, J}, sc);
    }
    const int sh = sc.enter();
    const int be = sc.e + 1 + (s ? 4 : 2) + 1054;
    for (int m = threadIdx.x; m <= L; m += blockDim.x) {
        const int r = m % J;
        const int rho = r < K ? r : r - K;
        const int rho2 = rho == 0 ? 0 : K - rho;
        // halves of A and conj B, so that their sum and difference have room
        const fx2 A = frshift(fshl(BLUE ? sm[rho] : sm[fft_pos(rho, K, rl)], sh), 2);
        const fx2 B = fconj(frshift(fshl(BLUE ? sm[rho2] : sm[fft_pos(rho2, K, rl)], sh), 2));
        const fx2 D = fsub(A, B);
        const fx2 Op = make_longlong2(D.y, -D.x);                              // D / i
        fx2 F = fadd(frshift(fadd(A, B), 2), fmul<true>(Op, ring_root(T, J, 2 * r)));
        if (s) F = fmul<true>(F, ring_root(T, J, m));
        outq[m] = make_double2(fix_to_double(F.x, be), fix_to_double(F.y, be));
    }
    if (lift) ring_scale_back(outq, L + 1, lift);
    __syncthreads();
}

}  // namespace shtb_dev
