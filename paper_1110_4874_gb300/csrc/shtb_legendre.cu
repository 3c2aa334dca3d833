// Kernel (b): the Legendre stage by the jump-two recurrence of Eq. (three-term),
// uncompressed ("zero levels of compression", Sec. 3.3) and split by l - m
// parity over rings mirrored about the equator (Eq. q-even-odd, q-even-odd2).
//
// Synthesis: for every order m and half-ring r (z_r >= 0)
//   q^t_m(z_r) = sum_j a_{m+t+2j, m} Ptilde_{m+t+2j}^m(z_r),  t = 0 (even), 1 (odd),
// then q_m(+z_r) = q^0 + q^1 and q_m(-z_r) = q^0 - q^1 (the mirror ring).
// A warp owns 32 consecutive half-rings of one m and one parity; each lane
// runs the chain of its ring in registers and accumulates all maps of the
// batch, so the per-l constants and a_lm are warp-uniform (broadcast) loads.
// Each chain starts at its own crop point (first |Ptilde| >= 1e-30, Appendix) with
// two precomputed values and advances by two FMAs per step:
//   w_j = mu_j x_r + C_j,   V_{j+1} = w_j V_j - V_{j-1},   Ptilde = sigma V,
// the scale sigma being folded into a_lm by the prescale kernel.
//
// Adjoint: a^t_{m+t+2j} = sum_r V_j(r) g^t_r with g^0 = F(+z) + F(-z) and
// g^1 = F(+z) - F(-z).  The sum runs across the rings, i.e. across lanes, so
// each warp writes a 32 (j) x 32 (ring) tile of V to shared memory and then
// lets lane = j sum over the tile's rings.
//
// The recurrence runs in FP64; the sums over the maps, 2 NB of them a value
// of V, are integer (LegSums): V and the a or g of a run of 32 are cut to limbs
// at common exponents, and a product is three 32-bit multiply-adds.  The FP64
// pipe, which takes a warp's DFMA in 16 clocks of an SM against half a clock
// for an integer multiply-add, held these kernels with both done in FP64.
// Legendre stage, FP64 sums -> this (ms):
//   nside 64, lmax 128, 1 map      synthesis  .047 -> .031  adjoint  .054 -> .039
//   nside 100, lmax 255, 1 map                .095 -> .056           .140 -> .068
//   nside 256, lmax 512, 4 maps               .996 -> .441          1.385 -> .576
//   nside 256, lmax 512, 8 maps              1.730 -> .762          2.416 -> .981
//   nside 512, lmax 1024, 8 maps             12.22 -> 5.13          13.94 -> 5.77
// What bounds them now is issue (48 % of the slots with 8 maps, the FP64 pipe
// at 31 %) and, with few maps, the chain of dependent FMAs of the recurrence.
// Precision: a or g are cut 49 bits or more below a run's largest, V 55 to 58
// below its largest so far, the products of low limbs left out; a run whose
// sizes differ enough for that to be less than FP64 keeps is summed in FP64.
// So each ring and each coefficient is as close to the recurrence's values as
// an FP64 sum of its terms, also beside much larger ones (one exponent for a
// whole chain, .42 and .55 ms at nside 256 with 4 maps, left 1e-9 of
// coefficients beside polar pixels 1e8 times the rest).
#include <cuda_runtime.h>

#include "shtb_internal.h"
#include "shtb_limbs.cuh"

namespace {

constexpr int kWarpsPerBlock = 4;

__device__ __forceinline__ int warp_min(int v)
{
    for (int o = 16; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__device__ __forceinline__ int dchain_len(int L, int m, int t)
{
    return m + t > L ? 0 : (L - m - t) / 2 + 1;
}

__device__ __forceinline__ long long dalm_index(int L, int l, int m)
{
    return (long long)m * (2 * L + 1 - m) / 2 + l;
}

// a'[idx][b] = a_lm[b][idx] * sigma_lm   (Im a_l0 dropped: real-field input, Sec. 2.1)
__global__ void alm_prescale_kernel(PlanView v, const double2 *__restrict__ alm,
                                    double2 *__restrict__ ap, int nmaps)
{
    const int m = blockIdx.x;
    const int L = v.lmax;
    const long long off = dalm_index(L, m, m);
    const int n = L - m + 1;
    for (int i = threadIdx.x; i < n * nmaps; i += blockDim.x) {
        const int b = i / n, dl = i - b * n;
        const long long idx = off + dl;
        double2 a = alm[(size_t)b * v.nalm + idx];
        const double s = v.coef[idx].sig;
        ap[(size_t)idx * nmaps + b] = make_double2(a.x * s, m == 0 ? 0.0 : a.y * s);
    }
}

// What a run's integer sums take; other runs are summed in FP64 (plain_steps,
// plain_rings).  Limbs are cut at one place for the whole run, and V grows
// along a chain from the crop on, so a run whose large values meet a small V
// and whose small ones a large V would lose what FP64 keeps: its largest
// exponent lies in a range, every four neighbours have one at most kLegDrop
// bits below any before them, the last two one at most kLegLast, and a run of a
// (a chain's end) has kLegShort entries or more.
constexpr int kLegExpLo = 300, kLegExpHi = 1700, kLegDrop = 7, kLegLast = 10, kLegShort = 8;
// A component's scale, the exponent its limbs are cut at, is set a bit above
// the largest of the run that needs it and kept for the runs whose largest
// lies at it or up to kLegKeep bits below.
constexpr int kLegKeep = 5;

// Bits of V, so that sums of n products of 55-bit a and V fit: between two
// carries 32 products of 27-bit by 30-bit high limbs stay below 2^62, and the
// words carried out, n 2^57 2^-40 in all, below 2^31 up to chains of 8192.
__device__ __forceinline__ int v_bits(int n)
{
    return 58 - max(0, 32 - __clz(n) - 13);
}

// 1 for subnormals, 0 for zeros alone
__device__ __forceinline__ unsigned exp_of(double v)
{
    const unsigned u = (unsigned)__double2hiint(v) << 1 | (__double2loint(v) != 0 ? 1u : 0u);
    return max(u >> 21, min(u, 1u));
}

// A run is the up to 32 values of a chain that a warp's sums weight next, of C
// components each, entry i at src + i stride (doubles).  Components 2b, 2b + 1
// belong to the lanes of b = lane mod NB, which hold entries r + q STEP, r =
// lane / NB.
template <int NB>
struct Run {
    static constexpr int STEP = 32 / NB;
    double2 x[NB];
    __device__ __forceinline__ void load(const double *src, size_t stride, int count, int lane)
    {
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            const int i = q * STEP + lane / NB;
            x[q] = i < count ? __ldg(reinterpret_cast<const double2 *>(src + (size_t)i * stride) + lane % NB)
                             : make_double2(0.0, 0.0);
        }
    }
    // the largest exponent: 0 for a component of zeros, -1 for one to take in FP64
    __device__ __forceinline__ int2 scan(int count, int least, int lane) const
    {
        unsigned top = 0, drop = 0, last = 0;                        // two components in halves
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            unsigned e = exp_of(x[q].x) | exp_of(x[q].y) << 16;      // of the four entries 4 (i / 4) ..
            e = __vmaxu2(e, __shfl_xor_sync(0xffffffffu, e, NB));
            if (q == (count - 1) / STEP) last = e;
            e = __vmaxu2(e, __shfl_xor_sync(0xffffffffu, e, 2 * NB));
            unsigned before = e;                                     // the largest up to them
#pragma unroll
            for (int o = 4 * NB; o < 32; o *= 2) {
                const unsigned y = __shfl_up_sync(0xffffffffu, before, o);
                if (lane >= o) before = __vmaxu2(before, y);
            }
            before = __vmaxu2(before, top);
            if (((q * STEP + lane / NB) & ~3) < count) drop = __vmaxu2(drop, before - e);
            top = NB == 8 ? before : __shfl_sync(0xffffffffu, before, 32 - NB + lane % NB);
        }
#pragma unroll
        for (int o = 4 * NB; o < 32; o *= 2) drop = __vmaxu2(drop, __shfl_xor_sync(0xffffffffu, drop, o));
        last = top - __shfl_sync(0xffffffffu, last, (count - 1) % STEP * NB + lane % NB);
        auto one = [count, least](int e, int below, int end) {
            return e == 0 ? 0 : e < kLegExpLo || e > kLegExpHi || below > kLegDrop || end > kLegLast || count < least ? -1 : e;
        };
        return make_int2(one(top & 0xffff, drop & 0xffff, last & 0xffff), one(top >> 16, drop >> 16, last >> 16));
    }
    // limbs of 55 bits at the scales of the components that e takes
    __device__ __forceinline__ void limbs(int2 e, int2 scale, int2 *lim, int lane) const
    {
        int4 *lim4 = reinterpret_cast<int4 *>(lim);
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            const int2 l0 = e.x > 0 ? shtb_dev::to_limbs(x[q].x, 9 + scale.x - shtb_dev::exp_bits(x[q].x)) : make_int2(0, 0);
            const int2 l1 = e.y > 0 ? shtb_dev::to_limbs(x[q].y, 9 + scale.y - shtb_dev::exp_bits(x[q].y)) : make_int2(0, 0);
            lim4[(q * STEP + lane / NB) * NB + lane % NB] = make_int4(l0.x, l0.y, l1.x, l1.y);
        }
    }
};

// entries of the next run of `left`: 32, or 24 where 32 would leave a short one
__device__ __forceinline__ int run_length(int left)
{
    return left > 32 && left < 32 + kLegShort ? 32 - kLegShort : min(32, left);
}

// the scale for a run of largest exponent e: none where the run adds nothing
// in integers, so that a sum is never moved to a V it has no products of
__device__ __forceinline__ int next_scale(int scale, int e)
{
    return e <= 0 ? 0 : e <= scale && e >= scale - kLegKeep ? scale : e + 1;
}

__device__ __forceinline__ bool scale_left(int2 scale, int2 next)
{
    return (scale.x != 0 && scale.x != next.x) || (scale.y != 0 && scale.y != next.y);
}

// component c's of a pair on the lanes of b
__device__ __forceinline__ int of_component(int2 v, int c)
{
    return __shfl_sync(0xffffffffu, c & 1 ? v.y : v.x, c >> 1);
}

// A warp's 32 running sums (one a lane) per component, on a common exponent E
// of the V seen so far (0: none yet) with up to kHead bits to spare, so that a
// growing V raises it only now and then: value (H 2^68 + P 2^28 + M) 2^28 2^(scale + E - ..)
constexpr int kHead = 3;
// chain steps between two looks at E (one for every map count: the same bits)
constexpr int kStep = 4;

template <int C>
struct LegSums {
    long long P[C], M[C];
    int H[C];
    int E, vb, base;                     // exponent of V, bits of V, limb shift at exponent 0
    __device__ __forceinline__ void clear(int n)
    {
        E = 0;
        vb = v_bits(n);
        base = 4096;                     // every V (a zero) shifted out
#pragma unroll
        for (int c = 0; c < C; ++c) P[c] = M[c] = H[c] = 0;
    }
    // before adding V of exponents up to e
    __device__ __forceinline__ void raise(int e)
    {
        if (!__any_sync(0xffffffffu, e > E)) return;
        int s = e > E ? e + kHead - E : 0;
        if (s > 0) {
            if (E == 0) s = 0;           // nothing summed yet
            E = e + kHead;
            base = 64 - vb + E;
        }
#pragma unroll 1
        while (__any_sync(0xffffffffu, s > 0)) {
            const int k = min(s, 20);
            const unsigned mask = (1u << k) - 1;
#pragma unroll
            for (int c = 0; c < C; ++c) {
                M[c] = (M[c] + ((long long)((unsigned)P[c] & mask) << 28)) >> k;
                P[c] = (P[c] + ((long long)((unsigned)H[c] & mask) << 40)) >> k;
                H[c] >>= k;
            }
            s -= k;
        }
    }
    __device__ __forceinline__ void add(double v, const int2 *lim)
    {
        const int2 w = shtb_dev::to_limbs(v, base - shtb_dev::exp_bits(v));
#pragma unroll
        for (int c = 0; c < C; c += 2) {
            const int4 a = *reinterpret_cast<const int4 *>(lim + c);
            P[c] = shtb_dev::mad_wide(a.y, w.y, P[c]);
            M[c] = shtb_dev::mad_wide(a.y, w.x, M[c]);
            M[c] = shtb_dev::mad_wide(a.x, w.y, M[c]);
            P[c + 1] = shtb_dev::mad_wide(a.w, w.y, P[c + 1]);
            M[c + 1] = shtb_dev::mad_wide(a.w, w.x, M[c + 1]);
            M[c + 1] = shtb_dev::mad_wide(a.z, w.y, M[c + 1]);
        }
    }
    // every 32 products, so that none overflows
    __device__ __forceinline__ void carry()
    {
#pragma unroll
        for (int c = 0; c < C; ++c) {
            P[c] += M[c] >> 28;
            M[c] &= (1LL << 28) - 1;
            H[c] += (int)(P[c] >> 40);
            P[c] &= (1LL << 40) - 1;
        }
    }
    __device__ __forceinline__ void drop(int c) { P[c] = M[c] = H[c] = 0; }
    // after a carry; a = X_a 2^(e_a - 1077), V = X_V 2^(E - 1022 - vb)
    __device__ __forceinline__ double value(int c, int ea) const
    {
        const long long p = (long long)H[c] << 30 | P[c] >> 10, l = ((long long)P[c] & 1023) << 18 | M[c] >> 10;
        return ea > 0 && E > 0 ? shtb_dev::limbs_to_double(p, l, 10 + 28 + 1054 + ea - 1077 + 28 + E - 1022 - vb) : 0.0;
    }
};

// One ring's chain of one parity, advanced step by step: value V_j at `cur`
struct Chain {
    double x, cur, prev;
    double2 start;
    int js;
    bool sform;
    __device__ __forceinline__ void begin(int j)
    {
        cur = js == j ? start.x : 0.0;
        prev = 0.0;
    }
    __device__ __forceinline__ void step(int j, const RecCoef &c)
    {
        const double w = fma(c.mu, x, sform ? c.cs : c.cz);
        double nxt = fma(w, cur, -prev);
        if (j == js) nxt = start.y;
        if (j + 1 == js) nxt = start.x;
        prev = cur;
        cur = nxt;
    }
};

// The products of the next `count` steps' V with the components (e < 0) that
// integers do not take, in FP64; a: their first entry, component c's sum at
// sum[32 c]
template <int NB>
__device__ __noinline__ void plain_steps(double v0, double v1, double v2, double v3, const double *a, size_t stride,
                                         int count, int2 e, double *sum)
{
    static_assert(kStep == 4, "four steps");
    const double V[kStep] = {v0, v1, v2, v3};
    const unsigned pairs = __ballot_sync(0xffffffffu, min(e.x, e.y) < 0);
#pragma unroll 1
    for (int b = 0; b < NB; ++b) {
        if (!(pairs >> b & 1)) continue;
        double2 x[kStep], s = make_double2(sum[64 * b], sum[64 * b + 32]);
#pragma unroll
        for (int i = 0; i < kStep; ++i)
            x[i] = __ldg(reinterpret_cast<const double2 *>(a + (size_t)min(i, count - 1) * stride) + b);
#pragma unroll
        for (int i = 0; i < kStep; ++i)
            if (i < count) {
                s.x = fma(x[i].x, V[i], s.x);
                s.y = fma(x[i].y, V[i], s.y);
            }
        if (of_component(e, 2 * b) < 0) sum[64 * b] = s.x;
        if (of_component(e, 2 * b + 1) < 0) sum[64 * b + 32] = s.y;
    }
}

// One warp per (m, 32 half-rings, parity); the two parities of a (m, rings)
// are neighbouring warps and trade their sums through shared memory.  With 8
// maps 3 CTAs an SM spare the spills of 4 (.711 against .744 ms, nside 256).
template <int NB>
__global__ void __launch_bounds__(32 * kWarpsPerBlock, NB == 8 ? 3 : 4)
legendre_synth_kernel(PlanView v, const double2 *__restrict__ ap, double2 *__restrict__ q,
                      int nmaps, int b0)
{
    constexpr int C = 2 * NB;
    __shared__ __align__(16) int2 slim[kWarpsPerBlock][32 * C];
    __shared__ double ssum[kWarpsPerBlock][C][32];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int Z = v.nhalf, L = v.lmax;
    const int nchunk = (Z + 31) >> 5;
    const long long item = ((long long)blockIdx.x * kWarpsPerBlock + warp) >> 1;
    const int t = warp & 1;
    const bool there = item < (long long)(L + 1) * nchunk;
    const int m = there ? (int)(item / nchunk) : 0;
    const int chunk = there ? (int)(item - (long long)m * nchunk) : 0;
    const int r = chunk * 32 + lane;
    const bool valid = there && r < Z;
    const int rr = valid ? r : Z - 1;
    const int n = there ? dchain_len(L, m, t) : 0;
    int2 *lim = slim[warp];

    double *sum = &ssum[warp][0][lane];                                // component c at sum[32 c]
#pragma unroll
    for (int c = 0; c < C; ++c) sum[32 * c] = 0.0;
    Chain ch;
    ch.x = v.xarg[rr];
    ch.sform = v.xform[rr] != 0;
    const size_t base = ((size_t)m * 2 + t) * Z + rr;
    ch.js = valid ? v.jstart[base] : n;
    ch.start = v.vstart[base];
    const int jlo = warp_min(ch.js < n ? ch.js : n);
    if (jlo < n) {
        const long long off = dalm_index(L, m, m) + t;
        const RecCoef *__restrict__ cf = v.coef + off;                // step j at cf[2 j]
        const double *a = reinterpret_cast<const double *>(ap + (size_t)off * nmaps + b0);
        const size_t stride = (size_t)4 * nmaps;                      // doubles between chain entries
        LegSums<C> sums;
        sums.clear(n);
        int2 scale = make_int2(0, 0);
        // integer sums so far, of the components whose next scale is another, into sum
        auto settle = [&](int2 next) {
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const int e = of_component(scale, c);
                if (e == 0 || e == of_component(next, c)) continue;
                sum[32 * c] += sums.value(c, e);
                sums.drop(c);
            }
        };
        ch.begin(jlo);
        for (int jb = jlo, nj; jb < n; jb += nj) {
            nj = run_length(n - jb);
            Run<NB> run;
            run.load(a + (size_t)jb * stride, stride, nj, lane);
            const int2 ea = run.scan(nj, kLegShort, lane);
            const bool plain = __any_sync(0xffffffffu, min(ea.x, ea.y) < 0);
            const int2 next = make_int2(next_scale(scale.x, ea.x), next_scale(scale.y, ea.y));
            if (__any_sync(0xffffffffu, scale_left(scale, next))) settle(next);
            scale = next;
            __syncwarp();
            run.limbs(ea, scale, lim, lane);
            __syncwarp();
            for (int i0 = 0; i0 < nj; i0 += kStep) {
                double V[kStep];
                int e = 0;
#pragma unroll
                for (int i = 0; i < kStep; ++i) {
                    V[i] = 0.0;
                    if (i0 + i < nj) {
                        V[i] = ch.cur;
                        e = max(e, shtb_dev::exp_bits(ch.cur));
                        ch.step(jb + i0 + i, cf[2 * (jb + i0 + i)]);
                    }
                }
                sums.raise(e);
#pragma unroll
                for (int i = 0; i < kStep; ++i)
                    if (i0 + i < nj) sums.add(V[i], lim + (i0 + i) * C);
                if (plain)
                    plain_steps<NB>(V[0], V[1], V[2], V[3], a + (size_t)(jb + i0) * stride, stride, nj - i0, ea, sum);
            }
            sums.carry();
        }
        settle(make_int2(-1, -1));
    }

    // q(+z) = q^0 + q^1 by the even warp, q(-z) = q^0 - q^1 by the odd one
    __syncthreads();
    if (!valid || (t == 1 && r == Z - 1)) return;                      // the equator ring has no mirror
    const double *other = &ssum[warp ^ 1][0][lane];
    const int ring = t == 0 ? r : v.nrings - 1 - r;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        const double x = sum[64 * b], y = sum[64 * b + 32], ox = other[64 * b], oy = other[64 * b + 32];
        q[((size_t)(b0 + b) * v.nrings + ring) * (L + 1) + m] =
            t == 0 ? make_double2(x + ox, y + oy) : make_double2(ox - x, oy - y);
    }
}


// ------------------------------------------------------------------ adjoint
// g[((m*2 + t)*Z + r)*nmaps + b]: parity combination of the ring-stage
// adjoint output, g^0 = F(+z_r) + F(-z_r), g^1 = F(+z_r) - F(-z_r); the
// equator ring (r = Z-1) has no mirror and contributes once.
// One CTA per (half-ring r, run of 64 orders m): reads each map's run of q_adj
// on ring r and its mirror, and writes the maps of one (m, t, r) entry of g
// next to each other, up to 16 maps at a time.  Shared memory turns the
// map-major reads into the entry-major writes, so both are coalesced.
constexpr int kParityM = 64, kParityMaps = 16;

__global__ void __launch_bounds__(256) adjoint_parity_kernel(PlanView v, const double2 *__restrict__ qa,
                                                             double2 *__restrict__ g, int nmaps, int columns)
{
    __shared__ double2 tile[2][kParityMaps][kParityM];     // north, south
    const int r = blockIdx.x, m0 = blockIdx.y * kParityM;
    const int Z = v.nhalf, L = v.lmax;
    const int nm = min(kParityM, L + 1 - m0);
    const bool equator = r == Z - 1;
    for (int b0 = 0; b0 < columns; b0 += kParityMaps) {
        const int nb = min(kParityMaps, columns - b0);
        for (int i = threadIdx.x; i < nb * nm; i += blockDim.x) {
            const int b = i / nm, ml = i - b * nm;
            const size_t row = (size_t)min(b0 + b, nmaps - 1) * v.nrings;
            tile[0][b][ml] = qa[(row + r) * (L + 1) + m0 + ml];
            tile[1][b][ml] = equator ? make_double2(0.0, 0.0) : qa[(row + (v.nrings - 1 - r)) * (L + 1) + m0 + ml];
        }
        __syncthreads();
        for (int i = threadIdx.x; i < nb * nm; i += blockDim.x) {
            const int ml = i / nb, b = i - ml * nb;
            const double2 a = tile[0][b][ml], c = tile[1][b][ml];
            const size_t m = (size_t)(m0 + ml);
            g[((m * 2 + 0) * Z + r) * columns + b0 + b] = make_double2(a.x + c.x, a.y + c.y);
            g[((m * 2 + 1) * Z + r) * columns + b0 + b] = make_double2(a.x - c.x, a.y - c.y);
        }
        __syncthreads();
    }
}

// Warps W of a CTA: an order's chains are as long as its tiles are many, and
// orders are too few to fill the chip by themselves.  4, 8, 16 warps: .786,
// .542, .682 ms at nside 256 with 4 maps, 1.31, .89, 1.06 with 8, .51, .35,
// .38 with 1.  16 where that is a chunk of rings for each and 8 would take two
// (5 to 8 chunks): .096 -> .076 ms at nside 128 with 1 map, .145 -> .114
// with 4, .245 -> .191 with 8; nside 100 .085 -> .068, .132 -> .102, .214 -> .173.
constexpr int kTilePad = 33;   // row stride (doubles) of the 32x32 tile: no bank conflicts

// per warp: the tile of V and the limbs of 32 rings' g (the sums' trade later)
template <int NB>
__host__ __device__ constexpr size_t adjoint_warp_smem_doubles()
{
    return 32 * kTilePad + 32 * 2 * NB;
}

// most chunks of rings a warp takes
__host__ __device__ constexpr int adjoint_warp_chunks(int nchunk, int W) { return (nchunk + W / 2 - 1) / (W / 2); }

// A run of rings' products with the components (e < 0) that integers do not
// take, in FP64, lane = chain step; rings whose V is cropped there are left
// out.  buf: 32 double2 of the warp's
template <int NB>
__device__ __noinline__ void plain_rings(const double *row, const double *g, size_t stride, int count, int2 e,
                                         double2 *buf, double *acc, int lane)
{
    const unsigned pairs = __ballot_sync(0xffffffffu, min(e.x, e.y) < 0);
#pragma unroll 1
    for (int b = 0; b < NB; ++b) {
        if (!(pairs >> b & 1)) continue;
        __syncwarp();
        buf[lane] = lane < count ? __ldg(reinterpret_cast<const double2 *>(g + (size_t)lane * stride) + b) : make_double2(0.0, 0.0);
        __syncwarp();
        double2 s[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) s[i] = make_double2(0.0, 0.0);
#pragma unroll 1
        for (int r = 0; r < 32; r += 4)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const double v = row[r + i];
                const double2 x = buf[r + i];
                const bool there = exp_of(v) != 0;
                s[i].x = fma(v, there ? x.x : 0.0, s[i].x);
                s[i].y = fma(v, there ? x.y : 0.0, s[i].y);
            }
        if (of_component(e, 2 * b) < 0) acc[2 * b] += (s[0].x + s[1].x) + (s[2].x + s[3].x);
        if (of_component(e, 2 * b + 1) < 0) acc[2 * b + 1] += (s[0].y + s[1].y) + (s[2].y + s[3].y);
    }
}

// One CTA per m: the even warps take the even chain, the odd ones the odd
// chain, each its share of the chunks of 32 rings.
template <int NB, int W>
__global__ void __launch_bounds__(32 * W, 16 / W)
legendre_adjoint_kernel(PlanView v, const double2 *__restrict__ g, double2 *__restrict__ aacc,
                        RecState *__restrict__ state, int nmaps, int b0)
{
    constexpr int C = 2 * NB;
    extern __shared__ __align__(16) double smd[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5, t = warp & 1, set = warp >> 1;
    const int Z = v.nhalf, L = v.lmax;
    const int m = blockIdx.x;
    const int n = dchain_len(L, m, t), n0 = dchain_len(L, m, 0);
    const int nchunk = (Z + 31) >> 5;
    const long long off = dalm_index(L, m, m);
    const RecCoef *__restrict__ cf = v.coef + off + t;                // step j at cf[2 j]
    double *tile = smd + (size_t)warp * adjoint_warp_smem_doubles<NB>();   // [32][kTilePad]
    int2 *lim = reinterpret_cast<int2 *>(tile + 32 * kTilePad);            // [32][C]
    double2 *st = reinterpret_cast<double2 *>(state + (size_t)blockIdx.x * Z) + t;   // ring r at st[2 r]
    const double *gm = reinterpret_cast<const double *>(g + ((size_t)m * 2 + t) * Z * nmaps + b0);
    const size_t gstride = (size_t)2 * nmaps;                         // doubles between rings
    const int ntiles = (n0 + 31) >> 5;
    const int Zt = Z - t;                                             // the odd functions vanish on the equator
    // the largest exponents of this warp's runs of g: chunk set + i W/2 at se[i NB + b]
    short2 *se = reinterpret_cast<short2 *>(smd + (size_t)W * adjoint_warp_smem_doubles<NB>()) +
               (size_t)warp * adjoint_warp_chunks(nchunk, W) * NB;
    // (a last run of few rings is no chain's end: V is level about the equator)
    auto rings = [&](int c) { return max(1, min(32, Zt - c * 32)); };
    for (int c = set, i = 0; c < nchunk; c += W / 2, ++i) {
        Run<NB> run;
        run.load(gm + (size_t)c * 32 * gstride, gstride, rings(c), lane);
        const int2 e = run.scan(rings(c), 1, lane);
        if (lane < NB) se[i * NB + lane] = make_short2((short)e.x, (short)e.y);
    }
    __syncwarp();

    for (int ti = 0; ti < ntiles; ++ti) {
        const int jt = ti * 32;
        LegSums<C> sums;
        sums.clear(Z);
        int2 scale = make_int2(0, 0);
        // sums of the tile that the integers no longer hold; most tiles need none,
        // so the (local memory) array is not touched before one does: 5.93 -> 5.77
        // ms with 8 maps at nside 512
        double acc[C];
        bool kept = false;
        auto keep = [&] {
            if (kept) return;
            kept = true;
#pragma unroll
            for (int c = 0; c < C; ++c) acc[c] = 0.0;
        };
        auto settle = [&](int2 next) {
            keep();
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const int e = of_component(scale, c);
                if (e == 0 || e == of_component(next, c)) continue;
                acc[c] += sums.value(c, e);
                sums.drop(c);
            }
        };
        for (int c = set; c < nchunk && jt < n; c += W / 2) {
            const int r = c * 32 + lane;
            const bool valid = r < Z;
            const int rr = valid ? r : Z - 1;
            const size_t base = ((size_t)m * 2 + t) * Z + rr;
            Chain ch;
            ch.js = valid ? v.jstart[base] : n;
            const int clo = warp_min(ch.js < n ? ch.js : n);
            if (clo >= n || jt + 32 <= clo) continue;   // chunk is zero in this tile
            ch.start = v.vstart[base];
            ch.x = v.xarg[rr];
            ch.sform = v.xform[rr] != 0;
            ch.begin(jt);
            if (ti != (clo >> 5) && valid) {       // lanes past the last ring keep V = 0
                const double2 sv = st[2 * rr];
                ch.cur = sv.x;
                ch.prev = sv.y;
            }
            // lane = ring: V_j for the tile's 32 chain steps
            for (int jj = 0; jj < 32; ++jj) {
                const int j = jt + jj;
                tile[jj * kTilePad + lane] = j < n ? ch.cur : 0.0;
                if (j < n) ch.step(j, cf[2 * j]);
            }
            if (valid) st[2 * r] = make_double2(ch.cur, ch.prev);
            const double *gc = gm + (size_t)c * 32 * gstride;
            const int nr = rings(c);
            const short2 es = se[(c - set) / (W / 2) * NB + lane % NB];
            const int2 eg = make_int2(es.x, es.y);
            const int2 next = make_int2(next_scale(scale.x, eg.x), next_scale(scale.y, eg.y));
            if (__any_sync(0xffffffffu, scale_left(scale, next))) settle(next);
            scale = next;
            Run<NB> run;
            run.load(gc, gstride, nr, lane);
            run.limbs(eg, scale, lim, lane);
            __syncwarp();
            // lane = chain step: sum over the tile's 32 rings (those past the last have V = 0)
            const double *row = tile + lane * kTilePad;
            int e = 0;
#pragma unroll 8
            for (int r2 = 0; r2 < 32; ++r2) e = max(e, shtb_dev::exp_bits(row[r2]));
            sums.raise(e);
#pragma unroll 4
            for (int r2 = 0; r2 < 32; ++r2) sums.add(row[r2], lim + r2 * C);
            sums.carry();
            if (__any_sync(0xffffffffu, min(eg.x, eg.y) < 0)) {
                keep();
                plain_rings<NB>(row, gc, gstride, nr, eg, reinterpret_cast<double2 *>(lim), acc, lane);
            }
            __syncwarp();
        }
        // add the warps' partial sums of each parity and store them
        double *mine = tile;                            // [C][32], rows of 33
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const double v = sums.value(c, of_component(scale, c));
            mine[c * kTilePad + lane] = kept ? acc[c] + v : v;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < 2 * 32 * NB; i += blockDim.x) {
            const int tt = i / (32 * NB), rem = i - tt * 32 * NB;
            const int jj = rem / NB, b = rem - jj * NB;
            const int j = jt + jj;
            if (j >= (tt == 0 ? n0 : dchain_len(L, m, 1))) continue;
            double2 sum = make_double2(0.0, 0.0);
#pragma unroll
            for (int w = tt; w < W; w += 2) {
                const double *p = smd + (size_t)w * adjoint_warp_smem_doubles<NB>() + 2 * b * kTilePad + jj;
                sum.x += p[0];
                sum.y += p[kTilePad];
            }
            aacc[(size_t)(off + tt + 2 * j) * nmaps + b0 + b] = sum;
        }
        __syncthreads();
    }
}

// alm[b][idx] = c_m sigma_idx aacc[idx][b], c_0 = 1 (Im a_l0 = 0), c_m = 2
__global__ void alm_finish_kernel(PlanView v, const double2 *__restrict__ aacc,
                                  double2 *__restrict__ alm, int nmaps)
{
    const int m = blockIdx.x;
    const int L = v.lmax;
    const long long off = dalm_index(L, m, m);
    const int n = L - m + 1;
    const double cm = m == 0 ? 1.0 : 2.0;
    for (int i = threadIdx.x; i < n * nmaps; i += blockDim.x) {
        const int b = i / n, dl = i - b * n;
        const long long idx = off + dl;
        const double s = cm * v.coef[idx].sig;
        const double2 a = aacc[(size_t)idx * nmaps + b];
        alm[(size_t)b * v.nalm + idx] = make_double2(a.x * s, m == 0 ? 0.0 : a.y * s);
    }
}

template <int NB, int W>
int launch_adjoint_nb(const shtb_plan_s *p, const double2 *g, double2 *aacc, RecState *state,
                      int nmaps, int b0, cudaStream_t st)
{
    const size_t smem = sizeof(double) * adjoint_warp_smem_doubles<NB>() * W +
                        sizeof(short2) * NB * W * adjoint_warp_chunks((p->nhalf + 31) / 32, W);
    SHTB_CUDA_TRY(cudaFuncSetAttribute(legendre_adjoint_kernel<NB, W>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    legendre_adjoint_kernel<NB, W><<<p->lmax + 1, 32 * W, smem, st>>>(p->view, g, aacc, state,
                                                                           nmaps, b0);
    ++p->launches;
    SHTB_CUDA_TRY(cudaGetLastError());
    return SHTB_OK;
}

template <int W>
int launch_adjoint_groups(const shtb_plan_s *p, const double2 *g, double2 *aacc, RecState *state, int nmaps,
                          cudaStream_t st)
{
    for (int b0 = 0; b0 < nmaps;) {
        const int left = nmaps - b0;
        int rc;
        if (left >= 8) { rc = launch_adjoint_nb<8, W>(p, g, aacc, state, nmaps, b0, st); b0 += 8; }
        else if (left >= 4) { rc = launch_adjoint_nb<4, W>(p, g, aacc, state, nmaps, b0, st); b0 += 4; }
        else if (left >= 2) { rc = launch_adjoint_nb<2, W>(p, g, aacc, state, nmaps, b0, st); b0 += 2; }
        else { rc = launch_adjoint_nb<1, W>(p, g, aacc, state, nmaps, b0, st); b0 += 1; }
        if (rc) return rc;
    }
    return SHTB_OK;
}

}  // namespace

int launch_alm_prescale(const shtb_plan_s *p, const double2 *alm, double2 *ap, int nmaps,
                        cudaStream_t st)
{
    alm_prescale_kernel<<<p->lmax + 1, 256, 0, st>>>(p->view, alm, ap, nmaps);
    ++p->launches;
    SHTB_CUDA_TRY(cudaGetLastError());
    return SHTB_OK;
}

int launch_legendre_synth(const shtb_plan_s *p, const double2 *ap, double2 *q, int nmaps,
                          cudaStream_t st)
{
    const int nchunk = (p->nhalf + 31) / 32;
    const long long items = (long long)(p->lmax + 1) * nchunk * 2;     // warps: both parities
    const unsigned grid = (unsigned)((items + kWarpsPerBlock - 1) / kWarpsPerBlock);
    const dim3 block(32 * kWarpsPerBlock);
    for (int b0 = 0; b0 < nmaps;) {
        const int left = nmaps - b0;
        if (left >= 8) {
            legendre_synth_kernel<8><<<grid, block, 0, st>>>(p->view, ap, q, nmaps, b0);
            b0 += 8;
        } else if (left >= 4) {
            legendre_synth_kernel<4><<<grid, block, 0, st>>>(p->view, ap, q, nmaps, b0);
            b0 += 4;
        } else if (left >= 2) {
            legendre_synth_kernel<2><<<grid, block, 0, st>>>(p->view, ap, q, nmaps, b0);
            b0 += 2;
        } else {
            legendre_synth_kernel<1><<<grid, block, 0, st>>>(p->view, ap, q, nmaps, b0);
            b0 += 1;
        }
        SHTB_CUDA_TRY(cudaGetLastError());
        ++p->launches;
    }
    return SHTB_OK;
}

size_t legendre_adjoint_state_bytes(const shtb_plan_s *p)
{
    return sizeof(RecState) * (size_t)(p->lmax + 1) * p->nhalf;
}

int launch_adjoint_parity(const shtb_plan_s *p, const double2 *qadj, double2 *g, int nmaps, int columns,
                          cudaStream_t st)
{
    adjoint_parity_kernel<<<dim3(p->nhalf, (p->lmax + kParityM) / kParityM), 256, 0, st>>>(p->view, qadj, g,
                                                                                           nmaps, columns);
    ++p->launches;
    SHTB_CUDA_TRY(cudaGetLastError());
    return SHTB_OK;
}

int launch_legendre_adjoint(const shtb_plan_s *p, const double2 *qadj, double2 *aacc, int nmaps,
                            void *ws, cudaStream_t st)
{
    // ws: [g: (L+1)*2*Z*nmaps double2][state: (L+1)*Z RecState]
    double2 *g = (double2 *)ws;
    RecState *state = (RecState *)(g + (size_t)(p->lmax + 1) * 2 * p->nhalf * nmaps);
    int rc = launch_adjoint_parity(p, qadj, g, nmaps, nmaps, st);
    if (rc) return rc;
    const int nchunk = (p->nhalf + 31) / 32;           // the same warps for every map count: the same bits
    return nchunk > 4 && nchunk <= 8 ? launch_adjoint_groups<16>(p, g, aacc, state, nmaps, st)
                                     : launch_adjoint_groups<8>(p, g, aacc, state, nmaps, st);
}

int launch_alm_finish(const shtb_plan_s *p, const double2 *aacc, double2 *alm, int nmaps,
                      cudaStream_t st)
{
    alm_finish_kernel<<<p->lmax + 1, 256, 0, st>>>(p->view, aacc, alm, nmaps);
    ++p->launches;
    SHTB_CUDA_TRY(cudaGetLastError());
    return SHTB_OK;
}
