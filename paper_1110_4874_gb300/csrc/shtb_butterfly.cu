// Kernel (a): application of the butterfly-compressed Legendre operator
// (Sec. 3.2, Eq. factor-into-block-diagonal) for synthesis, q^t = Lambda^T a,
// level by level over all (m, parity) chains at once.
//
//   bf_r_kernel      u = R^T a_I for every residual block (top level of each
//                    chain; depth-0 chains write q^t directly);
//   bf_level_kernel  one item = two sibling nodes sharing a candidate list:
//                    v = T_top^T u_top + T_bot^T u_bot, split into the parent
//                    level's two u vectors (or q^t on a leaf block at level 1);
//                    identity part = adds, dense part = k x nd products
//                    (Appendix: the identity-embedded interpolation matrices);
// and the ring stage of each map group then reads q_m(+z) = q^0 + q^1 and
// q_m(-z) = q^0 - q^1 (Eq. q-even-odd2) straight from the two parity halves.
// One warp per work item; all maps of a group (up to 8, 2 real components
// each) are carried per entry so every stored matrix element is read once
// per group.  The dense products run on the tensor cores in fixed-point
// digits (shtb_bf_fix.cuh).
#include <cuda_runtime.h>

#include <algorithm>

#include "shtb_bf_items.cuh"
#include "shtb_bf_regen.cuh"
#include "shtb_butterfly.h"

namespace {

constexpr int kBfWarps = 4;

// Staging between the caller's stacked a_lm [map][idx] and the butterfly's
// interleaved ai [idx][map]: tiles of T coefficients x MB maps pass through
// shared memory, so that both the map-major side and the interleaved side are
// read or written along consecutive addresses (one map is a plain copy).  The
// tile row is padded by one entry so the column walk spreads over the banks.
constexpr int kStageTile = 256;

struct StageTile {
    int T, MB;
    __device__ __forceinline__ explicit StageTile(int nmaps)
        : T(nmaps >= kStageTile ? 1 : kStageTile / nmaps), MB(nmaps < kStageTile ? nmaps : kStageTile) {}
};

// ai[idx][b] = a_lm[b][idx] (Im a_l0 = 0, Sec. 2.1: idx <= L is m = 0), times
// sigma_lm when sig is non-null (plans that regenerate R by the rescaled
// recurrence, Ptilde = sigma V)
__device__ __forceinline__ double2 staged(double2 a, long long i, long long L, const RecCoef *sig)
{
    const double s = sig ? sig[i].sig : 1.0;
    return sig ? make_double2(a.x * s, i <= L ? 0.0 : a.y * s) : make_double2(a.x, i <= L ? 0.0 : a.y);
}

// ai has `columns` >= nmaps columns, those past nmaps repeating the last map
__global__ void __launch_bounds__(256) bf_interleave_kernel(PlanView v, const double2 *__restrict__ alm,
                                                            double2 *__restrict__ ai, int nmaps, int columns,
                                                            const RecCoef *__restrict__ sig)
{
    __shared__ double2 tile[2 * kStageTile];
    const long long nalm = v.nalm, L = v.lmax;
    if (columns == 1) {
        for (long long i = blockIdx.x * 256LL + threadIdx.x; i < nalm; i += 256LL * gridDim.x)
            ai[i] = staged(alm[i], i, L, sig);
        return;
    }
    const StageTile st(columns);
    for (long long i0 = (long long)blockIdx.x * st.T; i0 < nalm; i0 += (long long)st.T * gridDim.x) {
        const int nt = (int)min((long long)st.T, nalm - i0);
        for (int b0 = 0; b0 < columns; b0 += st.MB) {
            const int mb = min(st.MB, columns - b0);
            for (int e = threadIdx.x; e < nt * mb; e += blockDim.x) {
                const int b = e / nt, t = e - b * nt;
                tile[b * (st.T + 1) + t] = alm[(size_t)min(b0 + b, nmaps - 1) * nalm + i0 + t];
            }
            __syncthreads();
            for (int e = threadIdx.x; e < nt * mb; e += blockDim.x) {
                const int t = e / mb, b = e - t * mb;
                ai[(size_t)(i0 + t) * columns + b0 + b] = staged(tile[b * (st.T + 1) + t], i0 + t, L, sig);
            }
            __syncthreads();
        }
    }
}

// grid of the staging kernels: every tile once, at most 16 blocks per SM
unsigned stage_grid(const shtb_plan_s *p, int nmaps)
{
    const long long T = nmaps >= kStageTile ? 1 : kStageTile / nmaps;
    const long long tiles = nmaps == 1 ? (p->nalm + 255) / 256 : (p->nalm + T - 1) / T;
    return (unsigned)std::max(1LL, std::min(tiles, 152LL * 16));
}

template <int NB>
__global__ void __launch_bounds__(32 * kBfWarps, 4)
bf_r_kernel(PlanView v, const BfRItem *__restrict__ items, int nitems, const int *__restrict__ ints,
            const uint2 *__restrict__ words, const double2 *__restrict__ ai, int nmaps, int b0,
            double *__restrict__ ubuf0, double *__restrict__ ubuf1, const int *__restrict__ depth_par,
            QtView qt)
{
    const int lane = threadIdx.x & 31;
    const int w = blockIdx.x * kBfWarps + (threadIdx.x >> 5);
    if (w >= nitems) return;
    const BfRItem it = items[w];
    double *ubuf = depth_par[it.m * 2 + it.t] ? ubuf1 : ubuf0;
    shtb_dev::bf_r_item<NB, false>(it, v.lmax, v.nhalf, ints, words, ai, nmaps, b0, ubuf, qt, lane);
}

// RING: the launch is the plan's level 1, whose items all write q^t (no
// other level's do), so each instantiation holds one output path.
template <int NB, bool RING>
__global__ void __launch_bounds__(32 * kBfWarps, 4)
bf_level_kernel(const BfItem *__restrict__ items, int nitems, int L, int nhalf, int maxnc,
                const int *__restrict__ ints, const uint2 *__restrict__ words,
                const double *__restrict__ uin, double *__restrict__ uout, QtView qt)
{
    extern __shared__ __align__(16) double sout[];     // [kBfWarps][maxnc * 2 NB]
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int w = blockIdx.x * kBfWarps + wib;
    if (w >= nitems) return;
    shtb_dev::bf_level_item<NB, false, RING ? 1 : 0>(items[w], L, nhalf, ints, words, uin, uout, qt,
                                                     sout + (size_t)wib * maxnc * 2 * NB, lane);
}

// regenerated residual blocks (residual_recurrence plans), one per warp
template <int NB>
__global__ void __launch_bounds__(32 * kBfWarps)
bf_r_rec_kernel(PlanView v, const BfRItem *__restrict__ items, int nitems, const RecStart *__restrict__ rs,
                const int *__restrict__ ints, const double2 *__restrict__ ai, int nmaps, int b0,
                double *__restrict__ ubuf0, double *__restrict__ ubuf1, const int *__restrict__ depth_par,
                QtView qt)
{
    const int lane = threadIdx.x & 31;
    const int w = blockIdx.x * kBfWarps + (threadIdx.x >> 5);
    if (w >= nitems) return;
    const BfRItem it = items[w];
    double *ubuf = depth_par[it.m * 2 + it.t] ? ubuf1 : ubuf0;
    shtb_dev::bf_r_rec_item<NB, false>(it, v, rs, ints, ai, nmaps, b0, ubuf, qt, lane);
}

// residual blocks of one map group (maps b0 .. b0+NB-1 of ai)
template <int NB>
int launch_r(const shtb_plan_s *p, const double2 *ai, int nmaps, int b0, double *u0, double *u1,
             QtView qt, cudaStream_t st)
{
    const BfPlanDev &bf = *p->bf;
    if (bf.n_ritems == 0) return SHTB_OK;
    if (bf.rec) {
        const unsigned grid = (unsigned)((bf.n_ritems + kBfWarps - 1) / kBfWarps);
        bf_r_rec_kernel<NB><<<grid, 32 * kBfWarps, 0, st>>>(p->view, bf.ritems, bf.n_ritems, bf.rstart, bf.ints,
                                                            ai, nmaps, b0, u0, u1, bf.depth_parity, qt);
        SHTB_CUDA_TRY(cudaGetLastError());
        ++p->launches;
        return SHTB_OK;
    }
    const unsigned grid = (unsigned)((bf.n_ritems + kBfWarps - 1) / kBfWarps);
    bf_r_kernel<NB><<<grid, 32 * kBfWarps, 0, st>>>(p->view, bf.ritems, bf.n_ritems, bf.ints, bf.words(), ai,
                                                    nmaps, b0, u0, u1, bf.depth_parity, qt);
    SHTB_CUDA_TRY(cudaGetLastError());
    ++p->launches;
    return SHTB_OK;
}

// butterfly levels of one map group, top down; level 1 writes q^t
template <int NB>
int launch_levels(const shtb_plan_s *p, double *u0, double *u1, QtView qt, cudaStream_t st)
{
    const BfPlanDev &bf = *p->bf;
    for (int lev = bf.depth_max; lev >= 1; --lev) {
        const int n = bf.level_counts[lev - 1];
        if (n == 0) continue;
        double *uin = (lev % 2) ? u1 : u0;
        double *uout = ((lev - 1) % 2) ? u1 : u0;
        const unsigned grid = (unsigned)((n + kBfWarps - 1) / kBfWarps);
        const int maxnc = bf.level_maxnc[lev - 1];
        const size_t smem = sizeof(double) * kBfWarps * maxnc * 2 * NB;
        auto *kern = lev == 1 ? bf_level_kernel<NB, true> : bf_level_kernel<NB, false>;
        SHTB_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        kern<<<grid, 32 * kBfWarps, smem, st>>>(bf.level_items[lev - 1], n, p->lmax, p->nhalf, maxnc, bf.ints,
                                                bf.words(), uin, uout, qt);
        SHTB_CUDA_TRY(cudaGetLastError());
        ++p->launches;
    }
    return SHTB_OK;
}

// One map group: residual blocks, butterfly levels, then (map != nullptr)
// the ring stage of the group's first `real` maps.  With map == nullptr the
// group's q^t is the caller's array (the Legendre stage alone).
template <int NB>
int run_group(const shtb_plan_s *p, const double2 *ai, int columns, int b0, int real, double *u0, double *u1,
              QtView qt, double *map, cudaStream_t st)
{
    shtb_plan_s *pp = const_cast<shtb_plan_s *>(p);
    const int ev_leg = profile_begin(pp, st);
    int ev = profile_begin(pp, st);
    int rc = launch_r<NB>(p, ai, columns, b0, u0, u1, qt, st);
    if (rc) return rc;
    profile_end(pp, st, 5, ev);
    ev = profile_begin(pp, st);
    if ((rc = launch_levels<NB>(p, u0, u1, qt, st))) return rc;
    profile_end(pp, st, 6, ev);
    profile_end(pp, st, 0, ev_leg);
    if (!map) return SHTB_OK;
    // ring stage of this group straight from q^0, q^1 (parity combine fused)
    ev = profile_begin(pp, st);
    rc = launch_phi_synth_qt(p, qt, real, map, b0, st);
    profile_end(pp, st, 1, ev);
    return rc;
}

// a_lm of merged maps (one device pointer per map) into ai[idx][map]
__global__ void bf_gather_kernel(PlanView v, const double2 *const *__restrict__ alm_of_map,
                                 double2 *__restrict__ ai, int nmaps)
{
    const int m = blockIdx.x;
    const int L = v.lmax;
    const long long off = shtb_dev::alm_off(L, m);
    const int n = L - m + 1;
    for (int i = threadIdx.x; i < n * nmaps; i += blockDim.x) {
        const int b = i / n, dl = i - b * n;
        const long long idx = off + dl;
        const double2 a = alm_of_map[b][idx];
        ai[(size_t)idx * nmaps + b] = make_double2(a.x, m == 0 ? 0.0 : a.y);
    }
}

// ------------------------------------------------------------------ adjoint
// a^t = Lambda g^t: the transposed butterfly.  Level items run bottom-up:
// item (parent P, group G) gathers its candidate vector (g on a leaf block at
// level 1, else the u of level l-1) and applies both children's T:
// u_s = [I | T_s] v  (identity entries copy, dense rows are k x nd dots).

// The contraction runs over T's dense columns, so their exponents go onto
// the candidates' values (shift) and the outputs have none.

// a level item's candidate vector in shared memory, dense column d at dpos[d]
template <int C>
struct AdjLevelVec {
    const double *in;
    const int *dpos;
    const uint2 *T;                     // the child's words: row 0 carries each column's exponent
    template <int W>
    __device__ __forceinline__ void load(int d, int i, double (&x)[W]) const
    {
        shtb_dev::ld_comps<shtb_dev::Ld::kPlain>(in + __ldg(dpos + d) * C, i, x);
    }
    __device__ __forceinline__ int shift(int d) const
    {
        const uint2 w = __ldg(T + d);
        return shtb::fix_word_exp(w.x, w.y);
    }
};

// u_i: the identity entry plus the dense product (later chunks on top)
template <int C>
struct AdjLevelOut {
    const double *in;
    const int *ipos;
    double *dst;
    // output i and its identity entry's position (both below 2^15)
    __device__ __forceinline__ int key(int i) const { return i << 16 | __ldg(ipos + i); }
    template <int W>
    __device__ __forceinline__ void put(int key, bool add, int c, const double (&v)[W]) const
    {
        double *d = dst + (size_t)(key >> 16) * C;
        if (add) {
            shtb_dev::st_comps(d, c, v, true);
            return;
        }
        double x[W];
        shtb_dev::ld_comps<shtb_dev::Ld::kPlain>(in + (key & 0xffff) * C, c, x);
#pragma unroll
        for (int q = 0; q < W; ++q) x[q] += v[q];
        shtb_dev::st_comps(d, c, x, false);
    }
};

template <int NB>
__global__ void __launch_bounds__(32 * kBfWarps, 4)
bf_adj_level_kernel(const BfItem *__restrict__ items, int nitems, int maxnc, const int *__restrict__ ints,
                    const uint2 *__restrict__ words, const double *__restrict__ uin,
                    const double2 *__restrict__ g, int nmaps, int b0, double *__restrict__ uout)
{
    constexpr int C = 2 * NB;
    extern __shared__ __align__(16) double sin_[];     // [kBfWarps][maxnc * C]
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int w = blockIdx.x * kBfWarps + wib;
    if (w >= nitems) return;
    const BfItem it = items[w];
    double *in = sin_ + (size_t)wib * maxnc * C;
    double2 *in2 = reinterpret_cast<double2 *>(in);
    if (it.to_rings) {
        const int *__restrict__ ent = ints + it.out_off;
        for (int i = lane; i < it.nc * NB; i += 32) {
            const int cpos = i / NB, b = i - cpos * NB;
            in2[i] = g[(size_t)ent[cpos] * nmaps + b0 + b];
        }
    } else {
        const double2 *src = reinterpret_cast<const double2 *>(uin + (size_t)it.out_off * C);
        for (int i = lane; i < it.nc * NB; i += 32) in2[i] = src[i];
    }
    __syncwarp();
#pragma unroll 1
    for (int s = 0; s < 2; ++s) {
        const int k = it.k[s], nd = it.nd[s];
        if (k == 0) continue;
        const uint2 *T = words + it.T_off[s];
        const int *__restrict__ ipos = ints + it.ipos_off[s];
        double *dst = uout + (size_t)it.u_off[s] * C;
        if (nd == 0) {                  // identity entries alone
            for (int i = lane; i < k * C; i += 32) dst[i] = in[ipos[i / C] * C + i % C];
            continue;
        }
        const AdjLevelVec<C> vec{in, ints + it.dpos_off[s], T};
        const AdjLevelOut<C> out{in, ipos, dst};
        shtb_dev::fix_product<C, false>(T, 1, nd, nd, k, vec, out, lane);
    }
}

// a residual block's u (or g at depth 0), column s of R
template <int C>
struct AdjResVec {
    const double *u;                    // u entries, or null: g entries ent
    const double *g;                    // component 0 of the group in g[entry][nmaps]
    const int *ent;
    int gstride;
    const uint2 *R;                     // row 0 carries each column's exponent
    __device__ __forceinline__ const double *at(int s) const
    {
        return u ? u + (size_t)s * C : g + (size_t)__ldg(ent + s) * gstride;
    }
    template <int W>
    __device__ __forceinline__ void load(int s, int i, double (&x)[W]) const
    {
        shtb_dev::ld_comps<shtb_dev::Ld::kGlobal>(at(s), i, x);
    }
    __device__ __forceinline__ int shift(int s) const
    {
        const uint2 w = __ldg(R + s);
        return shtb::fix_word_exp(w.x, w.y);
    }
};

template <int C>
struct AdjResOut {
    double *acc;
    __device__ __forceinline__ int key(int n) const { return n; }
    template <int W>
    __device__ __forceinline__ void put(int n, bool, int i, const double (&v)[W]) const
    {
        shtb_dev::st_comps(acc + n * C, i, v, true);
    }
};

// a rows of one (chain, row interval), kAdjRows at a time in shared memory:
// a_j = sum over the group's residual blocks of R[j, :] x.  Every row of the
// interval is written (zero when no block reaches it), so each chain row has
// exactly one writer.  32 rows hold most intervals (25 on average), and a
// longer pass would cost resident warps their shared memory.
constexpr int kAdjRows = 32;

template <int NB>
__global__ void __launch_bounds__(32 * kBfWarps, 4)
bf_adj_r_kernel(PlanView v, const BfRGroup *__restrict__ groups, int ngroups,
                const BfRItem *__restrict__ ritems, const int *__restrict__ ints,
                const uint2 *__restrict__ words, const double *__restrict__ u0,
                const double *__restrict__ u1, const int *__restrict__ depth_par,
                const double2 *__restrict__ g, int nmaps, int b0, double2 *__restrict__ aacc)
{
    constexpr int C = 2 * NB;
    __shared__ __align__(16) double srow[kBfWarps][kAdjRows * C];
    const int lane = threadIdx.x & 31;
    const int w = blockIdx.x * kBfWarps + (threadIdx.x >> 5);
    if (w >= ngroups) return;
    double *acc = srow[threadIdx.x >> 5];
    double2 *acc2 = reinterpret_cast<double2 *>(acc);
    const BfRGroup gr = groups[w];
    const double *ubuf = depth_par[gr.m * 2 + gr.t] ? u1 : u0;
    const long long aoff = shtb_dev::alm_off(v.lmax, gr.m) + gr.t;
    for (int j0 = gr.r0; j0 < gr.r1; j0 += kAdjRows) {
        const int nj = min(kAdjRows, gr.r1 - j0);
        for (int i = lane; i < nj * NB; i += 32) acc2[i] = make_double2(0.0, 0.0);
        __syncwarp();
        for (int q = 0; q < gr.nblk; ++q) {
            const BfRItem it = ritems[ints[gr.blk_off + q]];
            const int ja = max(j0, it.j0), jb = min(j0 + nj, it.j0 + it.nrows);
            if (ja >= jb) continue;                    // no row of this pass
            const uint2 *R = words + it.data_off;
            const AdjResVec<C> vec{it.to_rings ? nullptr : ubuf + (size_t)it.out_off * C,
                                   reinterpret_cast<const double *>(g + b0), it.to_rings ? ints + it.out_off : nullptr,
                                   2 * nmaps, R};
            const AdjResOut<C> out{acc + (ja - j0) * C};
            shtb_dev::fix_product<C, false>(R + (size_t)(ja - it.j0) * it.k, 1, it.k, it.k, jb - ja, vec, out, lane);
            __syncwarp();
        }
        for (int i = lane; i < nj * NB; i += 32) {
            const int j = i / NB, b = i - j * NB;
            aacc[(size_t)(aoff + 2 * (j0 + j)) * nmaps + b0 + b] = acc2[i];
        }
        __syncwarp();
    }
}

// adjoint of regenerated residual blocks, one (chain, row interval) per warp
template <int NB>
__global__ void __launch_bounds__(32 * kBfWarps)
bf_adj_r_rec_kernel(PlanView v, const BfRGroup *__restrict__ groups, int ngroups,
                    const BfRItem *__restrict__ ritems, const RecStart *__restrict__ rs,
                    const int *__restrict__ ints, const double *__restrict__ u0, const double *__restrict__ u1,
                    const int *__restrict__ depth_par, const double2 *__restrict__ g, int nmaps, int b0,
                    double2 *__restrict__ aacc)
{
    extern __shared__ double smem_rec[];     // [kBfWarps][32 x 33 + 32 x C]
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int w = blockIdx.x * kBfWarps + wib;
    if (w >= ngroups) return;
    const BfRGroup gr = groups[w];
    const double *ubuf = depth_par[gr.m * 2 + gr.t] ? u1 : u0;
    shtb_dev::bf_adj_r_rec_group<NB>(gr, v, ritems, rs, ints, ubuf, reinterpret_cast<const double *>(g), nmaps, b0,
                                     reinterpret_cast<double *>(aacc),
                                     smem_rec + (size_t)wib * (32 * 33 + 32 * 2 * NB), lane);
}

// alm[b][idx] = c_m aacc[idx][b] (c_0 = 1 with Im a_l0 = 0, c_m = 2), the
// transposed staging of bf_interleave_kernel; times sigma_lm when sig is
// non-null (plans that regenerate R: the residual adjoint sums V, not
// Ptilde = sigma V)
__global__ void __launch_bounds__(256) bf_finish_kernel(PlanView v, const double2 *__restrict__ aacc,
                                                        double2 *__restrict__ alm, int nmaps, int columns,
                                                        const RecCoef *__restrict__ sig)
{
    __shared__ double2 tile[2 * kStageTile];
    const long long nalm = v.nalm, L = v.lmax;
    auto scaled = [L, sig](double2 a, long long idx) {
        const double cs = (idx <= L ? 1.0 : 2.0) * (sig ? sig[idx].sig : 1.0);
        return idx <= L ? make_double2(sig ? a.x * cs : a.x, 0.0)
                        : make_double2(sig ? cs * a.x : 2.0 * a.x, sig ? cs * a.y : 2.0 * a.y);
    };
    if (columns == 1) {
        for (long long i = blockIdx.x * 256LL + threadIdx.x; i < nalm; i += 256LL * gridDim.x)
            alm[i] = scaled(aacc[i], i);
        return;
    }
    const StageTile st(nmaps);
    for (long long i0 = (long long)blockIdx.x * st.T; i0 < nalm; i0 += (long long)st.T * gridDim.x) {
        const int nt = (int)min((long long)st.T, nalm - i0);
        for (int b0 = 0; b0 < nmaps; b0 += st.MB) {
            const int mb = min(st.MB, nmaps - b0);
            for (int e = threadIdx.x; e < nt * mb; e += blockDim.x) {
                const int t = e / mb, b = e - t * mb;
                tile[b * (st.T + 1) + t] = aacc[(size_t)(i0 + t) * columns + b0 + b];
            }
            __syncthreads();
            for (int e = threadIdx.x; e < nt * mb; e += blockDim.x) {
                const int b = e / nt, t = e - b * nt;
                alm[(size_t)(b0 + b) * nalm + i0 + t] = scaled(tile[b * (st.T + 1) + t], i0 + t);
            }
            __syncthreads();
        }
    }
}

template <int NB>
int run_adj_group(const shtb_plan_s *p, const double2 *g, int nmaps, int b0, double *u0, double *u1,
                  double2 *aacc, cudaStream_t st)
{
    const BfPlanDev &bf = *p->bf;
    for (int lev = 1; lev <= bf.depth_max; ++lev) {
        const int n = bf.level_counts[lev - 1];
        if (n == 0) continue;
        const double *uin = ((lev - 1) % 2) ? u1 : u0;
        double *uout = (lev % 2) ? u1 : u0;
        const unsigned grid = (unsigned)((n + kBfWarps - 1) / kBfWarps);
        const int maxnc = bf.level_maxnc[lev - 1];
        const size_t smem = sizeof(double) * kBfWarps * maxnc * 2 * NB;
        SHTB_CUDA_TRY(cudaFuncSetAttribute(bf_adj_level_kernel<NB>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        bf_adj_level_kernel<NB><<<grid, 32 * kBfWarps, smem, st>>>(bf.level_items[lev - 1], n, maxnc, bf.ints,
                                                                   bf.words(), uin, g, nmaps, b0, uout);
        SHTB_CUDA_TRY(cudaGetLastError());
        ++p->launches;
    }
    if (bf.n_rgroups > 0 && bf.rec) {
        const unsigned grid = (unsigned)((bf.n_rgroups + kBfWarps - 1) / kBfWarps);
        const size_t smem = sizeof(double) * kBfWarps * (32 * 33 + 32 * 2 * NB);
        SHTB_CUDA_TRY(cudaFuncSetAttribute(bf_adj_r_rec_kernel<NB>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        bf_adj_r_rec_kernel<NB><<<grid, 32 * kBfWarps, smem, st>>>(p->view, bf.rgroups, bf.n_rgroups, bf.ritems,
                                                                   bf.rstart, bf.ints, u0, u1, bf.depth_parity,
                                                                   g, nmaps, b0, aacc);
        SHTB_CUDA_TRY(cudaGetLastError());
        ++p->launches;
    } else if (bf.n_rgroups > 0) {
        const unsigned grid = (unsigned)((bf.n_rgroups + kBfWarps - 1) / kBfWarps);
        bf_adj_r_kernel<NB><<<grid, 32 * kBfWarps, 0, st>>>(p->view, bf.rgroups, bf.n_rgroups, bf.ritems,
                                                            bf.ints, bf.words(), u0, u1, bf.depth_parity, g,
                                                            nmaps, b0, aacc);
        SHTB_CUDA_TRY(cudaGetLastError());
        ++p->launches;
    }
    return SHTB_OK;
}

// ------------------------------------------------ stored elements as words
// One warp per block of rows x cols doubles (row-major), a lane per column:
// the column's largest element sets its exponent, then every element becomes
// its word (shtb_fix.h) in place.  Runs once, when a plan is built or read.
__device__ __forceinline__ void pack_block(double *blk, int rows, int cols, int lane, int *err)
{
    for (int c = lane; c < cols; c += 32) {
        double big = 0.0;
        bool bad = false;
        for (int r = 0; r < rows; ++r) {
            const double v = fabs(blk[(size_t)r * cols + c]);
            bad |= !(v < 1.8e308);
            big = fmax(big, v);
        }
        int E = 0;
        if (big > 0.0) frexp(big, &E);                 // 2^(E-1) <= big < 2^E
        else E = -shtb::kFixExpBias;
        if (bad || E > shtb::kFixExpMax) {
            *err = 1;
            continue;
        }
        E = max(E, -shtb::kFixExpBias);
        const double scale = shtb::pow2(54 - E);
        for (int r = 0; r < rows; ++r) {
            double *p = blk + (size_t)r * cols + c;
            const long long X = __double2ll_rn(*p * scale) * 16;
            *p = __longlong_as_double((long long)shtb::fix_word(X, E + shtb::kFixExpBias));
        }
    }
}

__global__ void pack_r_kernel(const BfRItem *__restrict__ items, int n, double *dbl, int *err)
{
    const int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (w < n) pack_block(dbl + items[w].data_off, items[w].nrows, items[w].k, threadIdx.x & 31, err);
}

__global__ void pack_level_kernel(const BfItem *__restrict__ items, int n, double *dbl, int *err)
{
    const int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (w >= 2 * n) return;
    const BfItem &it = items[w >> 1];
    const int s = w & 1;
    pack_block(dbl + it.T_off[s], it.k[s], it.nd[s], threadIdx.x & 31, err);
}

}  // namespace

int bf_pack_operator(shtb_plan_s *p)
{
    const BfPlanDev &bf = *p->bf;
    double *dbl = const_cast<double *>(bf.dbl);
    int *err = nullptr, bad = 0;
    SHTB_CUDA_TRY(cudaMalloc(&err, sizeof(int)));
    cudaError_t e = cudaMemset(err, 0, sizeof(int));
    if (e == cudaSuccess && !bf.rec && bf.n_ritems > 0) {
        pack_r_kernel<<<(unsigned)((bf.n_ritems + 7) / 8), 256>>>(bf.ritems, bf.n_ritems, dbl, err);
        e = cudaGetLastError();
    }
    for (int l = 0; l < bf.depth_max && e == cudaSuccess; ++l) {
        const int n = bf.level_counts[l];
        if (n == 0) continue;
        pack_level_kernel<<<(unsigned)((2LL * n + 7) / 8), 256>>>(bf.level_items[l], n, dbl, err);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(&bad, err, sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(err);
    if (e != cudaSuccess) return shtb_fail(SHTB_ECUDA, std::string("packing the operator: ") + cudaGetErrorString(e));
    if (bad) return shtb_fail(SHTB_ENOTSUP, "operator element not finite or above 2^64");
    return SHTB_OK;
}

size_t bf_workspace_bytes(const shtb_plan_s *p)
{
    if (!p->bf) return 0;
    const size_t entry = sizeof(double) * 16;   // up to 8 maps x (re, im) per group
    return (2 * (size_t)p->bf->u_entries + (size_t)p->bf->qt_entries) * entry + 512;
}

int launch_bf_synth(const shtb_plan_s *p, const double2 *alm, double2 *ai, void *ws, double *map,
                    int nmaps, cudaStream_t st, double *qt_out, bool padded)
{
    const BfPlanDev &bf = *p->bf;
    const size_t entry = 16;
    double *u0 = (double *)ws;
    double *u1 = u0 + (size_t)bf.u_entries * entry;
    double *qt_ws = u1 + (size_t)bf.u_entries * entry;
    const int columns = padded ? padded_maps(nmaps) : nmaps;
    // q^t of map b in the caller's array of [columns][2][nhalf][L+1] complex (Legendre stage alone)
    const size_t qt_map = (size_t)4 * p->nhalf * (p->lmax + 1);
    const int ev = profile_begin(const_cast<shtb_plan_s *>(p), st);
    bf_interleave_kernel<<<stage_grid(p, columns), 256, 0, st>>>(p->view, alm, ai, nmaps, columns,
                                                                 p->bf->rec ? p->view.coef : nullptr);
    SHTB_CUDA_TRY(cudaGetLastError());
    ++p->launches;
    profile_end(const_cast<shtb_plan_s *>(p), st, 4, ev);
    for (int b0 = 0; b0 < columns;) {
        const int nb = group_width(columns - b0), real = std::min(nb, nmaps - b0);
        const QtView qt = qt_out ? QtView{qt_out + (size_t)b0 * qt_map, padded ? qt_pack(nb) : 0}
                                 : QtView{qt_ws, qt_pack(nb)};
        int rc;
        switch (nb) {
        case 8: rc = run_group<8>(p, ai, columns, b0, real, u0, u1, qt, map, st); break;
        case 4: rc = run_group<4>(p, ai, columns, b0, real, u0, u1, qt, map, st); break;
        case 2: rc = run_group<2>(p, ai, columns, b0, real, u0, u1, qt, map, st); break;
        default: rc = run_group<1>(p, ai, columns, b0, real, u0, u1, qt, map, st); break;
        }
        if (rc) return rc;
        b0 += nb;
    }
    return SHTB_OK;
}

int launch_bf_synth_to_host(shtb_plan_s *p, const double2 *alm, double2 *ai, void *ws, double *map,
                            double *map_host, int nmaps, cudaStream_t st)
{
    constexpr int NCH = shtb_plan_s::kPhiChunks;
    if (!p->copy_stream) {
        SHTB_CUDA_TRY(cudaStreamCreateWithFlags(&p->copy_stream, cudaStreamNonBlocking));
        for (auto &e : p->chunk_ev) SHTB_CUDA_TRY(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    }
    const BfPlanDev &bf = *p->bf;
    const size_t entry = 16;
    double *u0 = (double *)ws;
    double *u1 = u0 + (size_t)bf.u_entries * entry;
    double *qt_ws = u1 + (size_t)bf.u_entries * entry;
    const int columns = padded_maps(nmaps);
    bf_interleave_kernel<<<stage_grid(p, columns), 256, 0, st>>>(p->view, alm, ai, nmaps, columns,
                                                                 p->bf->rec ? p->view.coef : nullptr);
    SHTB_CUDA_TRY(cudaGetLastError());
    ++p->launches;
    int rc = SHTB_OK;
    for (int b0 = 0; b0 < columns && !rc;) {
        const int nb = group_width(columns - b0), real = std::min(nb, nmaps - b0);
        const QtView qt{qt_ws, qt_pack(nb)};
        rc = launch_bf_legendre_group(p, ai, columns, b0, nb, u0, u1, qt, st);
        // ring stage chunk by chunk; each chunk's pixels go back while the
        // next chunk (or the next map group) computes
        auto copy_back = [&](int c) -> int {
            const long long p0 = p->chunk_pix[c], p1 = p->chunk_pix[c + 1];
            if (p1 == p0) return SHTB_OK;
            if (int bad = join_stream(p->copy_stream, st, p->chunk_ev[c])) return bad;
            for (int b = b0; b < b0 + real; ++b)
                SHTB_CUDA_TRY(cudaMemcpyAsync(map_host + (size_t)b * p->npix + p0, map + (size_t)b * p->npix + p0,
                                              sizeof(double) * (size_t)(p1 - p0), cudaMemcpyDeviceToHost,
                                              p->copy_stream));
            return SHTB_OK;
        };
        for (int c = 0; c < NCH && !rc; ++c) {
            rc = launch_phi_synth_qt_chunk(p, qt, real, map, b0, c, st);
            if (!rc) rc = copy_back(c);
        }
        b0 += nb;
    }
    // the caller's stream completes after the last copy, also when a launch failed
    const int joined = join_stream(st, p->copy_stream, p->chunk_ev[0]);
    return rc ? rc : joined;
}

int launch_bf_adjoint(const shtb_plan_s *p, const double2 *g, double2 *aacc, void *ws, double2 *alm,
                      int nmaps, int columns, cudaStream_t st)
{
    const BfPlanDev &bf = *p->bf;
    const size_t entry = 16;
    double *u0 = (double *)ws;
    double *u1 = u0 + (size_t)bf.u_entries * entry;
    for (int b0 = 0; b0 < columns;) {
        const int nb = group_width(columns - b0);
        int rc;
        switch (nb) {
        case 8: rc = run_adj_group<8>(p, g, columns, b0, u0, u1, aacc, st); break;
        case 4: rc = run_adj_group<4>(p, g, columns, b0, u0, u1, aacc, st); break;
        case 2: rc = run_adj_group<2>(p, g, columns, b0, u0, u1, aacc, st); break;
        default: rc = run_adj_group<1>(p, g, columns, b0, u0, u1, aacc, st); break;
        }
        if (rc) return rc;
        b0 += nb;
    }
    bf_finish_kernel<<<stage_grid(p, nmaps), 256, 0, st>>>(p->view, aacc, alm, nmaps, columns,
                                                           p->bf->rec ? p->view.coef : nullptr);
    SHTB_CUDA_TRY(cudaGetLastError());
    ++p->launches;
    return SHTB_OK;
}

int launch_bf_gather(const shtb_plan_s *p, const double2 *const *alm_of_map, double2 *ai, int nmaps,
                     cudaStream_t st)
{
    bf_gather_kernel<<<p->lmax + 1, 256, 0, st>>>(p->view, alm_of_map, ai, nmaps);
    SHTB_CUDA_TRY(cudaGetLastError());
    ++p->launches;
    return SHTB_OK;
}

int launch_bf_legendre_group(const shtb_plan_s *p, const double2 *ai, int nmaps, int b0, int nb, double *u0,
                             double *u1, QtView qt, cudaStream_t st)
{
    int rc;
    switch (nb) {
    case 8: if ((rc = launch_r<8>(p, ai, nmaps, b0, u0, u1, qt, st))) return rc;
            return launch_levels<8>(p, u0, u1, qt, st);
    case 4: if ((rc = launch_r<4>(p, ai, nmaps, b0, u0, u1, qt, st))) return rc;
            return launch_levels<4>(p, u0, u1, qt, st);
    case 2: if ((rc = launch_r<2>(p, ai, nmaps, b0, u0, u1, qt, st))) return rc;
            return launch_levels<2>(p, u0, u1, qt, st);
    case 1: if ((rc = launch_r<1>(p, ai, nmaps, b0, u0, u1, qt, st))) return rc;
            return launch_levels<1>(p, u0, u1, qt, st);
    default: return shtb_fail(SHTB_EINVAL, "map group width must be 1, 2, 4 or 8");
    }
}
