// Per-work-item device bodies of the butterfly synthesis (Sec. 3.2) used by
// the stage kernels of shtb_butterfly.cu and by the persistent batch kernel
// of shtb_batch.cu.  One warp per item.  CG = true reads data through L2
// only (ld.global.cg), for data produced earlier in the same launch: L1 is
// not coherent between SMs within one launch.
#pragma once

#include <cuda_runtime.h>

#include "shtb_bf_fix.cuh"
#include "shtb_butterfly.h"

namespace shtb_dev {

__device__ __forceinline__ long long alm_off(int L, int m)
{
    return (long long)m * (2 * L + 1 - m) / 2 + m;
}

// q^t of a map group (QtView): the ring stage reads each map's q_m of one
// ring along m, the items write all maps of one entry e = (m * 2 + t) * nhalf + r.
// Entries fit 32 bits (e < 2 (L + 1) nhalf), so the split of e runs as a
// 32-bit division.
__device__ __forceinline__ size_t qt_index(int e, int nhalf, int L, int lp, int c)
{
    const unsigned mt = (unsigned)e / (unsigned)nhalf, r = (unsigned)e - mt * (unsigned)nhalf;
    const unsigned m = mt >> 1, t = mt & 1;
    const unsigned b = (unsigned)c >> 1, pack = b >> lp;
    return ((((((size_t)pack * 2 + t) * nhalf + r) * (L + 1) + m) << lp) + (b - (pack << lp))) * 2 + (c & 1);
}

// Every output of a residual block (one column) and of a level child (one
// dense row) is one block product of shtb_bf_fix.cuh, the same bits at every
// map-group width; in a level item the first child's outputs are stored and
// the second child's added.  So a map's result does not depend on how maps
// are grouped.

// ---- residual blocks: chain rows of a_lm contracted with R's columns
template <bool CG>
struct ResVec {
    const double *a0;                   // component 0 of the block's first chain row
    int astride;                        // doubles between chain rows
    template <int W>
    __device__ __forceinline__ void load(int k, int i, double (&x)[W]) const
    {
        ld_comps<CG ? Ld::kL2 : Ld::kGlobal>(a0 + (size_t)k * astride, i, x);
    }
    __device__ __forceinline__ int shift(int) const { return 0; }
};

template <int C>
struct ResOut {
    double *dst;                        // u entries of the block, or null: q^t entries ent
    const int *ent;
    QtView qt;
    int nhalf, L;
    __device__ __forceinline__ int key(int n) const { return dst ? n : __ldg(ent + n); }
    template <int W>
    __device__ __forceinline__ void put(int n, bool add, int i, const double (&v)[W]) const
    {
        if (dst) st_comps(dst + (size_t)n * C, i, v, add);
        else st_comps(qt.q + qt_index(n, nhalf, L, qt.lp, W * i), 0, v, add);
    }
};

// u = R^T a over one residual block.  ai: [idx][nmaps] complex, the group's
// maps at b0 .. b0+NB-1; chain row j of (m, t) is a_{m+t+2j}.
template <int NB, bool CG>
__device__ __forceinline__ void bf_r_item(const BfRItem &it, int L, int nhalf, const int *__restrict__ ints,
                                          const uint2 *__restrict__ words, const double2 *ai, int nmaps,
                                          int b0, double *ubuf, QtView qt, int lane)
{
    constexpr int C = 2 * NB;
    const long long aoff = alm_off(L, it.m) + it.t + 2 * it.j0;       // chain row j at aoff + 2j
    const ResVec<CG> vec{reinterpret_cast<const double *>(ai + (size_t)aoff * nmaps + b0), 4 * nmaps};
    const ResOut<C> out{it.to_rings ? nullptr : ubuf + (size_t)it.out_off * C, it.to_rings ? ints + it.out_off : nullptr,
                        qt, nhalf, L};
    if (it.nrows == 0) {                // a block without rows (a cropped chain range) writes zeros
        const double z[1] = {0.0};
        for (int i = lane; i < it.k * C; i += 32) out.put(out.key(i / C), false, i % C, z);
        return;
    }
    fix_product<C, true>(words + it.data_off, it.k, 1, it.nrows, it.k, vec, out, lane);
}

// ---- level items: v = T_top^T u_top + T_bot^T u_bot over the shared
// candidate list, written to the parent level's u (or to q^t at level 1).
// scr: this warp's shared-memory scratch of nc x C doubles.

// a child's u entries, which are also its identity entries: reading one
// stores it (or adds it, second child) at its candidate position
template <int C, bool CG>
struct LevelVec {
    const double *u;
    const int *ipos;
    double *scr;
    bool second;
    template <int W>
    __device__ __forceinline__ void load(int k, int i, double (&x)[W]) const
    {
        ld_comps<CG ? Ld::kL2 : Ld::kGlobal>(u + (size_t)k * C, i, x);
        st_comps(scr + __ldg(ipos + k) * C, i, x, second);
    }
    __device__ __forceinline__ int shift(int) const { return 0; }
};

template <int C>
struct LevelOut {
    const int *dpos;
    double *scr;
    bool second;
    __device__ __forceinline__ int key(int n) const { return __ldg(dpos + n); }
    template <int W>
    __device__ __forceinline__ void put(int pos, bool add, int i, const double (&v)[W]) const
    {
        st_comps(scr + pos * C, i, v, second || add);
    }
};

// A child's dense and identity positions are distinct, so lanes never update
// the same scratch entry within a child; the warp syncs between the children,
// whose positions may coincide.
// RING: 1 when every item of the launch writes q^t (the plan's level 1), 0
// when none does, -1 to follow each item's to_rings flag.
template <int NB, bool CG, int RING = -1>
__device__ __forceinline__ void bf_level_item(const BfItem &it, int L, int nhalf, const int *__restrict__ ints,
                                              const uint2 *__restrict__ words, const double *uin,
                                              double *uout, QtView qt, double *scr, int lane)
{
    constexpr int C = 2 * NB;
    double2 *scr2 = reinterpret_cast<double2 *>(scr);
    for (int i = lane; i < it.nc * NB; i += 32) scr2[i] = make_double2(0.0, 0.0);
    __syncwarp();
#pragma unroll 1
    for (int s = 0; s < 2; ++s) {
        const LevelVec<C, CG> vec{uin + (size_t)it.u_off[s] * C, ints + it.ipos_off[s], scr, s == 1};
        const LevelOut<C> out{ints + it.dpos_off[s], scr, s == 1};
        fix_product<C, true>(words + it.T_off[s], it.nd[s], 1, it.k[s], it.nd[s], vec, out, lane);
        __syncwarp();
    }
    if (RING == 1 || (RING < 0 && it.to_rings)) {
        // the entries of an item share (m, t); those of a lane share the map
        const int *__restrict__ ent = ints + it.out_off;
        const int e0 = __ldg(ent);
        double2 *q0 = reinterpret_cast<double2 *>(qt.q + qt_index(e0, nhalf, L, qt.lp, 2 * (lane % NB)));
        const size_t ring = (size_t)(L + 1) << qt.lp;
#pragma unroll 4
        for (int i = lane / NB; i < it.nc; i += 32 / NB)
            q0[(__ldg(ent + i) - e0) * (long long)ring] = scr2[i * NB + lane % NB];
    } else {
        double2 *dst = reinterpret_cast<double2 *>(uout + (size_t)it.out_off * C);
        for (int i = lane; i < it.nc * NB; i += 32) dst[i] = scr2[i];
    }
    __syncwarp();
}

}  // namespace shtb_dev
