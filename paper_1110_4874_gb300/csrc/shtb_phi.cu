// Kernel (c): the ring stage of Eq. (sh-baseline) -- per iso-latitude ring,
// the phase shift and wrap of Eq. (tau) followed by a backward real FFT of
// the ring's length J (Eq. pad-and-wrap), and its exact adjoint.
//
// With phi_kj = pi (2j + s)/J (s = 0 or 1) and q_{-m} = conj(q_m),
//   f_j = sum_{r=0}^{J-1} g_r e^{2 pi i r j / J},
//   g_r = sum_{m = r mod J, |m| <= L} q_m e^{i pi m s / J}
//       = e^{i pi r s / J} sum_t (-1)^{s t} q_{r + tJ}.
// g is Hermitian, so the real FFT of length J = 2K is done as one complex FFT
// of length K: Z_k = E_k + i e^{2 pi i k/J} O_k with E_k = g_k + g_{k+K},
// O_k = g_k - g_{k+K}; then z_n = sum_k Z_k e^{2 pi i k n / K} holds the
// pixels as f_{2n} + i f_{2n+1}.
// One CTA per (ring, map); the ring's data live in shared memory, as 64-bit
// fixed-point numbers (shtb_phi_items.cuh).  K factoring
// over 2, 3, 5, 7, 11, 13: in-place mixed-radix FFT (radices 4, 2, 3, 5, 7,
// 11, 13) from position-order input.  Otherwise Bluestein's chirp transform
// through a convolution of 7-smooth length M >= 2K-1 (decimation in
// frequency, pointwise product with a precomputed filter in position order,
// decimation in time), so no permutation pass is needed.
#include <cuda_runtime.h>

#include <vector>

#include "shtb_internal.h"
#include "shtb_phi_items.cuh"

namespace {

using namespace shtb_dev;

// most threads of a ring CTA: the Bluestein variant holds up to ~8.4k complex
// values of shared memory per CTA (one CTA per SM at the longest rings), so
// it runs twice the threads
template <int KIND>
constexpr int phi_threads()
{
    return KIND == kBluestein ? 512 : 256;
}

// CTAs per SM the ring kernels are compiled for: four of the common
// mixed-radix kind (64 registers; three, at 84, measured 1.20 against 1.14 ms
// for the ring stage of 8 maps at Nside = 512), two of the radix-11/13 kind
// and one of Bluestein's (128 registers)
template <int KIND>
constexpr int phi_min_blocks()
{
    return KIND == kDirect ? 4 : KIND == kDirectBig ? 2 : 1;
}

template <int KIND>
__global__ void __launch_bounds__(phi_threads<KIND>(), phi_min_blocks<KIND>())
phi_synth_kernel(PlanView v, const int *__restrict__ rings, const double2 *__restrict__ q,
                 double *__restrict__ map)
{
    extern __shared__ fx2 sm[];
    const int ring = rings[blockIdx.x];
    const int b = blockIdx.y;
    shtb_dev::phi_synth_ring<KIND, false>(v, ring, q + ((size_t)b * v.nrings + ring) * (v.lmax + 1),
                                          map + (size_t)b * v.npix + v.ring_start[ring], sm);
}

// ring stage of a compressed plan's map group, straight from the parity
// halves q^0, q^1 of the butterfly output (no separate combine pass)
// maps: either stacked at map + (b0 + b) npix, or one pointer per map
struct MapOut {
    double *map;
    double *const *table;
};

template <int KIND>
__global__ void __launch_bounds__(phi_threads<KIND>(), phi_min_blocks<KIND>())
phi_synth_qt_kernel(PlanView v, const int *__restrict__ rings, const double2 *__restrict__ qt,
                    int lp, MapOut mo, int b0)
{
    extern __shared__ fx2 sm[];
    const int ring = rings[blockIdx.x];
    const int b = blockIdx.y;
    double *base = mo.table ? mo.table[b0 + b] : mo.map + (size_t)(b0 + b) * v.npix;
    shtb_dev::phi_synth_ring_qt<KIND, false>(v, ring, qt, lp, b, base + v.ring_start[ring], sm);
}

template <int KIND>
__global__ void __launch_bounds__(phi_threads<KIND>(), phi_min_blocks<KIND>())
phi_adjoint_kernel(PlanView v, const int *__restrict__ rings, const double *__restrict__ map,
                   double2 *__restrict__ qa)
{
    extern __shared__ fx2 sm[];
    const int ring = rings[blockIdx.x];
    const int b = blockIdx.y;
    shtb_dev::phi_adjoint_ring<KIND>(v, ring, map + (size_t)b * v.npix + v.ring_start[ring],
                                     qa + ((size_t)b * v.nrings + ring) * (v.lmax + 1), sm);
}

// one launch per ring kind: grid (rings of that kind) x maps, shared memory
// for the kind's longest transform.  The Bluestein list is cut in two:
// rings [0, split) at phi_threads (one CTA per SM at the longest lengths),
// rings [split, n) -- transforms of at most kBlueSmallM points -- with fewer
// threads and with shared memory for their own longest transform, so that two
// or more CTAs share an SM and one's barriers between FFT passes are covered
// by the others' work.  Every body loops over blockDim.x.
// shared memory of a transform of `len` entries: the points and, while a
// spectrum is folded, a 16-bit exponent for each
size_t ring_smem_bytes(int len) { return (sizeof(fx2) + sizeof(short)) * (size_t)len + 16; }

struct RingSet {
    const int *rings;
    int n, len;
    int split, len_small;
};

RingSet ring_set(const shtb_plan_s *p, int kind)
{
    if (kind == kDirect)
        return {p->d_direct_rings, (int)p->direct_rings.size(), p->max_K_direct, (int)p->direct_rings.size(), 0};
    if (kind == kBluestein)
        return {p->d_blue_rings, (int)p->blue_rings.size(), p->max_M_mx, p->blue_split, p->max_M_small};
    return {p->d_big_rings, (int)p->big_rings.size(), p->max_K_big, (int)p->big_rings.size(), 0};
}

// Half the threads where no ring of the plan's kind is long: a radix-r pass
// over K points is K / r butterflies, which leaves most of 256 threads idle at
// each barrier, and twice the CTAs share an SM.  Ring stage of 8 maps, 256
// threads -> 128: Nside = 256 .346 -> .314 ms, 512 1.029 -> .915, 640 1.529 ->
// 1.395, 768 2.171 -> 2.056; 1024 3.748 -> 3.999, so the line lies between
// the longest rings of the last two (direct K 1536 and 2048).  The plan's
// longest ring decides, not the launch's, so that parts of a plan's rings
// take the same sums as the whole.
template <int KIND>
int part_threads(const shtb_plan_s *p, bool small)
{
    if (KIND == kBluestein)
        return !small ? phi_threads<KIND>() : p->max_M_small <= 3072 ? 128 : 256;
    return (KIND == kDirect ? p->max_K_direct <= 1536 : p->max_K_big <= 3072) ? 128 : phi_threads<KIND>();
}

// launch(rings, n, threads, smem bytes) for each non-empty part of rs
template <int KIND, class Launch>
int launch_parts(const shtb_plan_s *p, const RingSet &rs, const void *kernel, Launch launch)
{
    if (rs.n == 0) return SHTB_OK;
    SHTB_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)ring_smem_bytes(rs.len)));
    if (rs.split > 0) {
        launch(rs.rings, rs.split, part_threads<KIND>(p, false), ring_smem_bytes(rs.len));
        SHTB_CUDA_TRY(cudaGetLastError());
        ++p->launches;
    }
    if (rs.split < rs.n) {
        launch(rs.rings + rs.split, rs.n - rs.split, part_threads<KIND>(p, true),
               ring_smem_bytes(rs.len_small));
        SHTB_CUDA_TRY(cudaGetLastError());
        ++p->launches;
    }
    return SHTB_OK;
}

template <int KIND>
int launch_kind(const shtb_plan_s *p, bool synth, const void *in, void *out, int nmaps, cudaStream_t st)
{
    const RingSet rs = ring_set(p, KIND);
    const PlanView v = p->view;
    if (synth)
        return launch_parts<KIND>(p, rs, (const void *)phi_synth_kernel<KIND>,
                                  [&](const int *rings, int n, int threads, size_t smem) {
                                      phi_synth_kernel<KIND><<<dim3((unsigned)n, (unsigned)nmaps), threads, smem,
                                                               st>>>(v, rings, (const double2 *)in, (double *)out);
                                  });
    return launch_parts<KIND>(p, rs, (const void *)phi_adjoint_kernel<KIND>,
                              [&](const int *rings, int n, int threads, size_t smem) {
                                  phi_adjoint_kernel<KIND><<<dim3((unsigned)n, (unsigned)nmaps), threads, smem,
                                                             st>>>(v, rings, (const double *)in, (double2 *)out);
                              });
}

// The three ring kinds read and write disjoint rings, so they run side by
// side: the Bluestein rings on the caller's stream, the direct and the
// radix-11/13 or Rader rings on two plan-owned streams forked from it and
// joined back, and each launch's last wave overlaps the others' work.
// blue, direct, big: launch the kind on the stream they are given.
template <class Blue, class Direct, class Big>
int side_by_side(const shtb_plan_s *p, cudaStream_t st, Blue blue, Direct direct, Big big)
{
    shtb_plan_s *pp = const_cast<shtb_plan_s *>(p);
    if (int rs = side_streams(pp)) return rs;
    return fork_join(st, pp->ring_stream, pp->ring_ev, 2, [&] {
        int rc = blue(st);
        if (!rc) rc = direct(pp->ring_stream[0]);
        return rc ? rc : big(pp->ring_stream[1]);
    });
}

int launch_set(const shtb_plan_s *p, bool synth, const void *in, void *out, int nmaps,
               cudaStream_t st, bool one_stream)
{
    if (one_stream) {
        int rc;
        if ((rc = launch_kind<kBluestein>(p, synth, in, out, nmaps, st))) return rc;
        if ((rc = launch_kind<kDirect>(p, synth, in, out, nmaps, st))) return rc;
        return launch_kind<kDirectBig>(p, synth, in, out, nmaps, st);
    }
    return side_by_side(
        p, st, [&](cudaStream_t s2) { return launch_kind<kBluestein>(p, synth, in, out, nmaps, s2); },
        [&](cudaStream_t s2) { return launch_kind<kDirect>(p, synth, in, out, nmaps, s2); },
        [&](cudaStream_t s2) { return launch_kind<kDirectBig>(p, synth, in, out, nmaps, s2); });
}

template <int KIND>
int launch_qt_set(const shtb_plan_s *p, QtView qt, int nb, MapOut map, int b0, const RingSet &rs,
                  cudaStream_t st)
{
    const PlanView v = p->view;
    return launch_parts<KIND>(p, rs, (const void *)phi_synth_qt_kernel<KIND>,
                              [&](const int *rings, int n, int threads, size_t smem) {
                                  phi_synth_qt_kernel<KIND><<<dim3((unsigned)n, (unsigned)nb), threads, smem, st>>>(
                                      v, rings, (const double2 *)qt.q, qt.lp, map, b0);
                              });
}

template <int KIND>
int launch_qt_kind(const shtb_plan_s *p, QtView qt, int nb, MapOut map, int b0, cudaStream_t st)
{
    return launch_qt_set<KIND>(p, qt, nb, map, b0, ring_set(p, KIND), st);
}

template <int KIND>
int launch_qt_list(const shtb_plan_s *p, QtView qt, int nb, MapOut map, int b0,
                   const shtb_plan_s::ChunkKind &ck, cudaStream_t st)
{
    return launch_qt_set<KIND>(p, qt, nb, map, b0, RingSet{p->d_chunk_list + ck.off, ck.n, ck.len,
                                                           KIND == kBluestein ? ck.split : ck.n, ck.len_small}, st);
}

int launch_qt_all(const shtb_plan_s *p, QtView qt, int nb, MapOut mo, int b0, cudaStream_t st)
{
    int rc;
    if ((rc = launch_qt_kind<kBluestein>(p, qt, nb, mo, b0, st))) return rc;
    if ((rc = launch_qt_kind<kDirect>(p, qt, nb, mo, b0, st))) return rc;
    return launch_qt_kind<kDirectBig>(p, qt, nb, mo, b0, st);
}

// Tables from doubles to halves, in place
__global__ void ring_pack_kernel(double2 *t, size_t n, int bits)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const double2 v = t[i];
        const int2 re = shtb_dev::ring_half_pack(v.x, bits), im = shtb_dev::ring_half_pack(v.y, bits);
        reinterpret_cast<int4 *>(t)[i] = make_int4(re.x, re.y, im.x, im.y);
    }
}

}  // namespace

int side_streams(shtb_plan_s *p)
{
    if (p->ring_stream[0]) return SHTB_OK;
    for (auto &s2 : p->ring_stream) SHTB_CUDA_TRY(cudaStreamCreateWithFlags(&s2, cudaStreamNonBlocking));
    for (auto &e : p->ring_ev) SHTB_CUDA_TRY(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    return SHTB_OK;
}

int launch_phi_synth_qt(const shtb_plan_s *p, QtView qt, int nb, double *map, int b0,
                        cudaStream_t st)
{
    const MapOut mo{map, nullptr};
    return side_by_side(
        p, st, [&](cudaStream_t s2) { return launch_qt_kind<kBluestein>(p, qt, nb, mo, b0, s2); },
        [&](cudaStream_t s2) { return launch_qt_kind<kDirect>(p, qt, nb, mo, b0, s2); },
        [&](cudaStream_t s2) { return launch_qt_kind<kDirectBig>(p, qt, nb, mo, b0, s2); });
}

int launch_phi_synth_qt_chunk(const shtb_plan_s *p, QtView qt, int nb, double *map, int b0, int chunk,
                              cudaStream_t st)
{
    const MapOut mo{map, nullptr};
    const auto *ck = p->chunk_kind[chunk];
    int rc;
    if ((rc = launch_qt_list<kBluestein>(p, qt, nb, mo, b0, ck[1], st))) return rc;
    if ((rc = launch_qt_list<kDirect>(p, qt, nb, mo, b0, ck[0], st))) return rc;
    return launch_qt_list<kDirectBig>(p, qt, nb, mo, b0, ck[2], st);
}

int launch_phi_synth_qt_ptr(const shtb_plan_s *p, QtView qt, int nb, double *const *map_of_map,
                            int b0, cudaStream_t st)
{
    return launch_qt_all(p, qt, nb, MapOut{nullptr, map_of_map}, b0, st);
}

int launch_phi_synth(const shtb_plan_s *p, const double2 *q, double *map, int nmaps, cudaStream_t st, bool one_stream)
{
    return launch_set(p, true, q, map, nmaps, st, one_stream);
}

int launch_phi_adjoint(const shtb_plan_s *p, const double *map, double2 *q, int nmaps,
                       cudaStream_t st)
{
    return launch_set(p, false, map, q, nmaps, st, false);
}

std::vector<RingTable> ring_tables(const shtb_plan_s *p)
{
    const PlanView &v = p->view;
    return {{v.tw, shtb::kRootBits}, {v.mtw, shtb::kRootBits}, {v.mfb, shtb::kRootBits},
            {v.rdr_dbl, shtb::kRootBits}, {v.ab, shtb::kFoldBits}};
}

int ring_pack_tables(shtb_plan_s *p)
{
    for (const RingTable &t : ring_tables(p))
        for (size_t i = 0; i < p->allocations.size(); ++i) {
            if (p->allocations[i] != (const void *)t.table) continue;
            ring_pack_kernel<<<152 * 4, 256>>>((double2 *)p->allocations[i], p->alloc_bytes[i] / sizeof(double2), t.bits);
            SHTB_CUDA_TRY(cudaGetLastError());
        }
    SHTB_CUDA_TRY(cudaDeviceSynchronize());
    return SHTB_OK;
}
