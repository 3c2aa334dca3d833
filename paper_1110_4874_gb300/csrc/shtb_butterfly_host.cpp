// Butterfly compression of the per-(m, parity) Legendre matrices (Sec. 3.2)
// and its serialisation into flat work-item lists for the apply kernels.
//
// Lambda^{m,t} has rows j (l = m + t + 2j) and columns r (rings with z >= 0);
// synthesis needs q^t = Lambda^T a.  Columns are cut into 2^D leaf blocks of
// leaf_cols rings.  Level 1 splits the rows in two halves and takes the
// interpolative decomposition (ID, Eq. ID) of every (row half, leaf block)
// block; level l joins the skeletons of two neighbouring column groups of the
// parent row interval (Eq. joinsplit), halves the rows again and takes IDs
// again.  After p levels the residual R holds, for every (row interval,
// column group), the block Lambda[I, skeleton]; Eq. factor-into-block-
// diagonal gives Lambda = R S_p P_{p-1} ... P_1 S_1.
//
// Applying Lambda^T (synthesis): u(p, I, G) = R(I, G)^T a_I; then for l = p..1
// the two row-children I, I' of a parent interval share one candidate set C
// (the two child groups' skeletons at the parent), and
//   v_C = T(l, I, G)^T u(l, I, G) + T(l, I', G)^T u(l, I', G)
// gives u(l-1, parent, G_a) ++ u(l-1, parent, G_b) (at l = 1: q^t on the leaf
// block).  T has the identity on the skeleton positions (Appendix: filter
// into an identity part and a dense part) and a dense k x (|C| - k) part.
//
// On GB300 the FP64 pipe is the only bound (about 0.19 flop per byte of HBM),
// so the residual blocks are stored, not regenerated by recurrence (a stored
// element costs 2 FMAs per map, a recurrence step 2 more), and the depth p of
// each (m, parity) is the one that minimises stored elements plus identity
// entries -- the paper's rho trade-off (Sec. 3.3, 4.2) with rho = 1.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <numeric>
#include <string>
#include <vector>

#include "shtb_butterfly.h"
#include "shtb_id_gpu.h"
#include "shtb_plan_detail.h"

namespace shtb {

// ----------------------------------------------------------- the ID
// Interpolative decomposition of the rows x n block A (column-major, leading
// dimension lda) by Householder QR with column pivoting, truncated once the
// largest remaining column norm falls to eps times the first pivot (or to the
// absolute floor): A[:, C] ~= A[:, skel] * [I | T] (Cheng, Gimbutas,
// Martinsson & Rokhlin 2005; error bound Eq. ID-approximation).  Columns whose
// norm is at or below the floor are "zero" columns (in the 1e-30 crop).
IdResult interp_decomp(const double *A, int rows, int n, int lda, double eps, double abs_floor)
{
    IdResult res;
    res.kind.assign(n, kZeroCol);
    std::vector<int> nz;
    for (int c = 0; c < n; ++c) {
        double s = 0.0;
        for (int r = 0; r < rows; ++r) s += A[(size_t)c * lda + r] * A[(size_t)c * lda + r];
        if (std::sqrt(s) > abs_floor) nz.push_back(c);
    }
    const int nzc = (int)nz.size();
    if (nzc == 0 || rows == 0) {
        res.k = 0;
        return res;
    }
    std::vector<double> W((size_t)rows * nzc);
    for (int j = 0; j < nzc; ++j)
        std::memcpy(&W[(size_t)j * rows], &A[(size_t)nz[j] * lda], sizeof(double) * rows);
    std::vector<double> norms(nzc), ref(nzc);
    std::vector<int> perm(nzc);
    std::iota(perm.begin(), perm.end(), 0);
    auto exact_norm2 = [&](int j, int from) {
        double s = 0.0;
        const double *col = &W[(size_t)j * rows];
        for (int r = from; r < rows; ++r) s += col[r] * col[r];
        return s;
    };
    for (int j = 0; j < nzc; ++j) ref[j] = norms[j] = exact_norm2(j, 0);
    std::vector<double> v(rows);
    int k = 0;
    double r00 = 0.0;
    const int kmax = std::min(rows, nzc);
    for (int i = 0; i < kmax; ++i) {
        int p = i;
        for (int j = i + 1; j < nzc; ++j)
            if (norms[j] > norms[p]) p = j;
        double n2 = exact_norm2(p, i);
        norms[p] = n2;
        const double nrm = std::sqrt(n2);
        if (i == 0) r00 = nrm;
        if (nrm <= std::max(eps * r00, abs_floor)) break;
        if (p != i) {
            std::swap_ranges(&W[(size_t)p * rows], &W[(size_t)p * rows] + rows, &W[(size_t)i * rows]);
            std::swap(norms[p], norms[i]);
            std::swap(ref[p], ref[i]);
            std::swap(perm[p], perm[i]);
        }
        double *ci = &W[(size_t)i * rows];
        const double x0 = ci[i];
        const double alpha = x0 >= 0 ? -nrm : nrm;
        for (int r = i; r < rows; ++r) v[r] = ci[r];
        v[i] -= alpha;
        const double vnorm2 = 2.0 * nrm * (nrm + std::fabs(x0));
        const double beta = vnorm2 > 0 ? 2.0 / vnorm2 : 0.0;
        for (int j = i + 1; j < nzc; ++j) {
            double *cj = &W[(size_t)j * rows];
            double s = 0.0;
            for (int r = i; r < rows; ++r) s += v[r] * cj[r];
            s *= beta;
            for (int r = i; r < rows; ++r) cj[r] -= s * v[r];
            norms[j] -= cj[i] * cj[i];
            if (norms[j] <= 1e-8 * ref[j]) ref[j] = norms[j] = exact_norm2(j, i + 1);
        }
        ci[i] = alpha;
        for (int r = i + 1; r < rows; ++r) ci[r] = 0.0;
        k = i + 1;
    }
    res.k = k;
    // T = R11^{-1} R12 by back substitution, one dense column at a time
    const int nd = nzc - k;
    std::vector<std::pair<int, int>> dense;   // (cand position, W column)
    for (int c = k; c < nzc; ++c) dense.push_back({nz[perm[c]], c});
    std::sort(dense.begin(), dense.end());
    res.skel.resize(k);
    for (int i = 0; i < k; ++i) {
        res.skel[i] = nz[perm[i]];
        res.kind[res.skel[i]] = i;
    }
    res.T.assign((size_t)k * nd, 0.0);
    res.dense_pos.resize(nd);
    std::vector<double> x(k);
    for (int d = 0; d < nd; ++d) {
        const int c = dense[d].second;
        res.dense_pos[d] = dense[d].first;
        res.kind[dense[d].first] = -1 - d;
        for (int i = k - 1; i >= 0; --i) {
            double s = W[(size_t)c * rows + i];
            for (int q = i + 1; q < k; ++q) s -= W[(size_t)q * rows + i] * x[q];
            x[i] = s / W[(size_t)i * rows + i];
        }
        for (int i = 0; i < k; ++i) res.T[(size_t)i * nd + d] = x[i];
    }
    return res;
}

// ------------------------------------------------- compress one (m, t)
namespace {

int ceil_log2(long long x)
{
    int d = 0;
    while ((1LL << d) < x) ++d;
    return d;
}

struct Node {
    int r0 = 0, r1 = 0;            // chain rows [r0, r1)
    std::vector<int> cand;         // candidate columns (rings)
    IdResult id;
    std::vector<int> skel_cols;    // rings of the skeleton, in u order
};

struct Level {
    int nI = 0, nG = 0;
    std::vector<Node> nodes;       // index I * nG + g
};

}  // namespace

// Compresses Lambda (n rows x Z columns, column-major, column c holds
// P_{m+t+2j}^m(z_c) for j < n) and fills `out` with the chosen depth's items
// in local (per-(m, t)) offsets.
int compress_chain(const double *Lam, int n, int Z, const BfParams &prm, BfChain *out)
{
    out->n = n;
    out->depth = 0;
    const int w = prm.leaf_cols;
    const long long nleaf = (Z + w - 1) / w;
    const int D = ceil_log2(nleaf);
    const long long npad = 1LL << D;
    std::vector<int> first_nz(Z, n);   // first non-zero row of each column
    for (int c = 0; c < Z; ++c) {
        const double *col = Lam + (size_t)c * n;
        int j = 0;
        while (j < n && col[j] == 0.0) ++j;
        first_nz[c] = j;
    }
    // cost of stopping at level 0: whole leaf columns from their first non-zero row
    long long best_cost = 0;
    for (long long b = 0; b < nleaf; ++b) {
        int c0 = (int)(b * w), c1 = (int)std::min<long long>(Z, c0 + w);
        int mn = n;
        for (int c = c0; c < c1; ++c) mn = std::min(mn, first_nz[c]);
        best_cost += (long long)(n - mn) * (c1 - c0);
    }
    int best_depth = 0;
    std::vector<Level> levels;
    long long s_cum = 0;
    const int max_depth = prm.max_depth >= 0 ? std::min(prm.max_depth, D + 1) : D + 1;
    if (n > 0) {
        // row intervals, level by level (larger half on top)
        std::vector<std::vector<std::pair<int, int>>> rows(1, {{0, n}});
        for (int lev = 1; lev <= max_depth; ++lev) {
            std::vector<std::pair<int, int>> next;
            for (auto &iv : rows.back()) {
                int mid = iv.first + (iv.second - iv.first + 1) / 2;
                next.push_back({iv.first, mid});
                next.push_back({mid, iv.second});
            }
            rows.push_back(next);
            Level L;
            L.nI = 1 << lev;
            L.nG = (int)(npad >> (lev - 1));
            L.nodes.resize((size_t)L.nI * L.nG);
            bool too_wide = false;
            for (int I = 0; I < L.nI; ++I) {
                for (int g = 0; g < L.nG; ++g) {
                    Node &nd = L.nodes[(size_t)I * L.nG + g];
                    nd.r0 = rows[lev][I].first;
                    nd.r1 = rows[lev][I].second;
                    if (lev == 1) {
                        for (long long c = (long long)g * w; c < std::min<long long>(Z, (long long)g * w + w); ++c)
                            nd.cand.push_back((int)c);
                    } else {
                        const Level &up = levels.back();
                        const int P = I / 2;
                        const Node &a = up.nodes[(size_t)P * up.nG + 2 * g];
                        const Node &b = up.nodes[(size_t)P * up.nG + 2 * g + 1];
                        nd.cand = a.skel_cols;
                        nd.cand.insert(nd.cand.end(), b.skel_cols.begin(), b.skel_cols.end());
                    }
                    if ((int)nd.cand.size() > kMaxCand) too_wide = true;
                }
            }
            if (too_wide) break;
            // IDs of every node of this level: the blocks gathered into one
            // array, then decomposed on the host or as one GPU batch
            long long s_lev = 0, r_lev = 0;
            std::vector<IdBlock> blocks;
            std::vector<Node *> owner;
            long long total = 0;
            for (auto &nd : L.nodes) {
                const int rr = nd.r1 - nd.r0, nc = (int)nd.cand.size();
                if (nc == 0) continue;
                blocks.push_back({total, rr, nc});
                owner.push_back(&nd);
                total += (long long)rr * nc;
            }
            // the GPU path gathers straight into its slot's pinned buffer
            std::vector<double> host_blk;
            double *blk = nullptr;
            if (prm.gpu) {
                blk = gpu_id_staging(prm.gpu, prm.slot, total);
                if (!blk) return shtb_fail(SHTB_ENOMEM, "plan build: pinned staging");
            } else {
                host_blk.resize((size_t)total);
                blk = host_blk.data();
            }
            for (size_t b = 0; b < blocks.size(); ++b) {
                const Node &nd = *owner[b];
                const int rr = blocks[b].rows;
                for (int c = 0; c < blocks[b].nc; ++c)
                    std::memcpy(blk + blocks[b].off + (size_t)c * rr, Lam + (size_t)nd.cand[c] * n + nd.r0,
                                sizeof(double) * rr);
            }
            if (prm.gpu) {
                std::vector<IdResult> ids;
                const int rc = gpu_id_run(prm.gpu, prm.slot, blk, total, blocks, prm.eps, prm.abs_floor, ids);
                if (rc) return rc;
                for (size_t b = 0; b < blocks.size(); ++b) owner[b]->id = std::move(ids[b]);
            } else {
                for (size_t b = 0; b < blocks.size(); ++b)
                    owner[b]->id = interp_decomp(blk + blocks[b].off, blocks[b].rows, blocks[b].nc,
                                                 blocks[b].rows, prm.eps, prm.abs_floor);
            }
            for (auto &nd : L.nodes) {
                if (nd.cand.empty()) continue;
                for (int s : nd.id.skel) nd.skel_cols.push_back(nd.cand[s]);
                s_lev += (long long)nd.id.k * (long long)nd.id.dense_pos.size() + nd.id.k;
                int mn = nd.r1;
                for (int c : nd.skel_cols) mn = std::min(mn, first_nz[c]);
                const int j0 = std::max(nd.r0, mn);
                if (nd.r1 > j0) r_lev += (long long)(nd.r1 - j0) * nd.id.k;
            }
            s_cum += s_lev;
            levels.push_back(std::move(L));
            const long long cost = s_cum + r_lev;
            if (cost < best_cost) {
                best_cost = cost;
                best_depth = lev;
            }
            if (cost > 2 * best_cost) break;   // compression has stopped paying
        }
    }
    // ---------------------------------------------------- emit the chosen depth
    const int p = best_depth;
    out->depth = p;
    out->cost = best_cost;
    // u offsets of level l nodes (l = 1..p), in (I, g) order; region = max level size
    std::vector<std::vector<long long>> uoff(p + 1);
    long long region = 0;
    for (int lev = 1; lev <= p; ++lev) {
        const Level &L = levels[lev - 1];
        uoff[lev].resize(L.nodes.size());
        long long o = 0;
        for (size_t q = 0; q < L.nodes.size(); ++q) {
            uoff[lev][q] = o;
            o += L.nodes[q].id.k;
        }
        region = std::max(region, o);
    }
    out->region = region;
    // residual blocks
    if (p == 0) {
        out->top_rows.push_back({0, n});
        for (long long b = 0; b < nleaf; ++b) {
            int c0 = (int)(b * w), c1 = (int)std::min<long long>(Z, c0 + w);
            int mn = n;
            for (int c = c0; c < c1; ++c) mn = std::min(mn, first_nz[c]);
            BfRLocal r;   // kept even when empty (nrows = 0): it writes the zeros of its rings
            r.j0 = mn;
            r.nrows = n - mn;
            r.k = c1 - c0;
            r.to_rings = true;
            for (int c = c0; c < c1; ++c) r.rings.push_back(c);
            r.cols = r.rings;
            r.data.resize((size_t)r.nrows * r.k);
            for (int j = 0; j < r.nrows; ++j)
                for (int s = 0; s < r.k; ++s) r.data[(size_t)j * r.k + s] = Lam[(size_t)(c0 + s) * n + mn + j];
            out->rblocks.push_back(std::move(r));
        }
        return SHTB_OK;
    }
    const Level &top = levels[p - 1];
    for (int I = 0; I < top.nI; ++I) {
        const Node &first = top.nodes[(size_t)I * top.nG];
        out->top_rows.push_back({first.r0, first.r1});
    }
    for (size_t q = 0; q < top.nodes.size(); ++q) {
        const Node &nd = top.nodes[q];
        if (nd.id.k == 0) continue;
        int mn = nd.r1;
        for (int c : nd.skel_cols) mn = std::min(mn, first_nz[c]);
        const int j0 = std::max(nd.r0, mn);
        BfRLocal r;
        r.interval = (int)(q / top.nG);
        r.j0 = j0;
        r.nrows = std::max(0, nd.r1 - j0);
        r.k = nd.id.k;
        r.to_rings = false;
        r.out_off = uoff[p][q];
        r.cols = nd.skel_cols;
        r.data.resize((size_t)r.nrows * r.k);
        for (int j = 0; j < r.nrows; ++j)
            for (int s = 0; s < r.k; ++s)
                r.data[(size_t)j * r.k + s] = Lam[(size_t)nd.skel_cols[s] * n + j0 + j];
        out->rblocks.push_back(std::move(r));
    }
    // level items: parent interval P (level l-1) x group g (level l), children 2P, 2P+1
    for (int lev = p; lev >= 1; --lev) {
        const Level &L = levels[lev - 1];
        const int nP = L.nI / 2;
        for (int P = 0; P < nP; ++P) {
            for (int g = 0; g < L.nG; ++g) {
                const Node &top_n = L.nodes[(size_t)(2 * P) * L.nG + g];
                const Node &bot_n = L.nodes[(size_t)(2 * P + 1) * L.nG + g];
                const int nc = (int)top_n.cand.size();
                if (nc == 0) continue;
                BfItemLocal it;
                it.level = lev;
                it.nc = nc;
                const Node *ch[2] = {&top_n, &bot_n};
                for (int s = 0; s < 2; ++s) {
                    const IdResult &id = ch[s]->id;
                    it.k[s] = id.k;
                    it.u_off[s] = id.k ? uoff[lev][(size_t)(2 * P + s) * L.nG + g] : 0;
                    it.dense_pos[s] = id.dense_pos;
                    it.ident_pos[s] = id.skel;
                    it.T[s] = id.T;
                }
                if (lev == 1) {
                    it.to_rings = true;
                    it.rings = top_n.cand;
                } else {
                    it.to_rings = false;
                    const Level &up = levels[lev - 2];
                    it.out_off = uoff[lev - 1][(size_t)P * up.nG + 2 * g];
                }
                out->items.push_back(std::move(it));
            }
        }
    }
    return SHTB_OK;
}

// Recurrence start of one residual-block column (rows j0 .. j0 + nrows - 1 of
// chain (m, t), half-ring ring with argument x): the chain's own start (js,
// V_js, V_js+1) past the 1e-30 crop when that falls inside the block, else
// V at rows j0 and j0 + 1, reached from the chain start by the same fused
// steps the kernels take (w = mu x + C, V_{j+1} = w V_j - V_{j-1}), so that a
// block continues the chain bit for bit.  cf: the coefficients of order m,
// indexed by l - m.
RecStart block_column_start(int n, int t, int j0, int nrows, int ring, double x, bool sform, const RecCoef *cf,
                            int js, double2 vs)
{
    RecStart st{ring, nrows, 0.0, 0.0};
    if (js >= n || js >= j0 + nrows) return st;        // zero throughout this block
    if (js >= j0) {
        st.start = js - j0;
        st.v0 = vs.x;
        st.v1 = vs.y;
        return st;
    }
    double prev = vs.x, cur = vs.y;                      // V_js, V_js+1
    for (int j = js + 1; j <= j0; ++j) {
        const RecCoef &c = cf[2 * j + t];
        const double w = std::fma(c.mu, x, sform ? c.cs : c.cz);
        const double nxt = std::fma(w, cur, -prev);
        prev = cur;
        cur = nxt;
    }
    st.start = 0;
    st.v0 = prev;                                        // V_j0
    st.v1 = cur;                                         // V_j0+1
    return st;
}

// Lambda^{m,t} for both parities of one m: column-major, n_t rows x Z columns.
void build_lambda(int L, int m, int Z, const std::vector<HalfRing> &hr, DD cm,
                  std::vector<double> &lam0, std::vector<double> &lam1)
{
    const int n0 = chain_len(L, m, 0), n1 = chain_len(L, m, 1);
    lam0.assign((size_t)n0 * Z, 0.0);
    lam1.assign((size_t)n1 * Z, 0.0);
    const std::vector<double> b = one_step_coefs(L, m);
    std::vector<double> col(L - m + 1);
    for (int r = 0; r < Z; ++r) {
        legendre_column(L, m, hr[r], cm, b, col.data());
        for (int j = 0; j < n0; ++j) lam0[(size_t)r * n0 + j] = col[2 * j];
        for (int j = 0; j < n1; ++j) lam1[(size_t)r * n1 + j] = col[2 * j + 1];
    }
}

// F+ (sign = +1) or F- (sign = -1) = (2_lambda +- (-2)_lambda)/2 of one m,
// split into the two l - m parities like build_lambda.  F+ keeps the mirror
// parity (-1)^(l+m) of the scalar functions, F- has the opposite one; the
// ring stage's combine takes care of that.
void build_lambda_spin(int L, int m, int Z, const std::vector<HalfRing> &hr, DD cm, int sign,
                       std::vector<double> &lam0, std::vector<double> &lam1)
{
    const int n0 = chain_len(L, m, 0), n1 = chain_len(L, m, 1);
    lam0.assign((size_t)n0 * Z, 0.0);
    lam1.assign((size_t)n1 * Z, 0.0);
    std::vector<double> cp(L - m + 1), cmn(L - m + 1);
    for (int r = 0; r < Z; ++r) {
        spin_column(L, m, 2, hr[r], cm, cp.data());
        spin_column(L, m, -2, hr[r], cm, cmn.data());
        auto F = [&](int i) {
            const double v = 0.5 * (cp[i] + sign * cmn[i]);
            return std::fabs(v) >= kCrop ? v : 0.0;
        };
        for (int j = 0; j < n0; ++j) lam0[(size_t)r * n0 + j] = F(2 * j);
        for (int j = 0; j < n1; ++j) lam1[(size_t)r * n1 + j] = F(2 * j + 1);
    }
}

// ---------------------------------------------- host interpreter (tests)
// Applies the serialised items of one chain to a real vector a (length n)
// exactly as the device kernels do, in plain double: q (length Z).
void apply_chain_host(const BfChain &ch, int Z, const double *a, double *q)
{
    std::vector<double> buf[2];
    buf[0].assign(std::max<long long>(ch.region, 1), 0.0);
    buf[1].assign(std::max<long long>(ch.region, 1), 0.0);
    for (int r = 0; r < Z; ++r) q[r] = 0.0;
    for (const BfRLocal &rb : ch.rblocks) {
        for (int s = 0; s < rb.k; ++s) {
            double acc = 0.0;
            for (int j = 0; j < rb.nrows; ++j) acc += rb.data[(size_t)j * rb.k + s] * a[rb.j0 + j];
            if (rb.to_rings) q[rb.rings[s]] = acc;
            else buf[ch.depth % 2][rb.out_off + s] = acc;
        }
    }
    for (const BfItemLocal &it : ch.items) {
        const std::vector<double> &in = buf[it.level % 2];
        std::vector<double> outv(it.nc, 0.0);
        for (int s = 0; s < 2; ++s) {
            const int k = it.k[s];
            const int nd = (int)it.dense_pos[s].size();
            for (int d = 0; d < nd; ++d) {
                double acc = 0.0;
                for (int i = 0; i < k; ++i) acc += it.T[s][(size_t)i * nd + d] * in[it.u_off[s] + i];
                outv[it.dense_pos[s][d]] += acc;
            }
            for (int i = 0; i < k; ++i) outv[it.ident_pos[s][i]] += in[it.u_off[s] + i];
        }
        if (it.to_rings) {
            for (int c = 0; c < it.nc; ++c) q[it.rings[c]] = outv[c];
        } else {
            std::vector<double> &o = buf[(it.level - 1) % 2];
            for (int c = 0; c < it.nc; ++c) o[it.out_off + c] = outv[c];
        }
    }
}

}  // namespace shtb

// ------------------------------------------------------------------------
// Plan build: compress every chain (parallel over m), then lay all chains'
// items out in flat arrays and upload them.
int shtb_build_butterfly(shtb_plan_s *p)
{
    const int L = p->lmax, N = p->nside, Z = 2 * N;
    const int nthreads = p->opts.nthreads;
    shtb::BfParams prm;
    prm.eps = p->eps;
    prm.leaf_cols = p->opts.leaf_cols > 0 ? p->opts.leaf_cols : 32;
    prm.max_depth = p->opts.max_depth;
    if (p->kind != 0 && !(p->eps > 0)) prm.max_depth = 0;   // polarised, uncompressed: depth 0 only
    if (prm.leaf_cols > shtb::kMaxCand)
        return shtb_fail(SHTB_ENOTSUP, "leaf_cols above " + std::to_string(shtb::kMaxCand));
    const bool rec = p->opts.residual_recurrence != 0;
    if (rec && (p->kind != 0 || !(p->eps > 0)))
        return shtb_fail(SHTB_ENOTSUP, "residual_recurrence needs a compressed scalar plan");
    std::vector<shtb::HalfRing> hr(Z);
    for (int r = 0; r < Z; ++r) hr[r] = shtb::half_ring(N, r + 1);
    const std::vector<shtb::DD> cm = shtb::diag_norms(L);
    std::vector<shtb::BfChain> chains((size_t)(L + 1) * 2);
    // largest chains first for the thread pool
    std::vector<int> order(L + 1);
    std::iota(order.begin(), order.end(), 0);
    // with opts.gpu_build the IDs of each level of each chain run as one
    // batch on the plan's GPU; every host worker thread has its own slot
    int nworkers = nthreads > 0 ? nthreads : (int)std::max(1u, std::thread::hardware_concurrency());
    if (p->opts.gpu_build && nthreads <= 0) nworkers *= 2;   // workers also wait on their GPU batches
    shtb::GpuIdPool *pool = nullptr;
    if (p->opts.gpu_build) {
        pool = shtb::gpu_id_pool_create(p->device, nworkers);
        if (!pool) return shtb_fail(SHTB_ENOMEM, "plan build: GPU ID pool");
    }
    std::mutex slot_mu;
    std::map<std::thread::id, int> slot_of;
    std::atomic<int> first_err{0};
    shtb::parallel_for(L + 1, nworkers, [&](int i) {
        if (first_err.load()) return;
        const int m = order[i];
        shtb::BfParams my = prm;
        if (pool) {
            std::lock_guard<std::mutex> g(slot_mu);
            auto it = slot_of.find(std::this_thread::get_id());
            if (it == slot_of.end()) it = slot_of.emplace(std::this_thread::get_id(), (int)slot_of.size()).first;
            my.gpu = pool;
            my.slot = it->second;
        }
        std::vector<double> lam0, lam1;
        if (p->kind == 0) shtb::build_lambda(L, m, Z, hr, cm[m], lam0, lam1);
        else shtb::build_lambda_spin(L, m, Z, hr, cm[m], p->kind == 1 ? 1 : -1, lam0, lam1);
        int rc = shtb::compress_chain(lam0.data(), chain_len(L, m, 0), Z, my, &chains[(size_t)m * 2]);
        if (!rc) rc = shtb::compress_chain(lam1.data(), chain_len(L, m, 1), Z, my, &chains[(size_t)m * 2 + 1]);
        if (rc) {
            int zero = 0;
            first_err.compare_exchange_strong(zero, rc);
        }
    });
    if (pool) shtb::gpu_id_pool_destroy(pool);
    if (first_err.load()) return first_err.load();

    auto *bf = new BfPlanDev();
    p->bf = bf;
    std::vector<long long> ubase(chains.size());
    long long utot = 0;
    int depth_max = 0;
    std::vector<int> depth_par(chains.size());
    for (size_t c = 0; c < chains.size(); ++c) {
        ubase[c] = utot;
        utot += chains[c].region;
        depth_max = std::max(depth_max, chains[c].depth);
        depth_par[c] = chains[c].depth % 2;
        if (chains[c].depth < 16) p->stats.depth_hist[chains[c].depth]++;
    }
    // regenerated R: host copies of the recurrence tables of the dense plan
    std::vector<RecCoef> h_coef;
    std::vector<double> h_xarg;
    std::vector<int> h_xform, h_jstart;
    std::vector<double2> h_vstart;
    if (rec) {
        h_coef.resize((size_t)p->nalm);
        h_xarg.resize(Z);
        h_xform.resize(Z);
        h_jstart.resize((size_t)(L + 1) * 2 * Z);
        h_vstart.resize(h_jstart.size());
        const std::pair<void *, std::pair<const void *, size_t>> cp[] = {
            {h_coef.data(), {p->view.coef, sizeof(RecCoef) * h_coef.size()}},
            {h_xarg.data(), {p->view.xarg, sizeof(double) * h_xarg.size()}},
            {h_xform.data(), {p->view.xform, sizeof(int) * h_xform.size()}},
            {h_jstart.data(), {p->view.jstart, sizeof(int) * h_jstart.size()}},
            {h_vstart.data(), {p->view.vstart, sizeof(double2) * h_vstart.size()}}};
        for (const auto &c : cp)
            if (cudaMemcpy(c.first, c.second.first, c.second.second, cudaMemcpyDeviceToHost) != cudaSuccess)
                return shtb_fail(SHTB_ECUDA, "plan build: reading the recurrence tables");
    }
    std::vector<RecStart> rstart;
    long long n_rgen = 0;
    std::vector<int> ints;
    std::vector<double> dbl;
    std::vector<BfRGroup> rgroups;
    std::vector<BfRItem> ritems;
    std::vector<int> ritem_interval;         // chain-local interval of each residual item
    std::vector<int> ritem_chain;
    std::vector<std::vector<BfItem>> litems(depth_max);
    long long n_dense = 0, n_r = 0, n_ident = 0;
    for (size_t c = 0; c < chains.size(); ++c) {
        shtb::BfChain &ch = chains[c];
        const int m = (int)(c / 2), t = (int)(c % 2);
        const long long entry0 = (long long)c * Z;    // q^t entry of ring 0 of this chain
        for (auto &rb : ch.rblocks) {
            BfRItem it{};
            it.m = m;
            it.t = t;
            it.j0 = rb.j0;
            it.nrows = rb.nrows;
            it.k = rb.k;
            it.to_rings = rb.to_rings ? 1 : 0;
            if (rec) {
                it.data_off = 0;
                it.rs_off = (long long)rstart.size();
                const int n = chain_len(L, m, t);
                const RecCoef *cf = h_coef.data() + alm_index(L, m, m);
                for (int sc = 0; sc < rb.k; ++sc) {
                    const int r = rb.cols[sc];
                    const size_t idx = ((size_t)m * 2 + t) * Z + r;
                    rstart.push_back(shtb::block_column_start(n, t, rb.j0, rb.nrows, r, h_xarg[r], h_xform[r] != 0,
                                                              cf, h_jstart[idx], h_vstart[idx]));
                }
                n_rgen += (long long)rb.nrows * rb.k;
            } else {
                it.rs_off = 0;
                it.data_off = (long long)dbl.size();
                dbl.insert(dbl.end(), rb.data.begin(), rb.data.end());
                n_r += (long long)rb.data.size();
            }
            if (rb.to_rings) {
                it.out_off = (long long)ints.size();
                for (int r : rb.rings) ints.push_back((int)(entry0 + r));
            } else {
                it.out_off = ubase[c] + rb.out_off;
            }
            ritems.push_back(it);
            ritem_interval.push_back(rb.interval);
            ritem_chain.push_back((int)c);
            std::vector<double>().swap(rb.data);
        }
        for (auto &li : ch.items) {
            BfItem it{};
            it.nc = li.nc;
            for (int s = 0; s < 2; ++s) {
                it.k[s] = li.k[s];
                it.nd[s] = (int)li.dense_pos[s].size();
                it.u_off[s] = ubase[c] + li.u_off[s];
                it.dpos_off[s] = (long long)ints.size();
                ints.insert(ints.end(), li.dense_pos[s].begin(), li.dense_pos[s].end());
                it.ipos_off[s] = (long long)ints.size();
                ints.insert(ints.end(), li.ident_pos[s].begin(), li.ident_pos[s].end());
                it.T_off[s] = (long long)dbl.size();
                dbl.insert(dbl.end(), li.T[s].begin(), li.T[s].end());
                n_dense += (long long)li.T[s].size();
                n_ident += li.k[s];
            }
            it.to_rings = li.to_rings ? 1 : 0;
            if (li.to_rings) {
                it.out_off = (long long)ints.size();
                for (int r : li.rings) ints.push_back((int)(entry0 + r));
            } else {
                it.out_off = ubase[c] + li.out_off;
            }
            litems[li.level - 1].push_back(it);
        }
        shtb::BfChain().rblocks.swap(ch.rblocks);
        std::vector<shtb::BfItemLocal>().swap(ch.items);
    }
    if ((long long)ints.size() > INT_MAX)
        return shtb_fail(SHTB_ENOTSUP, "butterfly index table exceeds 2^31 entries");
    // the level kernels take level 1 as the one whose items write q^t
    for (int l = 0; l < depth_max; ++l)
        for (const BfItem &it : litems[l])
            if ((l == 0) != (it.to_rings != 0))
                return shtb_fail(SHTB_ENOTSUP, "butterfly item writing q^t outside level 1");
    // longest items first within each launch, so that the last wave is
    // short; items of similar shape end up adjacent, so a block's warps
    // finish together
    std::vector<int> rord(ritems.size());
    std::iota(rord.begin(), rord.end(), 0);
    std::stable_sort(rord.begin(), rord.end(), [&](int a, int b) {
        if (ritems[a].nrows != ritems[b].nrows) return ritems[a].nrows > ritems[b].nrows;
        return ritems[a].k > ritems[b].k;
    });
    {
        std::vector<BfRItem> sorted(ritems.size());
        std::vector<int> where(ritems.size());
        for (size_t i = 0; i < rord.size(); ++i) {
            sorted[i] = ritems[rord[i]];
            where[rord[i]] = (int)i;
        }
        ritems.swap(sorted);
        // adjoint groups: every top row interval of every chain, with its blocks
        std::vector<std::vector<std::vector<int>>> blk(chains.size());
        for (size_t c = 0; c < chains.size(); ++c) blk[c].resize(chains[c].top_rows.size());
        for (size_t i = 0; i < ritem_chain.size(); ++i)
            blk[ritem_chain[i]][ritem_interval[i]].push_back(where[i]);
        for (size_t c = 0; c < chains.size(); ++c) {
            for (size_t I = 0; I < chains[c].top_rows.size(); ++I) {
                BfRGroup gr{};
                gr.m = (int)(c / 2);
                gr.t = (int)(c % 2);
                gr.r0 = chains[c].top_rows[I].first;
                gr.r1 = chains[c].top_rows[I].second;
                if (gr.r1 <= gr.r0) continue;
                gr.nblk = (int)blk[c][I].size();
                gr.blk_off = (long long)ints.size();
                ints.insert(ints.end(), blk[c][I].begin(), blk[c][I].end());
                rgroups.push_back(gr);
            }
        }
        std::sort(rgroups.begin(), rgroups.end(), [](const BfRGroup &a, const BfRGroup &b) {
            return (long long)(a.r1 - a.r0) * (a.nblk + 1) > (long long)(b.r1 - b.r0) * (b.nblk + 1);
        });
    }
    // level items: heaviest first (a short last wave), then within runs of
    // 64 by longest child input and most dense rows, so that a block's warps
    // have similar shapes
    for (auto &lv : litems) {
        std::stable_sort(lv.begin(), lv.end(), [](const BfItem &a, const BfItem &b) {
            return (long long)a.k[0] * a.nd[0] + (long long)a.k[1] * a.nd[1] >
                   (long long)b.k[0] * b.nd[0] + (long long)b.k[1] * b.nd[1];
        });
        constexpr size_t kRun = 64;
        for (size_t a = 0; a < lv.size(); a += kRun)
            std::stable_sort(lv.begin() + a, lv.begin() + std::min(lv.size(), a + kRun),
                             [](const BfItem &x, const BfItem &y) {
                                 const int kx = std::max(x.k[0], x.k[1]), ky = std::max(y.k[0], y.k[1]);
                                 if (kx != ky) return kx > ky;
                                 return std::max(x.nd[0], x.nd[1]) > std::max(y.nd[0], y.nd[1]);
                             });
    }
    bf->depth_max = depth_max;
    bf->u_entries = std::max<long long>(utot, 1);
    bf->qt_entries = (long long)(L + 1) * 2 * Z;
    bf->n_dense = n_dense;
    bf->n_r = n_r;
    bf->n_ident = n_ident;
    int rc;
    void *d;
    if ((rc = plan_alloc_upload(p, &d, ints.data(), sizeof(int) * ints.size()))) return rc;
    bf->ints = (const int *)d;
    std::vector<int>().swap(ints);
    if ((rc = plan_alloc_upload(p, &d, dbl.data(), sizeof(double) * dbl.size()))) return rc;
    bf->dbl = (const double *)d;
    std::vector<double>().swap(dbl);
    if ((rc = plan_alloc_upload(p, &d, depth_par.data(), sizeof(int) * depth_par.size()))) return rc;
    bf->depth_parity = (const int *)d;
    const long long n_rstart = (long long)rstart.size();
    if ((rc = plan_alloc_upload(p, &d, rstart.data(), sizeof(RecStart) * rstart.size()))) return rc;
    bf->rstart = (const RecStart *)d;
    bf->rec = rec;
    bf->n_rgen = n_rgen;
    std::vector<RecStart>().swap(rstart);
    if ((rc = plan_alloc_upload(p, &d, ritems.data(), sizeof(BfRItem) * ritems.size()))) return rc;
    bf->ritems = (const BfRItem *)d;
    bf->n_ritems = (int)ritems.size();
    if ((rc = plan_alloc_upload(p, &d, rgroups.data(), sizeof(BfRGroup) * rgroups.size()))) return rc;
    bf->rgroups = (const BfRGroup *)d;
    bf->n_rgroups = (int)rgroups.size();
    bf->level_items.assign(depth_max, nullptr);
    bf->level_counts.assign(depth_max, 0);
    bf->level_maxnc.assign(depth_max, 1);
    for (int l = 0; l < depth_max; ++l) {
        for (const BfItem &it : litems[l]) bf->level_maxnc[l] = std::max(bf->level_maxnc[l], it.nc);
        if ((rc = plan_alloc_upload(p, &d, litems[l].data(), sizeof(BfItem) * litems[l].size()))) return rc;
        bf->level_items[l] = (const BfItem *)d;
        bf->level_counts[l] = (int)litems[l].size();
    }
    if ((rc = bf_pack_operator(p))) return rc;
    p->stats.n_dense = n_dense;
    p->stats.n_rstored = n_r;
    p->stats.n_rgen = n_rgen;
    p->stats.n_ident = n_ident;
    p->stats.compressed = 1;
    // per map: 2 FMAs (re, im) per stored or regenerated element, 2 adds per
    // identity entry; a regenerated element also costs one recurrence step
    // (2 FMAs) per call, counted here at one map
    p->stats.recurrence_flops = 4.0 * (double)n_rgen;
    p->stats.legendre_flops_per_map =
        4.0 * (double)(n_dense + n_r + n_rgen) + 2.0 * (double)n_ident + p->stats.recurrence_flops;
    // bytes one synthesis reads from the plan: stored elements, or the start
    // records and the recurrence coefficients
    p->stats.plan_read_bytes = (long long)(8 * (n_dense + n_r)) +
                               (rec ? (long long)(sizeof(RecStart) * n_rstart + sizeof(RecCoef) * p->nalm) : 0);
    return SHTB_OK;
}

void bf_release(shtb_plan_s *p)
{
    delete p->bf;
    p->bf = nullptr;
}

// ------------------------------------------------------------------------
// Private host-only checks (no GPU).

// ID of a rows x n column-major block: returns k, the skeleton positions and
// the full k x n interpolation matrix (identity on the skeleton, 0 on zero
// columns), row-major.
extern "C" int shtb_test_host_id(int rows, int n, const double *A, double eps, int *k_out,
                                 int *skel_out, double *T_out)
{
    if (rows < 0 || n < 0 || !A || !k_out || !skel_out || !T_out || !(eps > 0))
        return shtb_fail(SHTB_EINVAL, "bad arguments");
    shtb::IdResult id = shtb::interp_decomp(A, rows, n, rows, eps, 0.0);
    *k_out = id.k;
    const int nd = (int)id.dense_pos.size();
    for (int i = 0; i < id.k; ++i) {
        skel_out[i] = id.skel[i];
        for (int c = 0; c < n; ++c) {
            const int kd = id.kind[c];
            double v = 0.0;
            if (kd >= 0) v = kd == i ? 1.0 : 0.0;
            else if (kd != shtb::kZeroCol) v = id.T[(size_t)i * nd + (-1 - kd)];
            T_out[(size_t)i * n + c] = v;
        }
    }
    return SHTB_OK;
}

// The same ID through the GPU builder's batched kernel (one block), on the
// current device.
extern "C" int shtb_test_gpu_id(int rows, int n, const double *A, double eps, int *k_out, int *skel_out,
                                double *T_out)
{
    if (rows < 0 || n < 0 || n > shtb::kMaxCand || !A || !k_out || !skel_out || !T_out || !(eps > 0))
        return shtb_fail(SHTB_EINVAL, "bad arguments");
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return shtb_fail(SHTB_ECUDA, "no CUDA device");
    shtb::GpuIdPool *pool = shtb::gpu_id_pool_create(dev, 1);
    if (!pool) return shtb_fail(SHTB_ENOMEM, "GPU ID pool");
    std::vector<shtb::IdResult> ids;
    const int rc = shtb::gpu_id_run(pool, 0, A, (long long)rows * n, {shtb::IdBlock{0, rows, n}}, eps, 1e-30, ids);
    shtb::gpu_id_pool_destroy(pool);
    if (rc) return rc;
    const shtb::IdResult &r = ids[0];
    *k_out = r.k;
    for (int i = 0; i < r.k; ++i) skel_out[i] = r.skel[i];
    for (size_t i = 0; i < (size_t)r.k * n; ++i) T_out[i] = 0.0;
    for (int c = 0; c < n; ++c) {
        const int kd = r.kind[c];
        if (kd == shtb::kZeroCol) continue;
        for (int i = 0; i < r.k; ++i)
            T_out[(size_t)i * n + c] = kd >= 0 ? (i == kd ? 1.0 : 0.0) : r.T[(size_t)i * r.dense_pos.size() + (-1 - kd)];
    }
    return SHTB_OK;
}

// Compress Lambda^{m,t} of a HEALPix grid and apply the result on the host to
// a real vector a (chain length n = chain_len(lmax, m, t)): q_out gets the
// compressed Lambda^T a, q_exact the dense product; info = {depth, n_dense
// (T elements), n_r (stored residual elements), n_ident}.
extern "C" int shtb_test_host_butterfly(int nside, int lmax, double eps, int m, int t, int leaf_cols,
                                        const double *a, double *q_out, double *q_exact,
                                        long long *info)
{
    if (nside < 1 || lmax < 0 || m < 0 || m > lmax || t < 0 || t > 1 || !(eps > 0) ||
        leaf_cols < 1 || leaf_cols > shtb::kMaxCand || !a || !q_out || !q_exact || !info)
        return shtb_fail(SHTB_EINVAL, "bad arguments");
    const int Z = 2 * nside;
    std::vector<shtb::HalfRing> hr(Z);
    for (int r = 0; r < Z; ++r) hr[r] = shtb::half_ring(nside, r + 1);
    const std::vector<shtb::DD> cm = shtb::diag_norms(lmax);
    std::vector<double> lam0, lam1;
    shtb::build_lambda(lmax, m, Z, hr, cm[m], lam0, lam1);
    const std::vector<double> &lam = t == 0 ? lam0 : lam1;
    const int n = chain_len(lmax, m, t);
    for (int r = 0; r < Z; ++r) {
        double s = 0.0;
        for (int j = 0; j < n; ++j) s += lam[(size_t)r * n + j] * a[j];
        q_exact[r] = s;
    }
    shtb::BfParams prm;
    prm.eps = eps;
    prm.leaf_cols = leaf_cols;
    shtb::BfChain ch;
    (void)shtb::compress_chain(lam.data(), n, Z, prm, &ch);
    shtb::apply_chain_host(ch, Z, a, q_out);
    long long nd = 0, nr = 0, ni = 0;
    for (const auto &it : ch.items)
        for (int s = 0; s < 2; ++s) {
            nd += (long long)it.T[s].size();
            ni += it.k[s];
        }
    for (const auto &rb : ch.rblocks) nr += (long long)rb.data.size();
    info[0] = ch.depth;
    info[1] = nd;
    info[2] = nr;
    info[3] = ni;
    return SHTB_OK;
}
