// Assembly kernels on the fixed-point kernel evaluations of gamma_fixed.cuh:
// coupling blocks (Sec. 5.3), dense inadmissible leaf blocks (Sec. 5.2) and the
// density's far and near sums (Sec. 6.2).  They take the operators whose mesh
// and fields fit the formats (OpData::fx); assemble.cu holds the FP64 kernels
// for the others.
#include <algorithm>

#include "device_common.cuh"
#include "gamma_fixed.cuh"

namespace vfd {

// ---------------------------------------------------------------------------
// coupling blocks S_e[b][a] = -2 gamma(xi_a, xi_b)
// ---------------------------------------------------------------------------
template <int D>
__global__ void __launch_bounds__(256)
k_coupling_fx(int k, int nnode, int nfar, const int *__restrict__ fptr, const int *__restrict__ fcol,
              const i64 *__restrict__ ch, const i64 *__restrict__ ab, const u64 *__restrict__ tab,
              double *__restrict__ S)
{
    extern __shared__ __align__(16) u64 sh_tab[];
    const FxTab t = fx_stage(tab, sh_tab);
    __syncthreads();
    const size_t nn = (size_t)nnode * k;
    for (int e = blockIdx.x; e < nfar; e += gridDim.x) {
        int lo = 0, hi = nnode;   // row node of block e
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (fptr[mid] <= e) lo = mid; else hi = mid;
        }
        const int ia0 = lo * k, ib0 = fcol[e] * k;
        double *out = S + (size_t)e * k * k;
        for (int i = threadIdx.x; i < k * k; i += blockDim.x) {
            const int be = i / k, ia = ia0 + i - be * k, ib = ib0 + be;
            i64 x[D], y[D];
#pragma unroll
            for (int c = 0; c < D; ++c) {
                x[c] = ch[(size_t)ia * D + c];
                y[c] = ch[(size_t)ib * D + c];
            }
            out[i] = -2.0 * fx_gamma<D>(t, x, y, ab[ia] + ab[ib], (u64)(ab[nn + ia] + ab[nn + ib]));
        }
    }
}

void launch_coupling_fixed(const MeshData &m, OpData &op, cudaStream_t st)
{
    auto go = [&](int k, const DBuf<long long> &X, const DBuf<long long> &ab, double *S) {
        auto f = m.d == 1 ? k_coupling_fx<1> : m.d == 2 ? k_coupling_fx<2> : k_coupling_fx<3>;
        VFD_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FX_BYTES));
        f<<<std::min(m.nfar, 152 * 6), 256, FX_BYTES, st>>>(k, m.kt.nnode, m.nfar, m.far_ptr.p, m.far_col.p, X.p, ab.p,
                                                            m.fx_tab.p, S);
        VFD_CUDA(cudaGetLastError());
    };
    go(m.k, m.fx_ktX, op.kc_ab, op.S64.p);
    if (m.k_in && op.precision != VFD_FP64) go(m.k_in, m.fx_ktX_in, op.kc_ab_in, op.S64_in.p);
}

// ---------------------------------------------------------------------------
// dense inadmissible leaf blocks D[i][j] = -2 sum_q sum_q' c_i(q) c_j(q') gamma_T(q, q'),
// c_i(q) = w_q psi_i(q).  CTA per (computed block, slice of its row points); a
// thread holds one row point q and walks the column cells, which the whole
// warp shares: the points of a cell are evaluated together (independent
// chains), folded to the cell's vertices in registers,
//     sum_q' c_j(q') gamma = w' (mu sum_q' gamma + (lam - mu) gamma_j)
// (the rule's points have barycentric coordinate lam at their own vertex and mu
// at the others; w' is in the exponent), and added to T[j][q] in shared memory,
// one lane per q.  Then D[i][j] = sum over the support of i of c_i(q) T[j][q].
//
// Bound: 823M evaluations at 27k DoFs (rank-64 disk), each about 60 cycles of
// an SM and warp in the integer pipes, against 2.7 FP64 instructions of 16
// cycles for the two contractions in the FP64 pipe; the two overlap.  Near phase
// of an assembly: 61.4 ms with FP64 evaluations, 12.2 ms here (67 G
// evaluations/s); 3D ball of 751 DoFs, 724M evaluations: 357 and 10.0 ms.
// ---------------------------------------------------------------------------
namespace {

constexpr int NF_CELLS = 32;   // column cells per staged tile
constexpr int NF_RT = 128;     // row points per tile: one per thread

struct NearFx {
    int nQ, fl, maxleaf, nsplit;
    size_t part;                 // entries of one partial result (nsplit > 1)
    const int *near_col, *near_src, *prow, *panel_w, *kt_begin, *kt_end, *lp_ptr, *lp_pts, *supp_ptr, *supp_loc;
    const int64_t *near_off;
    const double *supp_coef;
    const int *qcell, *cells, *vdof;
    const i64 *X, *a, *b, *aw;   // coordinates (SoA), exponent terms, a + log2 of the weight
    const u64 *tab;
    double mu, rho;              // barycentric mu; (lam - mu) / mu
    double bary1[3][2];          // 1D: barycentrics of the three points
    double *D;
};

template <int D>
__global__ void __launch_bounds__(NF_RT) k_near_fx(NearFx P)
{
    constexpr int NV = D + 1, NQ = D == 3 ? 4 : 3, CT = NF_CELLS, RT = NF_RT, TS = RT + 1;
    extern __shared__ __align__(16) u64 sh_tab[];
    const int e = blockIdx.x;
    if (P.near_src[e] >= 0) return;   // transposed copy, filled by k_near_transpose
    const int a = P.prow[e], b = P.near_col[e];
    const int ra = P.kt_begin[P.fl + a], na = P.kt_end[P.fl + a] - ra;
    const int rb = P.kt_begin[P.fl + b], nb = P.kt_end[P.fl + b] - rb;
    const int pa0 = P.lp_ptr[a], npa = P.lp_ptr[a + 1] - pa0;
    const int pb0 = P.lp_ptr[b], ncb = (P.lp_ptr[b + 1] - pb0) / NQ;
    const int ntile = (npa + RT - 1) / RT;
    if ((int)blockIdx.y >= max(ntile, 1)) {   // no rows for this slice: its partial result is zero
        if (P.nsplit > 1)
            for (int t = threadIdx.x; t < na * nb; t += blockDim.x)
                P.D[blockIdx.y * P.part + P.near_off[e] + (size_t)(t / nb) * P.panel_w[a] + t % nb] = 0.0;
        return;
    }
    const FxTab tab = fx_stage(P.tab, sh_tab);
    double *T = (double *)(sh_tab + FX_WORDS);                 // maxleaf x TS (an odd stride)
    i64 *cx = (i64 *)(T + (size_t)P.maxleaf * TS);             // CT cells: NQ x D coordinates, NQ a, NQ b
    i64 *ca = cx + CT * NQ * D, *cb = ca + CT * NQ;
    int *cv = (int *)(cb + CT * NQ);                           // CT x NV vertex ids
    int *cj = cv + CT * NV;                                    // CT x NV DoFs of leaf b, or -1
    const int row = threadIdx.x;
    double *out = P.D + (P.nsplit > 1 ? blockIdx.y * P.part : 0) + P.near_off[e];
    const int W = P.panel_w[a];
    bool first = true;
    for (int tile = blockIdx.y; tile < ntile; tile += P.nsplit) {
        const int t0 = tile * RT, nt = min(RT, npa - t0);
        const bool live = row < nt;
        const int q = P.lp_pts[pa0 + t0 + (live ? row : 0)];
        i64 x[D];
#pragma unroll
        for (int c = 0; c < D; ++c) x[c] = P.X[(size_t)c * P.nQ + q];
        const i64 qa = P.a[q], qb = P.b[q];
        int v[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) v[k] = P.cells[(size_t)P.qcell[q] * NV + k];
        for (int j = 0; j < nb; ++j) T[(size_t)j * TS + row] = 0.0;
        for (int c0 = 0; c0 < ncb; c0 += CT) {
            const int nc = min(CT, ncb - c0);
            __syncthreads();
            for (int t = threadIdx.x; t < nc * NQ; t += blockDim.x) {
                const int id = P.lp_pts[pb0 + c0 * NQ + t];
#pragma unroll
                for (int c = 0; c < D; ++c) cx[t * D + c] = P.X[(size_t)c * P.nQ + id];
                ca[t] = P.aw[id];
                cb[t] = P.b[id];
            }
            for (int t = threadIdx.x; t < nc * NV; t += blockDim.x) {
                const int vert = P.cells[(size_t)P.qcell[P.lp_pts[pb0 + (c0 + t / NV) * NQ]] * NV + t % NV];
                const int j = P.vdof[vert] - rb;
                cv[t] = vert;
                cj[t] = j >= 0 && j < nb ? j : -1;
            }
            __syncthreads();
            if ((row & ~31) < nt)   // warps without a row point only stage
#pragma unroll 1
                for (int c = 0; c < nc; ++c) {
                    double g[NQ];
#pragma unroll
                    for (int k = 0; k < NQ; ++k) {
                        const int l = c * NQ + k;
                        g[k] = fx_gamma<D>(tab, x, cx + l * D, qa + ca[l], (u64)(qb + cb[l]));
                    }
                    bool touch = false;
#pragma unroll
                    for (int u = 0; u < NV; ++u)
#pragma unroll
                        for (int k = 0; k < NV; ++k) touch |= v[u] == cv[c * NV + k];
                    if (touch) {
#pragma unroll
                        for (int k = 0; k < NQ; ++k) g[k] = 0.0;
                    }
                    if (D == 1) {
#pragma unroll
                        for (int k = 0; k < NV; ++k) {
                            const int j = cj[c * NV + k];
                            if (j >= 0)
                                T[(size_t)j * TS + row] += g[0] * P.bary1[0][k] + g[1] * P.bary1[1][k] + g[2] * P.bary1[2][k];
                        }
                    } else {
                        double s = g[0] + g[1];
#pragma unroll
                        for (int k = 2; k < NQ; ++k) s += g[k];
#pragma unroll
                        for (int k = 0; k < NV; ++k) {
                            const int j = cj[c * NV + k];   // the same for the whole warp
                            if (j >= 0) T[(size_t)j * TS + row] += fma(P.rho, g[k], s);
                        }
                    }
                }
        }
        __syncthreads();
        // fold the rows: the support entries of DoF i that lie in this tile
        for (int idx = threadIdx.x; idx < na * nb; idx += blockDim.x) {
            const int i = idx / nb, j = idx - i * nb, di = ra + i;
            double s = 0.0;
            for (int s2 = P.supp_ptr[di]; s2 < P.supp_ptr[di + 1]; ++s2) {
                const int l = P.supp_loc[s2] - t0;
                if (l >= 0 && l < nt) s = fma(P.supp_coef[s2], T[(size_t)j * TS + l], s);
            }
            double *o = out + (size_t)i * W + j;
            const double add = -2.0 * P.mu * s;
            *o = first ? add : *o + add;   // always the same thread's entry
        }
        first = false;
        __syncthreads();
    }
}

// D = the partial results in slice order
__global__ void k_near_reduce(int nsplit, size_t part, const double *__restrict__ p, const int *__restrict__ src,
                              const int *__restrict__ prow, const int *__restrict__ ncol, const int *__restrict__ kb,
                              const int *__restrict__ ke, int fl, const int64_t *__restrict__ off,
                              const int *__restrict__ pw, double *__restrict__ D)
{
    const int e = blockIdx.x;
    if (src[e] >= 0) return;
    const int a = prow[e], b = ncol[e];
    const int na = ke[fl + a] - kb[fl + a], nb = ke[fl + b] - kb[fl + b];
    for (int t = threadIdx.x; t < na * nb; t += blockDim.x) {
        const size_t o = off[e] + (size_t)(t / nb) * pw[a] + t % nb;
        double s = 0.0;
        for (int q = 0; q < nsplit; ++q) s += p[q * part + o];
        D[o] = s;
    }
}

template <int D>
bool near_fx(const MeshData &m, OpData &op, cudaStream_t st)
{
    constexpr int NV = D + 1, NQ = D == 3 ? 4 : 3;
    NearFx P;
    P.nQ = m.nQ;
    P.fl = m.kt.first_leaf();
    P.maxleaf = m.max_leaf_size;
    P.near_col = m.near_col.p;
    P.near_src = m.near_src.p;
    P.prow = m.near_pair_row.p;
    P.near_off = m.near_off.p;
    P.panel_w = m.panel_w.p;
    P.kt_begin = m.kt_begin.p;
    P.kt_end = m.kt_end.p;
    P.lp_ptr = m.lp_ptr.p;
    P.lp_pts = m.lp_pts.p;
    P.supp_ptr = m.supp_ptr.p;
    P.supp_loc = m.supp_loc.p;
    P.supp_coef = m.supp_coef.p;
    P.qcell = m.qcell.p;
    P.cells = m.cells.p;
    P.vdof = m.vdof.p;
    P.X = m.fx_qX.p;
    P.a = op.q_ab.p;
    P.b = op.q_ab.p + m.nQ;
    P.aw = op.q_ab.p + 2 * (size_t)m.nQ;
    P.tab = m.fx_tab.p;
    if (D == 1) {
        const double g = 0.5 * std::sqrt(0.6), t[3] = {0.5 - g, 0.5, 0.5 + g};
        for (int q = 0; q < 3; ++q) {
            P.bary1[q][0] = 1.0 - t[q];
            P.bary1[q][1] = t[q];
        }
        P.mu = 1.0;
        P.rho = 0.0;
    } else {
        const double lam = D == 2 ? 2.0 / 3.0 : (5.0 + 3.0 * std::sqrt(5.0)) / 20.0;
        P.mu = D == 2 ? 1.0 / 6.0 : (5.0 - std::sqrt(5.0)) / 20.0;
        P.rho = (lam - P.mu) / P.mu;
    }
    // 128 row points a tile: two CTAs share an SM (leaves of at most 64 DoFs), so
    // that one's folds and staging run under the other's evaluations
    const size_t shm = FX_BYTES + (size_t)P.maxleaf * (NF_RT + 1) * 8 +
                       (size_t)NF_CELLS * (NQ * (D + 2) * 8 + 2 * NV * 4);
    if (shm > 227 * 1024) return false;
    // few blocks (small meshes): the row tiles of a block on several CTAs, their
    // partial results summed in order afterwards
    const int ntile = std::max(1, cdiv(m.max_leaf_pts, NF_RT)), ncomp = (m.nnear + m.kt.nleaf) / 2;
    P.nsplit = std::max(1, std::min(ntile, std::min(32, cdiv(2 * 304, std::max(ncomp, 1)))));
    DBuf<double> part;
    P.D = op.D64.p;
    P.part = op.D64.n;
    if (P.nsplit > 1) {
        part.alloc(P.part * P.nsplit);
        P.D = part.p;
    }
    VFD_CUDA(cudaFuncSetAttribute(k_near_fx<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
    k_near_fx<D><<<dim3(m.nnear, P.nsplit), NF_RT, shm, st>>>(P);
    VFD_CUDA(cudaGetLastError());
    if (P.nsplit > 1) {
        k_near_reduce<<<m.nnear, 256, 0, st>>>(P.nsplit, P.part, part.p, P.near_src, P.prow, P.near_col, P.kt_begin,
                                               P.kt_end, P.fl, P.near_off, P.panel_w, op.D64.p);
        VFD_CUDA(cudaGetLastError());
        VFD_CUDA(cudaStreamSynchronize(st));   // the partial results are released on return
    }
    return true;
}

}  // namespace

bool launch_near_build_fixed(const MeshData &m, OpData &op, cudaStream_t st)
{
    if (!(m.d == 1 ? near_fx<1>(m, op, st) : m.d == 2 ? near_fx<2>(m, op, st) : near_fx<3>(m, op, st))) return false;
    launch_near_transpose(m, op, st);
    return true;
}

// ---------------------------------------------------------------------------
// density: far sums at the target nodes' Chebyshev points, a thread per
// (node, alpha) over the node's blocks and their source nodes' points
// ---------------------------------------------------------------------------
template <int D>
__global__ void __launch_bounds__(128)
k_rho_coupling_fx(int k, int nnode_t, int nnode_s, const int *__restrict__ fptr, const int *__restrict__ fcol,
                  const i64 *__restrict__ tch, const i64 *__restrict__ tab_t, const i64 *__restrict__ sch,
                  const i64 *__restrict__ tab_s, const double *__restrict__ xs, const u64 *__restrict__ tab,
                  double *__restrict__ yt)
{
    extern __shared__ __align__(16) u64 sh_tab[];
    const FxTab t = fx_stage(tab, sh_tab);
    __syncthreads();
    const size_t nt = (size_t)nnode_t * k, ns = (size_t)nnode_s * k;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nt; i += (size_t)gridDim.x * blockDim.x) {
        const int n = (int)(i / k), e0 = fptr[n], e1 = fptr[n + 1];
        double acc0 = 0.0, acc1 = 0.0;
        if (e1 > e0) {
            i64 x[D];
#pragma unroll
            for (int c = 0; c < D; ++c) x[c] = tch[i * D + c];
            const i64 a = tab_t[i], b = tab_t[nt + i];
            for (int e = e0; e < e1; ++e) {
                const size_t j0 = (size_t)fcol[e] * k;
                int be = 0;
                for (; be + 1 < k; be += 2) {   // two independent chains
                    const size_t j = j0 + be;
                    acc0 = fma(fx_gamma<D>(t, x, sch + j * D, a + tab_s[j], (u64)(b + tab_s[ns + j])), xs[j], acc0);
                    acc1 = fma(fx_gamma<D>(t, x, sch + (j + 1) * D, a + tab_s[j + 1], (u64)(b + tab_s[ns + j + 1])),
                               xs[j + 1], acc1);
                }
                if (be < k) {
                    const size_t j = j0 + be;
                    acc0 = fma(fx_gamma<D>(t, x, sch + j * D, a + tab_s[j], (u64)(b + tab_s[ns + j])), xs[j], acc0);
                }
            }
        }
        yt[i] = acc0 + acc1;
    }
}

void launch_rho_coupling_fixed(const MeshData &m, OpData &op, double *yt, cudaStream_t st)
{
    auto f = m.d == 1 ? k_rho_coupling_fx<1> : m.d == 2 ? k_rho_coupling_fx<2> : k_rho_coupling_fx<3>;
    VFD_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FX_BYTES));
    const int n = m.tt.nnode * m.k;
    f<<<cdiv(n, 128), 128, FX_BYTES, st>>>(m.k, m.tt.nnode, m.st.nnode, m.rfar_ptr.p, m.rfar_col.p, m.fx_ttX.p,
                                           op.tc_ab.p, m.fx_stX.p, op.sc_ab.p, m.st_xhat.p, m.fx_tab.p, yt);
    VFD_CUDA(cudaGetLastError());
}

// ---------------------------------------------------------------------------
// density: direct sums over the near sources, rho[q] = sum_q' w' gamma_T(q, q').
// CTA per target leaf: 64 targets x 4 groups of sources; the sources are staged
// in tiles, the group sums added in order.  About 60 cycles of an SM and warp
// per evaluation (integer pipes) and one FP64 addition (16).  Density phase at
// 27k DoFs (143M near pairs, 313M far evaluations): 37.1 ms in FP64, 5.0 ms.
// ---------------------------------------------------------------------------
constexpr int RN_T = 64, RN_G = 4, RN_S = 128;

struct RhoNearFx {
    int nQ, tfl;
    const int *tt_begin, *tt_end, *tt_perm, *st_begin, *st_end, *st_perm, *rnear_ptr, *rnear_col, *qcell, *cells;
    const i64 *X, *a, *b, *aw;
    const u64 *tab;
    double *rho;
};

template <int D>
__global__ void __launch_bounds__(RN_T *RN_G) k_rho_near_fx(RhoNearFx P)
{
    constexpr int NV = D + 1;
    extern __shared__ __align__(16) u64 sh_tab[];
    __shared__ i64 sx[RN_S * D], sa[RN_S], sb[RN_S];
    __shared__ int sv[RN_S * NV];
    __shared__ double part[RN_G][RN_T];
    const FxTab t = fx_stage(P.tab, sh_tab);
    const int leaf = blockIdx.x, node = P.tfl + leaf, b0 = P.tt_begin[node], e0 = P.tt_end[node];
    const int tl = threadIdx.x % RN_T, grp = threadIdx.x / RN_T;   // grp: the same for a whole warp
    for (int i0 = b0; i0 < e0; i0 += RN_T) {
        const bool live = i0 + tl < e0;
        const int id = P.tt_perm[live ? i0 + tl : i0];
        i64 x[D];
#pragma unroll
        for (int c = 0; c < D; ++c) x[c] = P.X[(size_t)c * P.nQ + id];
        const i64 a = P.a[id], b = P.b[id];
        int v[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) v[k] = P.cells[(size_t)P.qcell[id] * NV + k];
        double acc0 = 0.0, acc1 = 0.0;
        for (int ne = P.rnear_ptr[leaf]; ne < P.rnear_ptr[leaf + 1]; ++ne) {
            const int sn = P.rnear_col[ne], sb0 = P.st_begin[sn], se = P.st_end[sn];
            for (int j0 = sb0; j0 < se; j0 += RN_S) {
                const int nj = min(RN_S, se - j0);
                __syncthreads();
                for (int q = threadIdx.x; q < nj; q += blockDim.x) {
                    const int jd = P.st_perm[j0 + q];
#pragma unroll
                    for (int c = 0; c < D; ++c) sx[q * D + c] = P.X[(size_t)c * P.nQ + jd];
                    sa[q] = P.aw[jd];
                    sb[q] = P.b[jd];
#pragma unroll
                    for (int k = 0; k < NV; ++k) sv[q * NV + k] = P.cells[(size_t)P.qcell[jd] * NV + k];
                }
                __syncthreads();
                auto term = [&](int q) {
                    const double g = fx_gamma<D>(t, x, sx + q * D, a + sa[q], (u64)(b + sb[q]));
                    bool touch = false;
#pragma unroll
                    for (int u = 0; u < NV; ++u)
#pragma unroll
                        for (int k = 0; k < NV; ++k) touch |= v[u] == sv[q * NV + k];
                    return touch ? 0.0 : g;
                };
                if ((tl & ~31) < e0 - i0) {
                    int q = grp;
#pragma unroll 1
                    for (; q + RN_G < nj; q += 2 * RN_G) {
                        const double g0 = term(q), g1 = term(q + RN_G);
                        acc0 += g0;
                        acc1 += g1;
                    }
                    if (q < nj) acc0 += term(q);
                }
            }
        }
        __syncthreads();
        part[grp][tl] = acc0 + acc1;
        __syncthreads();
        if (threadIdx.x < RN_T && live) {
            double s = 0.0;
#pragma unroll
            for (int g = 0; g < RN_G; ++g) s += part[g][tl];
            P.rho[id] = s;
        }
        __syncthreads();
    }
}

void launch_rho_near_fixed(const MeshData &m, OpData &op, cudaStream_t st)
{
    RhoNearFx P;
    P.nQ = m.nQ;
    P.tfl = m.tt.first_leaf();
    P.tt_begin = m.tt_begin.p;
    P.tt_end = m.tt_end.p;
    P.tt_perm = m.tt_perm.p;
    P.st_begin = m.st_begin.p;
    P.st_end = m.st_end.p;
    P.st_perm = m.st_perm.p;
    P.rnear_ptr = m.rnear_ptr.p;
    P.rnear_col = m.rnear_col.p;
    P.qcell = m.qcell.p;
    P.cells = m.cells.p;
    P.X = m.fx_qX.p;
    P.a = op.q_ab.p;
    P.b = op.q_ab.p + m.nQ;
    P.aw = op.q_ab.p + 2 * (size_t)m.nQ;
    P.tab = m.fx_tab.p;
    P.rho = op.rho.p;
    auto f = m.d == 1 ? k_rho_near_fx<1> : m.d == 2 ? k_rho_near_fx<2> : k_rho_near_fx<3>;
    VFD_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FX_BYTES));
    f<<<m.tt.nleaf, RN_T * RN_G, FX_BYTES, st>>>(P);
    VFD_CUDA(cudaGetLastError());
}

}  // namespace vfd
