// Singular near field B in 2D (Sec. 4): the tensor Gauss rules of the vertex
// (eq. e:int-v-2), edge (eq. e:int-e) and identical (eq. e:int-i-2) cases,
// one warp per touching pair.
//
// Each region's map sends (zeta, eta1, eta2, eta3) to (xhat, yhat), and xhat
// (yhat) depends on a subset of the four Gauss indices only (e.g. the vertex
// region 1 has xhat = xi (1, eta1)).  The warp first evaluates s and log kappa
// once per distinct mapped point into shared memory, then sweeps the 4D
// points with table lookups, so a 4D point costs one log and one exp.  The
// per-index powers and logarithms of zeta, t and eta1 are tabulated per CTA.
#include <algorithm>
#include <cmath>

#include "device_common.cuh"
#include "gamma_fixed.cuh"
#include "sing_maps.cuh"

namespace vfd {

void launch_singular_B_generic(const MeshData &m, OpData &op, DBuf<double> &Lbuf, cudaStream_t st);

namespace {

// index masks (bit 0: zeta, bit 1: eta1, bit 2: eta2 (t in the identical
// case), bit 3: eta3) of the point each region's xhat / yhat depends on
__constant__ unsigned char c_xmask[3][5] = {{0x3, 0xD, 0, 0, 0}, {0xB, 0x3, 0x7, 0xF, 0xF}, {0x7, 0xF, 0xF, 0, 0}};
__constant__ unsigned char c_ymask[3][5] = {{0xD, 0x3, 0, 0, 0}, {0x7, 0xF, 0xF, 0x3, 0x7}, {0xF, 0x7, 0x7, 0, 0}};

struct Tab {
    double lz[NSMAX], xi[NSMAX], lt[NSMAX], e2[NSMAX], le1[NSMAX];
};

__device__ __forceinline__ int ipow(int b, int e)
{
    int r = 1;
    for (int i = 0; i < e; ++i) r *= b;
    return r;
}

// table index of (iz,i1,i2,i3) for a mask; the table spans ns^popc(mask)
__device__ __forceinline__ int tindex(unsigned mask, int ns, const int *ind)
{
    int idx = 0, mul = 1;
    for (int j = 0; j < 4; ++j)
        if (mask & (1u << j)) {
            idx += ind[j] * mul;
            mul *= ns;
        }
    return idx;
}

__device__ __forceinline__ void tdecode(unsigned mask, int ns, int t, int *ind)
{
    for (int j = 0; j < 4; ++j) {
        ind[j] = 0;
        if (mask & (1u << j)) {
            ind[j] = t % ns;
            t /= ns;
        }
    }
}

__device__ __forceinline__ void phys(const double *V, const double *xh, double *x, double *bary)
{
    // chi(xh) = V0 + (V1 - V0) xh1 + (V2 - V1) xh2 ; barycentric (1-xh1, xh1-xh2, xh2)
    x[0] = V[0] + (V[2] - V[0]) * xh[0] + (V[4] - V[2]) * xh[1];
    x[1] = V[1] + (V[3] - V[1]) * xh[0] + (V[5] - V[3]) * xh[1];
    bary[0] = 1.0 - xh[0];
    bary[1] = xh[0] - xh[1];
    bary[2] = xh[1];
}

struct Sing2Params {
    int ns, npairs, cap;   // cap: field-table entries per warp
    double sbar;
    const int *pinfo;
    const double *vx;
    int M;
    const double *gx, *gw;
    const double *mt;
    DField Fs, Fk;
};

__global__ void __launch_bounds__(256) k_singular2d(Sing2Params P, double *__restrict__ Lbuf)
{
    extern __shared__ __align__(16) double shs[];
    __shared__ Tab tab;
    const int ns = P.ns;
    const double sbar = P.sbar, c = 4.0 - 2.0 * sbar, c2 = 2.0 - 2.0 * sbar;
    if (threadIdx.x < ns) {
        double g = P.gx[threadIdx.x], lg = log(g);
        tab.lz[threadIdx.x] = lg;
        tab.xi[threadIdx.x] = exp(lg / c);
        tab.lt[threadIdx.x] = lg;
        tab.e2[threadIdx.x] = exp(lg / c2);
        tab.le1[threadIdx.x] = lg;
    }
    __syncthreads();
    const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int pair = blockIdx.x * (blockDim.x >> 5) + wib;
    if (pair >= P.npairs) return;
    double *fs = shs + (size_t)wib * 2 * P.cap, *fk = fs + P.cap;
    const int *pi = P.pinfo + (size_t)pair * 8;
    const int type = pi[0];
    const double wgt = (double)pi[1];
    int pv[3] = {pi[2], pi[3], pi[4]}, qv[3] = {pi[5], pi[6], pi[7]};
    double Pv[6], Qv[6];
    for (int a = 0; a < 3; ++a)
        for (int j = 0; j < 2; ++j) {
            Pv[a * 2 + j] = P.vx[(size_t)j * P.M + pv[a]];
            Qv[a * 2 + j] = P.vx[(size_t)j * P.M + qv[a]];
        }
    const double JP[4] = {Pv[2] - Pv[0], Pv[4] - Pv[2], Pv[3] - Pv[1], Pv[5] - Pv[3]};
    const double JQ[4] = {Qv[2] - Qv[0], Qv[4] - Qv[2], Qv[3] - Qv[1], Qv[5] - Qv[3]};
    const double detP = fabs(JP[0] * JP[3] - JP[1] * JP[2]), detQ = fabs(JQ[0] * JQ[3] - JQ[1] * JQ[2]);
    const int ti = type - 1;   // 0 vertex, 1 edge, 2 identical
    const int nreg = type == 1 ? 2 : (type == 2 ? 5 : 3);
    const double *Vy = (type == 3) ? Pv : Qv;
    const int *vy = (type == 3) ? pv : qv;
    // ---- phase 1: fields at the distinct mapped points
    int xo[5], yo[5];
    {
        int off = 0;
        for (int reg = 0; reg < nreg; ++reg) {
            xo[reg] = off;
            off += ipow(ns, __popc(c_xmask[ti][reg]));
            yo[reg] = off;
            off += ipow(ns, __popc(c_ymask[ti][reg]));
        }
    }
    for (int reg = 0; reg < nreg; ++reg)
        for (int side = 0; side < 2; ++side) {
            const unsigned mask = side == 0 ? c_xmask[ti][reg] : c_ymask[ti][reg];
            const int size = ipow(ns, __popc(mask)), off = side == 0 ? xo[reg] : yo[reg];
            for (int t = lane; t < size; t += 32) {
                int ind[4];
                tdecode(mask, ns, t, ind);
                const double xi = tab.xi[ind[0]], e1 = P.gx[ind[1]], e3 = P.gx[ind[3]];
                double a[2], b[2], aux[2], jac;
                if (type == 3) map_id(reg, e1, tab.e2[ind[2]], e3, a, b, aux);
                else map_ve(type, reg, e1, P.gx[ind[2]], e3, a, b, jac);
                double h[2], x[2], bary[3], sv, kv;
                if (side == 0) {
                    h[0] = xi * a[0]; h[1] = xi * a[1];
                    phys(Pv, h, x, bary);
                    fields2(P.Fs, P.Fk, 2, x, pv, bary, sv, kv, P.mt);
                } else {
                    h[0] = xi * b[0]; h[1] = xi * b[1];
                    phys(Vy, h, x, bary);
                    fields2(P.Fs, P.Fk, 2, x, vy, bary, sv, kv, P.mt);
                }
                fs[off + t] = sv;
                fk[off + t] = kv;
            }
        }
    __syncwarp();
    // ---- phase 2: the 4D tensor rule
    double acc[15];
    for (int i = 0; i < 15; ++i) acc[i] = 0.0;
    const int per = ns * ns * ns * ns, tot = nreg * per;
    if (type != 3) {
        const double pre = detP * detQ / c;
        for (int idx = lane; idx < tot; idx += 32) {
            int reg = idx / per, r = idx - reg * per;
            int ind[4] = {r % ns, (r / ns) % ns, (r / (ns * ns)) % ns, r / (ns * ns * ns)};
            const double e1 = P.gx[ind[1]], e2 = P.gx[ind[2]], e3 = P.gx[ind[3]];
            double a[2], b[2], jac;
            map_ve(type, reg, e1, e2, e3, a, b, jac);
            const int ix = xo[reg] + tindex(c_xmask[ti][reg], ns, ind), iy = yo[reg] + tindex(c_ymask[ti][reg], ns, ind);
            const double S = fs[ix] + fs[iy];
            double dx = JP[0] * a[0] + JP[1] * a[1] - JQ[0] * b[0] - JQ[1] * b[1];
            double dy = JP[2] * a[0] + JP[3] * a[1] - JQ[2] * b[0] - JQ[3] * b[1];
            double D2 = dx * dx + dy * dy;
            double w = P.gw[ind[0]] * P.gw[ind[1]] * P.gw[ind[2]] * P.gw[ind[3]] * pre * jac *
                       fast_exp(P.mt, (2.0 * sbar - S) / c * tab.lz[ind[0]] + 0.5 * (fk[ix] + fk[iy]) -
                                          0.5 * (2.0 + S) * fast_log(P.mt, D2));
            // basis differences (psi(x) - psi(y))/xi, reference basis 1-x1, x1-x2, x2
            double f[5];
            if (type == 1) {
                f[0] = b[0] - a[0]; f[1] = a[0] - a[1]; f[2] = a[1]; f[3] = -(b[0] - b[1]); f[4] = -b[1];
            } else {
                f[0] = b[0] - a[0]; f[1] = (a[0] - a[1]) - (b[0] - b[1]); f[2] = a[1]; f[3] = -b[1]; f[4] = 0.0;
            }
            int t = 0;
            for (int i = 0; i < 5; ++i)
                for (int j = i; j < 5; ++j) acc[t++] += w * f[i] * f[j];
        }
    } else {
        const double pre = 2.0 * detP * detP / (c * c2);   // the mirror regions T_I^(4..6) double the sum
        for (int idx = lane; idx < tot; idx += 32) {
            int reg = idx / per, r = idx - reg * per;
            int ind[4] = {r % ns, (r / ns) % ns, (r / (ns * ns)) % ns, r / (ns * ns * ns)};
            const double e1 = P.gx[ind[1]], e2 = tab.e2[ind[2]], e3 = P.gx[ind[3]];
            double a[2], b[2], dr[2];
            map_id(reg, e1, e2, e3, a, b, dr);
            const int ix = xo[reg] + tindex(c_xmask[2][reg], ns, ind), iy = yo[reg] + tindex(c_ymask[2][reg], ns, ind);
            const double S = fs[ix] + fs[iy];
            double dx = JP[0] * dr[0] + JP[1] * dr[1], dy = JP[2] * dr[0] + JP[3] * dr[1];
            double D2 = dx * dx + dy * dy;
            double w = P.gw[ind[0]] * P.gw[ind[1]] * P.gw[ind[2]] * P.gw[ind[3]] * pre *
                       fast_exp(P.mt, (2.0 * sbar - S) * (tab.lz[ind[0]] / c + tab.lt[ind[2]] / c2) +
                                          (2.0 - S) * tab.le1[ind[1]] + 0.5 * (fk[ix] + fk[iy]) -
                                          0.5 * (2.0 + S) * fast_log(P.mt, D2));
            double f[3] = {-dr[0], dr[0] - dr[1], dr[1]};
            int t = 0;
            for (int i = 0; i < 3; ++i)
                for (int j = i; j < 5; ++j) acc[t++] += (j < 3) ? w * f[i] * f[j] : 0.0;
        }
    }
    const int nl = type == 1 ? 5 : (type == 2 ? 4 : 3);
    for (int i = 0; i < 15; ++i) acc[i] = warp_sum(acc[i]);
    if (lane == 0) {
        double *L = Lbuf + (size_t)pair * 25;
        int t = 0;
        for (int i = 0; i < 5; ++i)
            for (int j = i; j < 5; ++j, ++t) {
                double v = (i < nl && j < nl) ? wgt * acc[t] : 0.0;
                L[i * 5 + j] = v;
                L[j * 5 + i] = v;
            }
    }
}

// ---------------------------------------------------------------------------
// The same sums on the fixed-point kernel evaluations (gamma_fixed.cuh).
//
// What of a 4D point does not depend on the pair is tabulated once per assembly
// (k_sing_table): the coefficients a, b of the scaled difference x - y, the
// products w f_i f_j of rule weight, map Jacobian and basis differences, and the
// part of the exponent that comes from zeta, t and eta1,
//   (2 sbar - S) q + (2 - S) l = cst - (b_x + b_y) nu,   S = 2 (b_x + b_y) - 2,
// q = ln zeta / c (+ ln t / c2) and l = ln eta1 in the identical case: nu adds to N
// = -ln |difference|^2 and cst to the sum of the a terms.  The basis differences
// sum to zero, so row and column 0 of a local matrix are minus the sums of the
// others and 10, 6 or 3 products (vertex, edge, identical) are enough.
// A 4D point then takes 10 FP64 instructions for the difference, 3 to 10 for the
// sums, and one evaluation (FP64 kernel: about 150 in all); the fields at the
// mapped points, about one evaluation of s and log kappa per 4D point, are as
// before.  87.8M 4D points (27k DoFs): 48.1 -> 25.0 ms; P1 fields, 13.1M points
// (4k DoFs): 3.3 -> 1.7 ms.
// ---------------------------------------------------------------------------
constexpr int ST_A = 0, ST_NU = 4, ST_CST = 5, ST_F = 6, ST_SLOTS = 16;

__global__ void k_sing_table(int ns, double sbar, const double *__restrict__ gx, const double *__restrict__ gw,
                             double *__restrict__ out)
{
    const int per = ns * ns * ns * ns, t = blockIdx.x * blockDim.x + threadIdx.x, ne = 10 * per;
    if (t >= ne) return;
    const int type = t < 2 * per ? 1 : (t < 7 * per ? 2 : 3);
    const int i = t - sing_first(type) * per, reg = i / per, r = i - reg * per;
    const int iz = r % ns, i1 = (r / ns) % ns, i2 = (r / (ns * ns)) % ns, i3 = r / (ns * ns * ns);
    double a[2], b[2], d[4];
    const SingPoint p = sing_point(type, reg, sbar, gx[iz], gx[i1], gx[i2], gx[i3], a, b, d);
    const double w = p.w * gw[iz] * gw[i1] * gw[i2] * gw[i3];
    for (int q = 0; q < 4; ++q) out[(size_t)(ST_A + q) * ne + t] = d[q];
    out[(size_t)ST_NU * ne + t] = fx_bits(p.nu, 56);
    out[(size_t)ST_CST * ne + t] = fx_bits(p.cst, 53);
    const int nf = type == 1 ? 4 : (type == 2 ? 3 : 2);
    int s = ST_F;
    for (int u = 1; u <= nf; ++u)
        for (int v = u; v <= nf; ++v, ++s) out[(size_t)s * ne + t] = w * p.f[u] * p.f[v];
}

struct SingFx {
    Sing2Params S;
    int w;             // scale of the fixed-point coordinates
    const double *st;  // k_sing_table
    const u64 *tab;
    int *err;
};

// sum of v[0..15] over the warp, halving the values at every step: lane 2 q and 2 q + 1 get sum q
template <int NF>
__device__ __forceinline__ double warp_sum16(double *v, int lane)
{
#pragma unroll
    for (int q = NF; q < 16; ++q) v[q] = 0.0;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        const int o = 16 >> h, n = 8 >> h;
        const bool up = lane & o;
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (q < n && q < NF) {
                const double send = up ? v[q] : v[q + n], keep = up ? v[q + n] : v[q];
                v[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// phase 2 of one pair with NF products
template <int NF, bool IDENT>
__device__ __forceinline__ void sing_sum(const SingFx &P, const FxTab &tab, int type, const double *JP, const double *JQ,
                                         const i64 *fa, const i64 *fb, const int *xo, const int *yo, double pre,
                                         double *__restrict__ L, int lane)
{
    const int ns = P.S.ns, per = ns * ns * ns * ns, tot = sing_regions(type) * per, ne = 10 * per, ti = type - 1;
    const double *st = P.st + (size_t)sing_first(type) * per;
    double acc[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) acc[q] = 0.0;
    for (int idx = lane; idx < tot; idx += 32) {
        const int reg = idx / per, r = idx - reg * per;
        const int ind[4] = {r % ns, (r / ns) % ns, (r / (ns * ns)) % ns, r / (ns * ns * ns)};
        const int ix = xo[reg] + tindex(c_xmask[ti][reg], ns, ind), iy = yo[reg] + tindex(c_ymask[ti][reg], ns, ind);
        const double a0 = st[idx], a1 = st[ne + idx];
        double dx = JP[0] * a0 + JP[1] * a1, dy = JP[2] * a0 + JP[3] * a1;
        if (!IDENT) {
            const double b0 = st[2 * (size_t)ne + idx], b1 = st[3 * (size_t)ne + idx];
            dx = dx - JQ[0] * b0 - JQ[1] * b1;
            dy = dy - JQ[2] * b0 - JQ[3] * b1;
        }
        u64 M;
        int K;
        fx_r2(dx * dx + dy * dy, P.w, M, K);
        const u64 N = fx_neglog(tab, M, K) + (u64)__double_as_longlong(st[(size_t)ST_NU * ne + idx]);
        const i64 A = fa[ix] + fa[iy] + __double_as_longlong(st[(size_t)ST_CST * ne + idx]);
        const double w = fx_exp(tab, A, (u64)(fb[ix] + fb[iy]), N);
#pragma unroll
        for (int q = 0; q < NF; ++q) acc[q] = fma(w, st[(size_t)(ST_F + q) * ne + idx], acc[q]);
    }
    const double mine = pre * warp_sum16<NF>(acc, lane);   // lanes 2 q hold sum q
    // local matrix: rows 1..nf from the sums, row and column 0 from the zero row sums
    constexpr int nf = NF == 10 ? 4 : (NF == 6 ? 3 : 2);
    double m[5][5] = {};
    int s = 0;
#pragma unroll
    for (int u = 1; u <= nf; ++u)
#pragma unroll
        for (int v = u; v <= nf; ++v, ++s) m[u][v] = m[v][u] = __shfl_sync(0xffffffffu, mine, 2 * s);
    double all = 0.0;
#pragma unroll
    for (int u = 1; u <= nf; ++u) {
        double t = 0.0;
#pragma unroll
        for (int v = 1; v <= nf; ++v) t += m[u][v];
        m[0][u] = m[u][0] = -t;
        all += t;
    }
    m[0][0] = all;
    double out = 0.0;   // one entry per lane
#pragma unroll
    for (int u = 0; u < 5; ++u)
#pragma unroll
        for (int v = 0; v < 5; ++v)
            if (lane == u * 5 + v) out = m[u][v];
    if (lane < 25) L[lane] = out;
}

__global__ void __launch_bounds__(256) k_singular2d_fx(SingFx P, double *__restrict__ Lbuf)
{
    extern __shared__ __align__(16) u64 sh_sing[];
    const Sing2Params &Q = P.S;
    const int ns = Q.ns;
    const FxTab tab = fx_stage(P.tab, sh_sing);
    __shared__ double txi[NSMAX], te2[NSMAX];
    if ((int)threadIdx.x < ns) {
        const double lg = log(Q.gx[threadIdx.x]);
        txi[threadIdx.x] = exp(lg / (4.0 - 2.0 * Q.sbar));
        te2[threadIdx.x] = exp(lg / (2.0 - 2.0 * Q.sbar));
    }
    __syncthreads();
    const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    i64 *fa = (i64 *)(sh_sing + FX_WORDS) + (size_t)wib * 2 * Q.cap, *fb = fa + Q.cap;
    for (int pair = blockIdx.x * nw + wib; pair < Q.npairs; pair += gridDim.x * nw) {
        const int *pi = Q.pinfo + (size_t)pair * 8;
        const int type = pi[0], ti = type - 1, nreg = sing_regions(type);
        int pv[3] = {pi[2], pi[3], pi[4]}, qv[3] = {pi[5], pi[6], pi[7]};
        double Pv[6], Qv[6];
        for (int a = 0; a < 3; ++a)
            for (int j = 0; j < 2; ++j) {
                Pv[a * 2 + j] = Q.vx[(size_t)j * Q.M + pv[a]];
                Qv[a * 2 + j] = Q.vx[(size_t)j * Q.M + qv[a]];
            }
        const double JP[4] = {Pv[2] - Pv[0], Pv[4] - Pv[2], Pv[3] - Pv[1], Pv[5] - Pv[3]};
        const double JQ[4] = {Qv[2] - Qv[0], Qv[4] - Qv[2], Qv[3] - Qv[1], Qv[5] - Qv[3]};
        const double detP = fabs(JP[0] * JP[3] - JP[1] * JP[2]), detQ = fabs(JQ[0] * JQ[3] - JQ[1] * JQ[2]);
        // phase 1: exponent terms at the distinct mapped points
        int xo[5], yo[5], off = 0;
        for (int reg = 0; reg < nreg; ++reg) {
            xo[reg] = off;
            off += ipow(ns, __popc(c_xmask[ti][reg]));
            yo[reg] = off;
            off += ipow(ns, __popc(c_ymask[ti][reg]));
        }
        bool fits = true;
        __syncwarp();
        for (int t = lane; t < off; t += 32) {
            int reg = 0;
            while (reg + 1 < nreg && t >= xo[reg + 1]) ++reg;
            const bool second = t >= yo[reg];
            const unsigned mask = second ? c_ymask[ti][reg] : c_xmask[ti][reg];
            int ind[4];
            tdecode(mask, ns, t - (second ? yo[reg] : xo[reg]), ind);
            const double xi = txi[ind[0]], e1 = Q.gx[ind[1]], e3 = Q.gx[ind[3]];
            double a[2], b[2], aux[2], jac;
            if (type == 3) map_id(reg, e1, te2[ind[2]], e3, a, b, aux);
            else map_ve(type, reg, e1, Q.gx[ind[2]], e3, a, b, jac);
            double h[2], x[2], bary[3], sv, kv;
            h[0] = xi * (second ? b[0] : a[0]);
            h[1] = xi * (second ? b[1] : a[1]);
            const bool onq = second && type != 3;
            phys(onq ? Qv : Pv, h, x, bary);
            fields2(Q.Fs, Q.Fk, 2, x, onq ? qv : pv, bary, sv, kv, Q.mt);
            i64 A, B;
            fits &= fx_terms(2, P.w, sv, kv, A, B);
            fa[t] = A;
            fb[t] = B;
        }
        if (!fits) atomicOr(P.err, 1);
        __syncwarp();
        // phase 2
        const double wgt = (double)pi[1];
        double *L = Lbuf + (size_t)pair * 25;
        if (type == 1) sing_sum<10, false>(P, tab, 1, JP, JQ, fa, fb, xo, yo, wgt * detP * detQ, L, lane);
        else if (type == 2) sing_sum<6, false>(P, tab, 2, JP, JQ, fa, fb, xo, yo, wgt * detP * detQ, L, lane);
        else sing_sum<3, true>(P, tab, 3, JP, JQ, fa, fb, xo, yo, wgt * detP * detP, L, lane);
    }
}

}  // namespace

void launch_singular_B(const MeshData &m, OpData &op, DBuf<double> &Lbuf, bool fixed, cudaStream_t st)
{
    const int ns = m.opts.n_sing;
    // largest field table: the edge case, 4 ns^4 + 4 ns^3 + 2 ns^2 points
    const int cap = 4 * ns * ns * ns * ns + 4 * ns * ns * ns + 2 * ns * ns;
    const size_t per_warp = (size_t)cap * 2 * sizeof(double);
    int wpb = 8;
    while (wpb > 1 && per_warp * wpb > 200 * 1024) wpb /= 2;
    if (m.d != 2 || per_warp * wpb > 200 * 1024) {
        launch_singular_B_generic(m, op, Lbuf, st);
        return;
    }
    Lbuf.alloc((size_t)m.npairs * 25);
    if (!m.npairs) return;
    Sing2Params P;
    P.ns = ns;
    P.npairs = m.npairs;
    P.cap = cap;
    P.sbar = op.s_bar;
    P.pinfo = m.pair_info.p;
    P.vx = m.vx.p;
    P.M = m.M;
    P.gx = m.gl_x.p;
    P.gw = m.gl_w.p;
    P.mt = m.mtab.p;
    P.Fs = op.fs;
    P.Fk = op.fk;
    wpb = 8;
    while (wpb > 1 && FX_BYTES + per_warp * wpb > 110 * 1024) wpb /= 2;
    if (fixed && sing_fixed_fits(m, op.s_bar) && FX_BYTES + per_warp * wpb <= 220 * 1024) {
        const int ne = 10 * ns * ns * ns * ns;
        op.sing_tab.alloc((size_t)ST_SLOTS * ne);
        k_sing_table<<<cdiv(ne, 128), 128, 0, st>>>(ns, op.s_bar, P.gx, P.gw, op.sing_tab.p);
        SingFx F;
        F.S = P;
        F.w = m.fx_w;
        F.st = op.sing_tab.p;
        F.tab = m.fx_tab.p;
        F.err = op.errflag.p;
        const size_t shm = FX_BYTES + per_warp * wpb;
        VFD_CUDA(cudaFuncSetAttribute(k_singular2d_fx, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
        k_singular2d_fx<<<std::min(cdiv(m.npairs, wpb), 152 * 16), 32 * wpb, shm, st>>>(F, Lbuf.p);
        VFD_CUDA(cudaGetLastError());
        return;
    }
    wpb = 8;
    while (wpb > 1 && per_warp * wpb > 200 * 1024) wpb /= 2;
    size_t shm = per_warp * wpb;
    VFD_CUDA(cudaFuncSetAttribute(k_singular2d, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
    k_singular2d<<<cdiv(m.npairs, wpb), 32 * wpb, shm, st>>>(P, Lbuf.p);
    VFD_CUDA(cudaGetLastError());
}

}  // namespace vfd
