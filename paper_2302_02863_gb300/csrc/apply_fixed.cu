// The FP64 operator apply with its far field in fixed-point arithmetic.
//
// One FP64 multiply-add takes a warp 16 cycles of an SM on this part, so the
// FP64 kernels of apply.cu are bound by the FP64 pipe at any number of columns
// (98M multiply-adds a column at 27k DoFs and rank 64: 156 us at the pipe's
// rate, against 115 us for the bytes of one pass over the operator).  Here the
// far field's entries (three quarters of the products) and its vectors are
// 61-bit integers, scaled by a power of two per row of a coupling block or per
// leaf (flattened bases), and per leaf's or node's piece of a vector:
//   v = (hi 2^30 + lo) 2^(E - 60), |v| < 2^E, lo in [-2^29, 2^29), |hi| <= 2^30
// and a product takes three 32 x 32 + 64 bit multiply-adds,
//   hh += a.hi x.hi,   mid += a.hi x.lo + a.lo x.hi
// (3 cycles a warp; a.lo x.lo is below the last place kept).  Every fourth product
// the bits of hh and mid from 2^40 on move to 32-bit counters (2^20 a full-scale
// product, at most 64 levels x KMAX / 8 of them in a lane), so that nothing
// overflows (2^60 a product).  The sums are exact in the integers, so their order
// does not matter.
//
// What is rounded, and why it is no more than FP64 loses.  An entry of at least
// 2^-8 of the largest of its row of a block has all 53 bits of its FP64 value in
// 61; blocks with a smaller entry (fields that jump inside a box) stay FP64
// (OpData::fa_hard).  The bases and the vectors are rounded to 2^-61 of the
// largest entry of their leaf's or node's piece.  A basis row sums to its DoF's
// weight (Lagrange functions sum to one) and a block's entries are positive and of one size, so
// the largest entry of a piece is a part of every sum |U||S||U^T||x| that the
// piece goes into, and 2^-61 of it is below the 2^-53 by which FP64 rounds that
// sum.  Near rows have no such bound: their entries span up to 2^24 from the
// diagonal to the panel's far end, and a row scale would cut the small ones.
// They are FP64 products, which the FP64 pipe does beside the integer work of the
// far chain.
//
// Non-finite or nearly denormal vectors (a piece whose largest entry is Inf,
// NaN or below 2^-895) take plain FP64 sums over the FP64 operator instead, so
// that Inf, NaN and denormals come out as they do there.
//
//   1. k_fa_proj    per leaf: Ul^T x of every far level
//   2. k_fa_couple  a warp per admissible block: S_e xhat, xhat summed over the
//                   column node's leaves while it is gathered
//   3. k_fa_near    per row, the near panel row and the B + M row, FP64
//                   (concurrently with 1-2)
//   4. k_fa_expand  Y[i] += sum over levels of Ul[i] . yhat, yhat summed over the
//                   node's blocks while it is gathered
// With 3 or more columns the two sums are kernels of their own (apply.cu): a
// gather that repeats them for every block or leaf then costs more than it saves.
// Columns of the far chain go in groups of NC = 8 (4, 2, 1 for the remainder): an
// entry is loaded once for NC products.  The near rows take the remainder as it is:
// a column that is not there would cost FP64 time.
//
// Measured (FP64 kernels first): one column at 27k DoFs and rank 64 243 -> 170 us, at
// 16129 DoFs and rank 16 97 -> 66.  Errors in units of |A||x| on 900 DoFs, against extended
// precision with the FP64 operator's columns, FP64 kernels and here: normal x 6.4e-17
// and 5.8e-17 rms, x over six decades 8.8e-17 and 9.7e-17, x falling by 14 decades across
// the mesh 5.4e-17 and 5.0e-17, a Gaussian of width 0.1 1.0e-16 both.  A unit vector
// gives the near entries as they are stored.
#include <algorithm>
#include <type_traits>

#include "apply_common.cuh"
#include "apply_fixed.cuh"

namespace vfd {

namespace {

// products of a column: out_a = sum_b M[b stride + a] x[b], thread per a, x in
// shared memory [b][NC]
template <int NC>
__device__ __forceinline__ void fa_column(const int2 *__restrict__ M, size_t stride, int n, int step, const int2 *x,
                                          double *out)
{
    FaAcc s[NC];
    int b = 0;
#pragma unroll 2
    for (; b + 3 * step < n; b += 4 * step) {
        int2 m[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) m[q] = M[(size_t)(b + q * step) * stride];
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int c = 0; c < NC; ++c) s[c].mac(m[q], x[(b + q * step) * NC + c]);
#pragma unroll
        for (int c = 0; c < NC; ++c) s[c].carry();
    }
    for (; b < n; b += step) {
        const int2 m = M[(size_t)b * stride];
#pragma unroll
        for (int c = 0; c < NC; ++c) s[c].mac(m, x[b * NC + c]);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        s[c].carry();
        s[c].fold();
        out[c] = s[c].value();
    }
}

// ---------------------------------------------------------------------------
// 1. projections: CTA per (leaf, 128 of the nlev k columns, group of columns)
// ---------------------------------------------------------------------------
template <int NC>
__global__ void __launch_bounds__(128) k_fa_proj(FaFar P, const double *__restrict__ X, int64_t ld,
                                                 double *__restrict__ part, FaWhen when)
{
    extern __shared__ __align__(16) unsigned char fa_sm[];
    __shared__ unsigned key[NC];
    const int w = P.nlev * P.k, r0 = P.c0 + blockIdx.z * NC;
    if (fa_none(when)) return;
    double *raw = (double *)fa_sm;   // [i][NC]
    int2 *xs = (int2 *)fa_sm;
    const int col = blockIdx.y * blockDim.x + threadIdx.x;
    for (int leaf = blockIdx.x; leaf < P.nleaf; leaf += gridDim.x) {
        if (fa_off(when, leaf, r0)) continue;
        const int b = P.kb[P.fl + leaf], n = P.ke[P.fl + leaf] - b;
        __syncthreads();
        if (threadIdx.x < NC) key[threadIdx.x] = 0;
        __syncthreads();
        for (int t = threadIdx.x; t < n * NC; t += blockDim.x) {
            const int c = t / n, i = t - c * n;
            const double v = r0 + c < P.nrhs ? X[(size_t)(r0 + c) * ld + b + i] : 0.0;
            raw[i * NC + c] = v;
            atomicMax(&key[c], fa_key(v));
        }
        __syncthreads();
        bool slow = false;
#pragma unroll
        for (int c = 0; c < NC; ++c) slow |= fa_slow(key[c]);
        if (!slow) {
            for (int t = threadIdx.x; t < n * NC; t += blockDim.x) xs[t] = fa_split(fa_round(raw[t], key[t % NC]));
            __syncthreads();
        }
        if (col >= w) continue;
        const int2 *M = P.U + (size_t)b * P.wp + col;
        const int eu = P.ue[leaf], lv = col / P.k, a = col - lv * P.k;
        double out[NC];
        if (!slow) {
            fa_column<NC>(M, P.wp, n, 1, xs, out);
#pragma unroll
            for (int c = 0; c < NC; ++c) out[c] = out[c] * fa_pow2(eu - 30) * fa_scale(key[c]);
        } else {
#pragma unroll
            for (int c = 0; c < NC; ++c) out[c] = 0.0;
            for (int i = 0; i < n; ++i) {
                const double m = P.Ud[((size_t)lv * P.N + b + i) * P.k + a];
#pragma unroll
                for (int c = 0; c < NC; ++c) out[c] = fma(m, raw[i * NC + c], out[c]);
            }
        }
#pragma unroll
        for (int c = 0; c < NC; ++c)
            if (r0 + c < P.nrhs) part[(((size_t)(r0 + c) * P.nlev + lv) * P.nleaf + leaf) * P.k + a] = out[c];
    }
}

// ---------------------------------------------------------------------------
// 2. coupling: warp per admissible block; k <= 16 columns: 32/k' groups of lanes
//    share the rows
// ---------------------------------------------------------------------------
constexpr int FC_WARPS = 4;

template <int NC>
__global__ void __launch_bounds__(32 * FC_WARPS)
k_fa_couple(FaFar P, const double *__restrict__ part, const double *__restrict__ xhat, double *__restrict__ ye,
            FaWhen when)
{
    __shared__ int2 xs_[FC_WARPS][KMAX * NC];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r0 = P.c0 + blockIdx.y * NC, k = P.k;
    if (fa_none(when)) return;
    for (int e = blockIdx.x * FC_WARPS + warp; e < P.nfar; e += gridDim.x * FC_WARPS) {
        if (fa_off(when, when.mask ? P.row[e] : 0, r0)) continue;
        __syncwarp();
        int2 *xs = xs_[warp];
        double *raw = (double *)xs;
        const int node = P.fcol[e], l = 31 - __clz(node + 1), sh = P.L - l;
        const int leaf0 = ((node + 1) << sh) - (1 << P.L);
        const bool hard = P.hard[e];
        unsigned key[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const int r = r0 + c;
            unsigned mk = 0;
            for (int b = lane; b < k; b += 32) {
                double v = 0.0;
                if (r < P.nrhs) {
                    if (xhat) {
                        v = xhat[((size_t)r * P.nnode + node) * k + b];
                    } else {
                        const double *p = part + (((size_t)r * P.nlev + l - P.lmin) * P.nleaf + leaf0) * k + b;
#pragma unroll 8
                        for (int j = 0; j < (1 << sh); ++j) v += p[(size_t)j * k];
                    }
                }
                raw[b * NC + c] = v;
                mk = max(mk, fa_key(v));
            }
            key[c] = __reduce_max_sync(0xffffffffu, mk);
        }
        bool slow = false;
#pragma unroll
        for (int c = 0; c < NC; ++c) slow |= fa_slow(key[c]);
        __syncwarp();
        const int2 *S = P.S + (size_t)e * k * P.kp;
        if (slow || hard) {
            for (int a = lane; a < k; a += 32)
                for (int c = 0; c < NC && r0 + c < P.nrhs; ++c) {
                    double v = 0.0;
                    for (int b = 0; b < k; ++b) v = fma(P.Sd[((size_t)e * k + b) * k + a], raw[b * NC + c], v);
                    ye[((size_t)(r0 + c) * P.nfar + e) * k + a] = v;
                }
            continue;
        }
#pragma unroll
        for (int c = 0; c < NC; ++c)
            for (int b = lane; b < k; b += 32) xs[b * NC + c] = fa_split(fa_round(raw[b * NC + c], key[c]));
        __syncwarp();
        // lanes over a; with k <= 16 the groups of ga lanes take every (32 / ga)-th row
        const int ga = k > 16 ? 32 : k > 8 ? 16 : 8, gb = 32 / ga, la = lane & (ga - 1), lb = lane / ga;
        for (int a0 = 0; a0 < k; a0 += ga) {
            const int a = a0 + la, es = a < k ? P.se[(size_t)e * k + a] : 0;
            double out[NC];
            if (a < k) {
                fa_column<NC>(S + a + (size_t)lb * P.kp, P.kp, max(0, k - lb), gb, xs + lb * NC, out);
            } else {
#pragma unroll
                for (int c = 0; c < NC; ++c) out[c] = 0.0;
            }
            for (int o = ga; o < 32; o <<= 1) {
#pragma unroll
                for (int c = 0; c < NC; ++c) out[c] += __shfl_xor_sync(0xffffffffu, out[c], o);
            }
            if (a < k && lb == 0) {
#pragma unroll
                for (int c = 0; c < NC; ++c)
                    if (r0 + c < P.nrhs)
                        ye[((size_t)(r0 + c) * P.nfar + e) * k + a] =
                            out[c] * fa_pow2(max(es, -900) - 30) * fa_scale(key[c]);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// rows: sums over the entries of matrix rows, 8 lanes to a row and four rows to
// a warp, x in shared memory: [pair of columns][j]
// ---------------------------------------------------------------------------
template <int NC>
__device__ __forceinline__ void fa_row(const int2 *__restrict__ row, int w, int l8, const int4 *xs, int ws, FaAcc *s)
{
    auto term = [&](int2 a, int j) {
#pragma unroll
        for (int p = 0; p < NC / 2; ++p) {
            const int4 x = xs[(size_t)p * ws + j];
            s[2 * p].mac(a, make_int2(x.x, x.y));
            s[2 * p + 1].mac(a, make_int2(x.z, x.w));
        }
    };
    int j = l8;
#pragma unroll 1
    for (; j + 24 < w; j += 32) {
        int2 a[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] = row[j + 8 * q];
#pragma unroll
        for (int q = 0; q < 4; ++q) term(a[q], j + 8 * q);
#pragma unroll
        for (int c = 0; c < NC; ++c) s[c].carry();
    }
    for (; j < w; j += 8) term(row[j], j);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        s[c].carry();
        s[c].fold();
    }
}

// sum over the 8 lanes of a row (th and hh); every lane ends with one column,
// returned, and its sum in s[0]
template <int NC>
__device__ __forceinline__ int fa_sum8(FaAcc *s, int l8)
{
    int n = NC, col = 0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        if (n > 1) {
            n >>= 1;
            const bool up = l8 & o;
#pragma unroll
            for (int q = 0; q < NC / 2; ++q)
                if (q < n) {
                    const int st = up ? s[q].th : s[q + n].th, kt = up ? s[q + n].th : s[q].th;
                    const i64 sl = up ? s[q].hh : s[q + n].hh, kl = up ? s[q + n].hh : s[q].hh;
                    s[q].th = kt + __shfl_xor_sync(0xffffffffu, st, o);
                    s[q].hh = kl + __shfl_xor_sync(0xffffffffu, sl, o);
                }
            col += up ? n : 0;
        } else {
            s[0].th += __shfl_xor_sync(0xffffffffu, s[0].th, o);
            s[0].hh += __shfl_xor_sync(0xffffffffu, s[0].hh, o);
        }
    }
    return col;
}

// convert the gathered piece (raw FP64 in the layout of fa_row) in place
template <int NC>
__device__ __forceinline__ void fa_convert(unsigned char *sm, int ws, const unsigned *key)
{
    double *raw = (double *)sm;
    int2 *xs = (int2 *)sm;
    for (int t = threadIdx.x; t < ws * NC; t += blockDim.x) {
        const int c = NC == 1 ? 0 : 2 * (t / (2 * ws)) + (t & 1);
        xs[t] = fa_split(fa_round(raw[t], (int)key[c]));
    }
}
template <int NC>
__device__ __forceinline__ int fa_slot(int j, int c, int ws)   // of column c's entry j
{
    return NC == 1 ? j : (c >> 1) * 2 * ws + 2 * j + (c & 1);
}

// ---------------------------------------------------------------------------
// 3. near rows, FP64: CTA per (leaf, slice of NR rows, group of NC columns), 8 lanes to a
// row; x in shared memory as [pair of columns][j].  Bound by the FP64 pipe (16 cycles of
// an SM a warp and multiply-add), so that a group has no more columns than there are and
// an entry is loaded once for all of them.  (The next four entries loaded ahead cost more
// registers than they hide: 5 columns at 3721 DoFs 91 us instead of 76, 8 at 9025 202 / 165.)
// ---------------------------------------------------------------------------
template <int NC>
__global__ void __launch_bounds__(128) k_fa_near(FaNear P, const double *__restrict__ X, int64_t ld,
                                                 double *__restrict__ Y, FaWhen when)
{
    extern __shared__ __align__(16) unsigned char fa_sm[];
    const int lf = blockIdx.x, r0 = P.c0 + blockIdx.z * NC;
    if (fa_none(when) || fa_off(when, 0, r0)) return;
    const int b_leaf = P.kb[P.fl + lf], b = b_leaf + blockIdx.y * P.NR, e = min(P.ke[P.fl + lf], b + P.NR);
    if (b >= e) return;
    const int W = P.pw[lf];
    const int *gc = P.gcol + P.goff[lf];
    const double *x0 = X + (size_t)r0 * ld;
    const int nc = min(NC, P.nrhs - r0);              // columns of the group (fewer than NC where it is redone)
    constexpr int NP = NC > 4 ? 8 : NC > 2 ? 4 : 2;   // lanes of a row with a column
    double *xs = (double *)fa_sm;
#pragma unroll 4
    for (int t = threadIdx.x; t < W; t += blockDim.x) {
        const int j = gc[t];
#pragma unroll
        for (int c = 0; c < ((NC + 1) & ~1); ++c)
            xs[(c >> 1) * 2 * W + 2 * t + (c & 1)] = j >= 0 && c < nc ? x0[(size_t)c * ld + j] : 0.0;
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, l8 = lane & 7, nw = blockDim.x >> 5;
    for (int g0 = b + 4 * warp; g0 < e; g0 += 4 * nw) {
        const int i = g0 + (lane >> 3);
        const bool on = i < e;
        double s[NP];
#pragma unroll
        for (int c = 0; c < NP; ++c) s[c] = 0.0;
        if (on) {
            const double *row = P.Dd + P.poff[lf] + (size_t)(i - b_leaf) * W + l8;
            auto term = [&](double a, int j) {
#pragma unroll
                for (int p = 0; p < (NC + 1) / 2; ++p) {
                    const double2 x = *(const double2 *)(xs + (size_t)p * 2 * W + 2 * j);
                    s[2 * p] = fma(a, x.x, s[2 * p]);
                    if (2 * p + 1 < NC) s[2 * p + 1] = fma(a, x.y, s[2 * p + 1]);
                }
            };
            int j = l8;
#pragma unroll 1
            for (; j + 24 < W; j += 32) {
                double a[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) a[q] = row[j - l8 + 8 * q];
#pragma unroll
                for (int q = 0; q < 4; ++q) term(a[q], j + 8 * q);
            }
#pragma unroll 1
            for (; j < W; j += 8) term(row[j - l8], j);
#pragma unroll 1
            for (int q = P.rowptr[i] + l8; q < P.rowptr[i + 1]; q += 8) {
                const double *xj = x0 + P.colidx[q];
                const double v = P.val[q];
#pragma unroll
                for (int c = 0; c < NC; ++c)
                    if (c < nc) s[c] = fma(v, xj[(size_t)c * ld], s[c]);
            }
        }
        const int c = fa_sum8d<NP>(s, l8);
        if (on && (l8 & (8 / NP - 1)) == 0 && c < nc) Y[(size_t)(r0 + c) * ld + i] = s[0];
    }
}

// ---------------------------------------------------------------------------
// 4. expansion: CTA per (leaf, slice of NR rows, group of columns)
// ---------------------------------------------------------------------------
template <int NC>
__global__ void __launch_bounds__(128)
k_fa_expand(FaFar P, int NR, const double *__restrict__ ye, const double *__restrict__ yhat, double *__restrict__ Y,
            int64_t ld, FaWhen when)
{
    extern __shared__ __align__(16) unsigned char fa_sm[];
    __shared__ unsigned key[NC];
    const int lf = blockIdx.x, r0 = P.c0 + blockIdx.z * NC, k = P.k, w = P.nlev * k, ws = P.wp;
    if (fa_none(when) || fa_off(when, lf, r0)) return;
    const int b_leaf = P.kb[P.fl + lf], b = b_leaf + blockIdx.y * NR, e = min(P.ke[P.fl + lf], b + NR);
    if (b >= e) return;
    double *raw = (double *)fa_sm;
    if (threadIdx.x < NC) key[threadIdx.x] = 0;
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        unsigned mk = 0;
        const int r = r0 + c;
        for (int t = threadIdx.x; t < ws; t += blockDim.x) {
            double v = 0.0;
            if (t < w && r < P.nrhs) {
                const int lv = t / k, a = t - lv * k;
                const int node = ((P.fl + lf + 1) >> (P.nlev - 1 - lv)) - 1;
                if (yhat) {
                    v = yhat[((size_t)r * P.nnode + node) * k + a];
                } else {
                    const int q0 = P.fptr[node], q1 = P.fptr[node + 1];
                    const double *p = ye + (size_t)r * P.nfar * k + a;
#pragma unroll 4
                    for (int q = q0; q < q1; ++q) v += p[(size_t)q * k];
                }
            }
            raw[fa_slot<NC>(t, c, ws)] = v;
            mk = max(mk, fa_key(v));
        }
        mk = __reduce_max_sync(0xffffffffu, mk);
        if ((threadIdx.x & 31) == 0) atomicMax(&key[c], mk);
    }
    __syncthreads();
    bool slow = false;
#pragma unroll
    for (int c = 0; c < NC; ++c) slow |= fa_slow(key[c]);
    if (!slow) fa_convert<NC>(fa_sm, ws, key);
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, l8 = lane & 7, nw = blockDim.x >> 5;
    const int eu = P.ue[lf];
    for (int g0 = b + 4 * warp; g0 < e; g0 += 4 * nw) {
        const int i = g0 + (lane >> 3);
        const bool on = i < e;
        const int2 *row = P.U + (size_t)i * P.wp;
        if (!slow) {
            FaAcc s[NC];
            if (on) fa_row<NC>(row, w, l8, (const int4 *)fa_sm, ws, s);
            const int c = fa_sum8<NC>(s, l8), r = r0 + c;
            if (on && (l8 & (8 / NC - 1)) == 0 && r < P.nrhs)
                Y[(size_t)r * ld + i] += s[0].value() * fa_pow2(eu - 30) *
                                         fa_scale(key[c]);
        } else if (on) {
            for (int c = l8; c < NC && r0 + c < P.nrhs; c += 8) {
                double v = 0.0;
                for (int j = 0; j < w; ++j)
                    v = fma(P.Ud[((size_t)(j / k) * P.N + i) * k + j % k], raw[fa_slot<NC>(j, c, ws)], v);
                Y[(size_t)(r0 + c) * ld + i] += v;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// One column: the kernels stream the operator (781 MB at 27k DoFs and rank 64),
// so what bounds them is the number of loads in flight.  Every lane keeps two
// batches of eight 16-byte loads going; the first is issued before x is gathered.
// Measured against the column kernels above with NC = 1 (four loads ahead, none
// before the gather): coupling 94 -> 66 us, expansion 46 -> 38, projections 32 -> 22 us.
// The near rows are FP64 and bound by its pipe (k_fa_near1).
// ---------------------------------------------------------------------------
constexpr int FA_B = 8;

template <class L>
__device__ __forceinline__ void fa_batch(int4 *a, int t0, int n, L load)
{
#pragma unroll
    for (int q = 0; q < FA_B; ++q) a[q] = t0 + q < n ? load(t0 + q) : make_int4(0, 0, 0, 0);
}

// items 0..n-1 of a lane, a holding the first batch; use(item, t), zero items to
// the end of the last batch; carry() after every EVERY items
template <int EVERY, class L, class U, class C>
__device__ __forceinline__ void fa_pipe(int4 *a, int n, L load, U use, C carry)
{
#pragma unroll 1
    for (int t0 = 0; t0 < n; t0 += FA_B) {
        int4 b[FA_B];
        fa_batch(b, t0 + FA_B, n, load);
#pragma unroll
        for (int q = 0; q < FA_B; ++q) {
            use(a[q], min(t0 + q, n - 1));
            if ((q + 1) % EVERY == 0) carry();
        }
#pragma unroll
        for (int q = 0; q < FA_B; ++q) a[q] = b[q];
    }
}

__device__ __forceinline__ int4 fa_ld(const int4 *p) { return __ldcs(p); }   // streamed once

__global__ void __launch_bounds__(128)
k_fa_proj1(FaFar P, const double *__restrict__ X, double *__restrict__ part, const int *skip)
{
    extern __shared__ __align__(16) unsigned char fa_sm[];
    __shared__ unsigned key;
    if (skip && *skip) return;
    const int leaf = blockIdx.x, b = P.kb[P.fl + leaf], n = P.ke[P.fl + leaf] - b, w2 = P.wp >> 1;
    const int cp = blockIdx.y * blockDim.x + threadIdx.x;
    const int4 *M = (const int4 *)P.U + (size_t)b * w2 + min(cp, w2 - 1);
    auto load = [&](int t) { return __ldg(M + (size_t)t * w2); };   // read again by the expansion
    int4 a[FA_B];
    fa_batch(a, 0, n, load);
    double *raw = (double *)fa_sm;
    int2 *xs = (int2 *)fa_sm;
    if (threadIdx.x == 0) key = 0;
    __syncthreads();
    unsigned mk = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        raw[i] = X[b + i];
        mk = max(mk, fa_key(raw[i]));
    }
    mk = __reduce_max_sync(0xffffffffu, mk);
    if ((threadIdx.x & 31) == 0 && mk) atomicMax(&key, mk);
    __syncthreads();
    const unsigned ky = key;
    const bool slow = fa_slow(ky);
    if (!slow)
        for (int i = threadIdx.x; i < n; i += blockDim.x) xs[i] = fa_split(fa_round(raw[i], ky));
    __syncthreads();
    FaAcc s0, s1;
    if (!slow)
        fa_pipe<4>(a, n, load,
                [&](int4 m, int t) {
                    const int2 x = xs[t];
                    s0.mac(make_int2(m.x, m.y), x);
                    s1.mac(make_int2(m.z, m.w), x);
                },
                [&] { s0.carry(), s1.carry(); });
    s0.fold();
    s1.fold();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int col = 2 * cp + h, lv = col / P.k, al = col - lv * P.k;
        if (cp >= w2 || lv >= P.nlev) continue;
        double v = (h ? s1 : s0).value() * fa_pow2(P.ue[leaf] - 30) * fa_scale(ky);
        if (slow) {
            v = 0.0;
            for (int i = 0; i < n; ++i) v = fma(P.Ud[((size_t)lv * P.N + b + i) * P.k + al], raw[i], v);
        }
        part[((size_t)lv * P.nleaf + leaf) * P.k + al] = v;
    }
}

__global__ void __launch_bounds__(32 * FC_WARPS)
k_fa_couple1(FaFar P, const double *__restrict__ part, const double *__restrict__ xhat, double *__restrict__ ye,
             const int *skip)
{
    __shared__ int2 xs_[FC_WARPS][KMAX];
    if (skip && *skip) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, e = blockIdx.x * FC_WARPS + warp, k = P.k;
    if (e >= P.nfar) return;
    // lanes over the pairs of columns, the rest of the warp over the rows
    const int np = P.kp >> 1, ga = np > 16 ? 32 : np > 8 ? 16 : np > 4 ? 8 : 4, gb = 32 / ga;
    const int pr = lane & (ga - 1), lb = lane / ga, n = (k + gb - 1) / gb;
    const int4 *S = (const int4 *)P.S + (size_t)e * k * np + min(pr, np - 1);
    auto load = [&](int t) {
        const int b = lb + t * gb;
        return b < k ? fa_ld(S + (size_t)b * np) : make_int4(0, 0, 0, 0);
    };
    int4 a[FA_B];
    fa_batch(a, 0, n, load);
    int2 *xs = xs_[warp];
    double *raw = (double *)xs;
    const bool hard = P.hard[e];
    const short *se = P.se + (size_t)e * k + 2 * min(pr, np - 1);
    const int es0 = se[0], es1 = 2 * min(pr, np - 1) + 1 < k ? se[1] : 0;
    const int node = P.fcol[e], l = 31 - __clz(node + 1), sh = P.L - l, leaf0 = ((node + 1) << sh) - (1 << P.L);
    unsigned ky = 0;
    for (int b = lane; b < k; b += 32) {
        double v = 0.0;
        if (xhat) {
            v = xhat[(size_t)node * k + b];
        } else {
            const double *p = part + ((size_t)(l - P.lmin) * P.nleaf + leaf0) * k + b;
#pragma unroll 8
            for (int j = 0; j < (1 << sh); ++j) v += p[(size_t)j * k];
        }
        raw[b] = v;
        ky = max(ky, fa_key(v));
    }
    ky = __reduce_max_sync(0xffffffffu, ky);
    __syncwarp();
    double *out = ye + (size_t)e * k;
    if (fa_slow(ky) || hard) {
        for (int al = lane; al < k; al += 32) {
            double v = 0.0;
#pragma unroll 8
            for (int b = 0; b < k; ++b) v = fma(P.Sd[((size_t)e * k + b) * k + al], raw[b], v);
            out[al] = v;
        }
        return;
    }
    for (int b = lane; b < k; b += 32) xs[b] = fa_split(fa_round(raw[b], ky));
    __syncwarp();
    FaAcc s0, s1;
    fa_pipe<4>(a, n, load,
            [&](int4 m, int t) {
                const int2 x = xs[min(lb + t * gb, k - 1)];   // the row past the end is zero
                s0.mac(make_int2(m.x, m.y), x);
                s1.mac(make_int2(m.z, m.w), x);
            },
            [&] { s0.carry(), s1.carry(); });
    s0.fold();
    s1.fold();
    double v0 = s0.value(), v1 = s1.value();
    for (int o = ga; o < 32; o <<= 1) {
        v0 += __shfl_xor_sync(0xffffffffu, v0, o);
        v1 += __shfl_xor_sync(0xffffffffu, v1, o);
    }
    if (lb == 0 && pr < np) {
        const double sx = fa_scale(ky);
        out[2 * pr] = v0 * fa_pow2(max(es0, -900) - 30) * sx;
        if (2 * pr + 1 < k) out[2 * pr + 1] = v1 * fa_pow2(max(es1, -900) - 30) * sx;
    }
}

// gathered piece of one column (W entries of raw), its key in *key: fixed-point in place; true where it stays FP64
__device__ __forceinline__ bool fa_piece(unsigned char *sm, int W, unsigned mk, unsigned *key, unsigned &ky)
{
    mk = __reduce_max_sync(0xffffffffu, mk);
    if ((threadIdx.x & 31) == 0 && mk) atomicMax(key, mk);
    __syncthreads();
    ky = *key;
    const bool slow = fa_slow(ky);
    if (!slow) fa_convert<1>(sm, W, &ky);
    __syncthreads();
    return slow;
}

// partial of X . Y over the rows of this CTA (CG's p . A p comes with the apply): v the
// product of a row in the lanes with l8 = 0, zero in the others
__device__ __forceinline__ void fa_dot(double v, double *dot)
{
    __shared__ double sh[4];
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    v += __shfl_xor_sync(0xffffffffu, v, 16);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) dot[blockIdx.x * gridDim.y + blockIdx.y] = (sh[0] + sh[1]) + (sh[2] + sh[3]);
}

// 16 rows a CTA, 4 a warp, 8 lanes a row, FP64; dot: see fa_dot, or null.  What bounds it is
// the FP64 pipe (26M multiply-adds at 27k DoFs: 42 us at its rate), so batches of four loads
// and more CTAs: one column at 16129 DoFs and rank 16 / at 27k and rank 64, batches of eight
// 73 / 181 us, of four and at least 8 CTAs an SM 66 / 171, of two and 16 CTAs 71 / 171.
__global__ void __launch_bounds__(128, 8)
k_fa_near1(FaNear P, const double *__restrict__ X, double *__restrict__ Y, double *__restrict__ dot, FaWhen when)
{
    extern __shared__ __align__(16) unsigned char fa_sm[];
    if (fa_none(when) || fa_off(when, 0, P.c0)) return;
    const int lf = blockIdx.x, b_leaf = P.kb[P.fl + lf], b = b_leaf + blockIdx.y * 16, e = min(P.ke[P.fl + lf], b + 16);
    if (b >= e) {
        if (dot && threadIdx.x == 0) dot[blockIdx.x * gridDim.y + blockIdx.y] = 0.0;
        return;
    }
    const int W = P.pw[lf], lane = threadIdx.x & 31, l8 = lane & 7, i = b + 4 * (threadIdx.x >> 5) + (lane >> 3);
    const double2 *row = (const double2 *)(P.Dd + P.poff[lf] + (size_t)(min(i, e - 1) - b_leaf) * W);
    const int nv = W >> 1, n = (nv + 7) >> 3;
    auto fill = [&](double2 *a, int t0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int v = l8 + 8 * (t0 + q);
            a[q] = v < nv ? __ldcs(row + v) : make_double2(0.0, 0.0);
        }
    };
    double2 a[4];
    fill(a, 0);
    const int *gc = P.gcol + P.goff[lf];
    double *xs = (double *)fa_sm;
#pragma unroll 4
    for (int t = threadIdx.x; t < W; t += blockDim.x) {
        const int j = gc[t];
        xs[t] = j >= 0 ? X[j] : 0.0;
    }
    double bm = 0.0, s0 = 0.0, s1 = 0.0;
    if (i < e)
        for (int q = P.rowptr[i] + l8; q < P.rowptr[i + 1]; q += 8) bm = fma(P.val[q], X[P.colidx[q]], bm);
    __syncthreads();
    const double2 *x2 = (const double2 *)xs;
#pragma unroll 1
    for (int t0 = 0; t0 < n; t0 += 4) {
        double2 next[4];
        fill(next, t0 + 4);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (t0 + q >= n) break;   // the same for the CTA: a product of zeros would take its FP64 time
            const int v = l8 + 8 * (t0 + q);
            const double2 x = v < nv ? x2[v] : make_double2(0.0, 0.0);   // (an Inf times the zero entry past the end)
            s0 = fma(a[q].x, x.x, s0);
            s1 = fma(a[q].y, x.y, s1);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] = next[q];
    }
    // B + M last: the diagonal's product is the largest term of a row
    s0 = (s0 + s1) + bm;
    fa_sum8d<1>(&s0, l8);
    double xy = 0.0;
    if (i < e && !l8) {
        Y[i] = s0;
        if (dot) xy = X[i] * s0;
    }
    if (dot) fa_dot(xy, dot);
}

__global__ void __launch_bounds__(128)
k_fa_expand1(FaFar P, const double *__restrict__ ye, const double *__restrict__ yhat, double *__restrict__ Y,
             const double *__restrict__ X, double *__restrict__ dot, const int *skip)
{
    extern __shared__ __align__(16) unsigned char fa_sm[];
    __shared__ unsigned key;
    if (skip && *skip) return;
    const int lf = blockIdx.x, k = P.k, w = P.nlev * k, b0 = P.kb[P.fl + lf];
    const int b = b0 + blockIdx.y * 16, e = min(P.ke[P.fl + lf], b + 16);
    if (b >= e) {
        if (dot && threadIdx.x == 0) dot[blockIdx.x * gridDim.y + blockIdx.y] = 0.0;
        return;
    }
    const int lane = threadIdx.x & 31, l8 = lane & 7, i = b + 4 * (threadIdx.x >> 5) + (lane >> 3);
    const int nv = P.wp >> 1, n = (nv + 7) >> 3;
    const int4 *row = (const int4 *)P.U + (size_t)min(i, e - 1) * nv + l8;
    auto load = [&](int t) { return l8 + 8 * t < nv ? __ldg(row + 8 * t) : make_int4(0, 0, 0, 0); };
    int4 a[FA_B];
    fa_batch(a, 0, n, load);
    double *raw = (double *)fa_sm;
    if (threadIdx.x == 0) key = 0;
    __syncthreads();
    unsigned mk = 0, ky;
#pragma unroll 2
    for (int t = threadIdx.x; t < P.wp; t += blockDim.x) {
        double v = 0.0;
        if (t < w) {
            const int lv = t / k, al = t - lv * k, node = ((P.fl + lf + 1) >> (P.nlev - 1 - lv)) - 1;
            if (yhat) {
                v = yhat[(size_t)node * k + al];
            } else {
                const int q1 = P.fptr[node + 1];
#pragma unroll 8
                for (int q = P.fptr[node]; q < q1; ++q) v += ye[(size_t)q * k + al];
            }
        }
        raw[t] = v;
        mk = max(mk, fa_key(v));
    }
    const bool slow = fa_piece(fa_sm, P.wp, mk, &key, ky);
    FaAcc s;
    if (!slow)
        fa_pipe<2>(a, n, load,
                [&](int4 m, int t) {
                    const int4 x = ((const int4 *)fa_sm)[min(l8 + 8 * t, nv - 1)];
                    s.mac(make_int2(m.x, m.y), make_int2(x.x, x.y));
                    s.mac(make_int2(m.z, m.w), make_int2(x.z, x.w));
                },
                [&] { s.carry(); });
    s.fold();
    fa_sum8<1>(&s, l8);
    double xy = 0.0;
    if (i < e && !l8) {
        double v = s.value() * fa_pow2(P.ue[lf] - 30) * fa_scale(ky);
        if (slow) {
            v = 0.0;
            for (int j = 0; j < w; ++j) v = fma(P.Ud[((size_t)(j / k) * P.N + i) * k + j % k], raw[j], v);
        }
        v += Y[i];
        Y[i] = v;
        if (dot) xy = X[i] * v;
    }
    if (dot) fa_dot(xy, dot);
}


// ---------------------------------------------------------------------------
// the operands
// ---------------------------------------------------------------------------
// whether a piece with this largest key is in the format's range
__device__ __forceinline__ bool fa_fits(unsigned key) { return !key || (key >= 200u && key <= 1900u); }

// largest exponent key of n values (warp), as the exponent E with |v| < 2^E;
// flags what the format cannot hold
__device__ __forceinline__ int fa_exponent(unsigned key, int *err)
{
    key = __reduce_max_sync(0xffffffffu, key);
    if (!fa_fits(key)) {
        if ((threadIdx.x & 31) == 0) atomicOr(err, 4);
        return 0;
    }
    return key ? (int)key - 1022 : 0;
}

// near panel rows, a warp each, for the many-column apply: the entries at the positions of B + M
// (the row's largest, 2^5 to 2^8 above the next) go to val8 with B + M and stay FP64
__global__ void k_fa_build_near(int N, int fl, const int *__restrict__ vleaf, const int *__restrict__ kb,
                                const int *__restrict__ pw, const int64_t *__restrict__ poff,
                                const double *__restrict__ D, const int *__restrict__ rowptr,
                                const int64_t *__restrict__ bpos, const double *__restrict__ val,
                                double *__restrict__ val8, int2 *__restrict__ out, int *__restrict__ re, int *err)
{
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (i >= N) return;
    const int lf = vleaf[i], W = pw[lf];
    const size_t o = poff[lf] + (size_t)(i - kb[fl + lf]) * W;
    for (int j = lane; j < W; j += 32) out[o + j] = make_int2(0, 0);
    __syncwarp();
    for (int q = rowptr[i] + lane; q < rowptr[i + 1]; q += 32) {   // distinct positions, marked
        const int64_t p = bpos[q];
        val8[q] = val[q] + (p >= 0 ? D[p] : 0.0);
        if (p >= 0) out[p] = make_int2(1, 0);
    }
    __syncwarp();
    unsigned key = 0;
    for (int j = lane; j < W; j += 32)
        if (!out[o + j].x) key = max(key, fa_key(D[o + j]));
    const int E = fa_exponent(key, err);
    for (int j = lane; j < W; j += 32) out[o + j] = out[o + j].x ? make_int2(0, 0) : fa_split(fa_round(D[o + j], E + 1022));
    if (lane == 0) re[i] = E;
}

// coupling blocks, a CTA per row node, rows padded to an even length; an exponent per row of a
// block.  Entries down to 2^-8 of their row's largest keep all their bits; a block with a
// smaller one is marked hard.  low, least: smallest entry of a row (in its scale) and of the block.
__global__ void __launch_bounds__(256)
k_fa_build_S(const int *__restrict__ fptr, int k, int kp, const double *__restrict__ S, int2 *__restrict__ out,
             short *__restrict__ se, float *__restrict__ low, unsigned char *__restrict__ hard, int *__restrict__ row,
             double *__restrict__ least, int *err)
{
    const int node = blockIdx.x, e0 = fptr[node], ne = fptr[node + 1] - e0;
    for (int e = threadIdx.x; e < ne; e += 256) {
        hard[e0 + e] = 0;
        row[e0 + e] = node;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < ne * k; t += 256) {
        const int e = t / k, a = t - e * k;
        const double *in = S + (size_t)(e0 + e) * k * k + a;
        unsigned key = 0, lk = 0x7ffu;
        double v = INFINITY;
        for (int b = 0; b < k; ++b) {
            const double x = fabs(in[(size_t)b * k]);
            const unsigned q = fa_key(x);
            key = max(key, q);
            if (q) lk = min(lk, q);
            v = fmin(v, x);
        }
        if (!fa_fits(key)) atomicOr(err, 4);
        if (key > lk + 7) hard[e0 + e] = 1;
        se[(size_t)(e0 + e) * k + a] = (short)(key ? (int)key - 1022 : -2000);   // a row of zeros: below all others
        low[(size_t)(e0 + e) * k + a] = key ? (float)scalbn(v, 1022 - (int)key) : 0.0f;
        int2 *o = out + (size_t)(e0 + e) * k * kp + a;
        for (int b = 0; b < k; ++b) o[(size_t)b * kp] = fa_split(fa_round(in[(size_t)b * k], (int)key));
        if (a == k - 1 && kp > k)
            for (int b = 0; b < k; ++b) o[(size_t)b * kp + 1] = make_int2(0, 0);
    }
    for (int e = threadIdx.x >> 5; e < ne; e += 8) {   // a warp per block
        double v = INFINITY;
        for (int i = threadIdx.x & 31; i < k * k; i += 32) v = fmin(v, fabs(S[(size_t)(e0 + e) * k * k + i]));
        for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
        if ((threadIdx.x & 31) == 0) least[e0 + e] = v;
    }
}

// flattened bases, CTA per leaf: [level][N][k] -> [N][level k], rows padded to an even length
__global__ void __launch_bounds__(256) k_fa_build_U(int fl, int N, int k, int nlev, const int *__restrict__ kb, const int *__restrict__ ke,
                             const double *__restrict__ U, int2 *__restrict__ out, int *__restrict__ ue,
                             float *__restrict__ umin, int *err)
{
    __shared__ unsigned key;
    __shared__ int E;
    __shared__ float least[8];
    const int b = kb[fl + blockIdx.x], n = ke[fl + blockIdx.x] - b, w = nlev * k, wp = (w + 1) & ~1;
    if (threadIdx.x == 0) key = 0;
    __syncthreads();
    unsigned mk = 0;
    for (int t = threadIdx.x; t < n * w; t += blockDim.x) {
        const int i = b + t / w, q = t % w;
        mk = max(mk, fa_key(U[((size_t)(q / k) * N + i) * k + q % k]));
    }
    atomicMax(&key, mk);
    __syncthreads();
    if (threadIdx.x < 32) {
        const int e = fa_exponent(key, err);
        if (threadIdx.x == 0) E = e;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < n * wp; t += blockDim.x) {
        const int i = b + t / wp, q = t % wp;
        out[(size_t)i * wp + q] =
            q < w ? fa_split(fa_round(U[((size_t)(q / k) * N + i) * k + q % k], E + 1022)) : make_int2(0, 0);
    }
    float r = INFINITY;   // the rows sum to the DoFs' weights, the same at every level
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        double t = 0.0;
        for (int q = 0; q < k; ++q) t += U[(size_t)(b + i) * k + q];
        r = fminf(r, (float)(fabs(t) * fa_pow2(-E)));
    }
    for (int o = 16; o > 0; o >>= 1) r = fminf(r, __shfl_xor_sync(0xffffffffu, r, o));
    if ((threadIdx.x & 31) == 0) least[threadIdx.x >> 5] = r;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < 8; ++q) r = fminf(r, least[q]);
        ue[blockIdx.x] = E;
        umin[blockIdx.x] = r;
    }
}

}  // namespace

// the mesh's flattened bases (geometry only, end of the mesh setup)
void build_fixed_bases(MeshData &m)
{
    const int nlev = m.nfar > 0 ? m.kt.L - m.far_lmin + 1 : 0;
    m.fa_ok = true;
    if (!nlev) return;
    DBuf<int> err;
    m.fa_ok = if_memory([&] {
        err.alloc(1);
        m.fa_U.alloc((size_t)((nlev * m.k + 1) & ~1) * m.N);
        m.fa_ue.alloc(m.kt.nleaf);
        m.fa_umin.alloc(m.kt.nleaf);
    });
    if (!m.fa_ok) {
        m.fa_U.release();
        return;
    }
    err.zero(nullptr);
    k_fa_build_U<<<m.kt.nleaf, 256>>>(m.kt.first_leaf(), m.N, m.k, nlev, m.kt_begin.p, m.kt_end.p, m.Ul64.p,
                                      (int2 *)m.fa_U.p, m.fa_ue.p, m.fa_umin.p, err.p);
    VFD_CUDA(cudaGetLastError());
    int h = 0;
    VFD_CUDA(cudaMemcpy(&h, err.p, sizeof(int), cudaMemcpyDeviceToHost));
    if (h) {
        m.fa_ok = false;
        m.fa_U.release();
    }
}

void release_fixed_operator(OpData &op)
{
    op.fa_D.release();
    op.fa_re.release();
    op.fa_val.release();
    op.fa_S.release();
    op.fa_se.release();
    op.fa_low.release();
    op.fa_hard.release();
    op.fa_row.release();
    op.fa_min.release();
}

// The operator's coupling blocks, and its near panels where the mesh has the lists of the
// many-column apply; err gets bit 2 where an entry does not fit.  The copies are as large as
// the FP64 operator: they are made where they take at most half of the memory that is left
// (false: not), so that what fits without them fits.
bool build_fixed_operator(const MeshData &m, OpData &op, int *err, cudaStream_t st)
{
    const int kp = (m.k + 1) & ~1;
    const bool panels = m.td_rows.n > 0;
    size_t left = 0, total = 0;
    VFD_CUDA(cudaMemGetInfo(&left, &total));
    const size_t need = (panels ? (size_t)m.near_entries * 8 : 0) + (size_t)m.nfar * m.k * (kp * 8 + 8);
    const bool ok = need <= left / 2 && if_memory([&] {
        if (panels) {
            op.fa_D.alloc(m.near_entries);
            op.fa_re.alloc(m.N);
            op.fa_val.alloc(m.nnz);
        }
        if (m.nfar) {
            op.fa_S.alloc((size_t)m.nfar * m.k * kp);
            op.fa_se.alloc((size_t)m.nfar * m.k);
            op.fa_low.alloc((size_t)m.nfar * m.k);
            op.fa_hard.alloc(m.nfar);
            op.fa_row.alloc(m.nfar);
            op.fa_min.alloc(m.nfar);
        }
    });
    if (!ok) {
        release_fixed_operator(op);
        return false;
    }
    if (panels)
        k_fa_build_near<<<cdiv((long long)m.N * 32, 256), 256, 0, st>>>(
            m.N, m.kt.first_leaf(), m.vleaf.p, m.kt_begin.p, m.panel_w.p, m.panel_off.p, op.D64.p, m.rowptr.p, m.bm_pos.p,
            op.valBM.p, op.fa_val.p, (int2 *)op.fa_D.p, op.fa_re.p, err);
    if (m.nfar)
        k_fa_build_S<<<m.kt.nnode, 256, 0, st>>>(m.far_ptr.p, m.k, kp, op.S64.p, (int2 *)op.fa_S.p, op.fa_se.p, op.fa_low.p,
                                                 op.fa_hard.p, op.fa_row.p, op.fa_min.p, err);
    VFD_CUDA(cudaGetLastError());
    return true;
}

namespace {

// rows of a CTA: the whole leaf, or down to 16 rows where that leaves SMs idle, although each
// CTA gathers the columns again (the apply, 64 rows / this rule: 5 columns at 9025 DoFs and rank 16
// 106 / 73 us, 8 columns at 3997 DoFs and rank 64 235 / 116, 64 columns at 817 DoFs 128 / 83)
int rows_of(const MeshData &m, int ctas)
{
    int nr = 64;
    while (nr > 16 && (long long)ctas * cdiv(m.max_leaf_size, nr) < 304) nr >>= 1;
    return nr;
}

template <class K>
void allow_shared(K kernel, size_t shm)
{
    VFD_REQUIRE(shm <= 227 * 1024, VFD_EUNSUPPORTED,
                "apply: a near panel is wider than shared memory holds (use a low-rank operator, lambda > 0)");
    if (shm > 47 * 1024)
        VFD_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
}

// the far field's kernels up to the expansion, on the side stream, for ng groups of NC columns from column c0
template <int NC>
void far_group(const MeshData &m, OpData &op, const double *X, int c0, int ng, int nrhs, int64_t ld, bool summed,
               const int *skip)
{
    FaWhen when;
    when.skip = skip;
    const int k = m.k, nleaf = m.kt.nleaf;
    FaFar P = fa_far_view(m, op);
    P.nrhs = nrhs;
    P.c0 = c0;
    const int w = P.nlev * k, cols = std::min(nrhs - c0, ng * NC);
    // one column: the kernels get its own pieces
    const size_t ps = (size_t)P.nlev * nleaf * k, hs = (size_t)m.kt.nnode * k, ys = (size_t)m.nfar * k;
    const size_t shp = (size_t)m.max_leaf_size * NC * 8;
    if constexpr (NC == 1)
        k_fa_proj1<<<dim3(nleaf, cdiv(w, 256)), 128, shp, op.side>>>(P, X + (size_t)c0 * ld, op.P64.p + c0 * ps, skip);
    else
        k_fa_proj<NC><<<dim3(nleaf, cdiv(w, 128), ng), 128, shp, op.side>>>(P, X, ld, op.P64.p, when);
    if (summed) launch_far_sum(m, op, c0, cols, op.side, skip);
    if constexpr (NC == 1)
        k_fa_couple1<<<cdiv(m.nfar, FC_WARPS), 32 * FC_WARPS, 0, op.side>>>(
            P, op.P64.p + c0 * ps, summed ? op.xhat.p + c0 * hs : nullptr, op.ye64.p + c0 * ys, skip);
    else
        k_fa_couple<NC><<<dim3(cdiv(m.nfar, FC_WARPS), ng), 32 * FC_WARPS, 0, op.side>>>(
            P, op.P64.p, summed ? op.xhat.p : nullptr, op.ye64.p, when);
    if (summed) launch_far_couple_sum(m, op, c0, cols, op.side, skip);
    VFD_CUDA(cudaGetLastError());
}

template <int NC>
void expand_group(const MeshData &m, OpData &op, const double *X, double *Y, int c0, int ng, int nrhs, int64_t ld,
                  bool summed, cudaStream_t st, const FaWhen &when, ApplyDot *dot)
{
    FaFar P = fa_far_view(m, op);
    P.nrhs = nrhs;
    P.c0 = c0;
    const size_t hs = (size_t)m.kt.nnode * m.k, ys = (size_t)m.nfar * m.k, shm = (size_t)P.wp * NC * 8;
    if constexpr (NC == 1) {
        k_fa_expand1<<<dim3(m.kt.nleaf, cdiv(m.max_leaf_size, 16)), 128, shm, st>>>(
            P, op.ye64.p + c0 * ys, summed ? op.yhat.p + c0 * hs : nullptr, Y + (size_t)c0 * ld, X + (size_t)c0 * ld,
            dot ? dot->part : nullptr, when.skip);
    } else {
        allow_shared(k_fa_expand<NC>, shm);
        const int nr = rows_of(m, m.kt.nleaf * ng);
        k_fa_expand<NC><<<dim3(m.kt.nleaf, cdiv(m.max_leaf_size, nr), ng), 128, shm, st>>>(
            P, nr, op.ye64.p, summed ? op.yhat.p : nullptr, Y, ld, when);
    }
    VFD_CUDA(cudaGetLastError());
}

template <int NC>
void near_group(const MeshData &m, OpData &op, const double *X, double *Y, int c0, int ng, int nrhs, int64_t ld,
                cudaStream_t st, const FaWhen &when, double *dot)
{
    FaNear R = fa_near_view(m, op);
    R.nrhs = nrhs;
    R.c0 = c0;
    const size_t shm = (size_t)m.max_panel_w * (NC == 1 ? 1 : (NC + 1) & ~1) * 8;
    if constexpr (NC == 1) {
        allow_shared(k_fa_near1, shm);
        k_fa_near1<<<dim3(m.kt.nleaf, cdiv(m.max_leaf_size, 16)), 128, shm, st>>>(R, X + (size_t)c0 * ld,
                                                                                 Y + (size_t)c0 * ld, dot, when);
    } else {
        allow_shared(k_fa_near<NC>, shm);
        R.NR = rows_of(m, m.kt.nleaf * ng);
        k_fa_near<NC><<<dim3(m.kt.nleaf, cdiv(m.max_leaf_size, R.NR), ng), 128, shm, st>>>(R, X, ld, Y, when);
    }
    VFD_CUDA(cudaGetLastError());
}

// f(NC) with the number of columns of a group as a constant, 1 .. 8
template <class F>
void with_columns(int n, F f)
{
    switch (n) {
    case 1: f(std::integral_constant<int, 1>()); break;
    case 2: f(std::integral_constant<int, 2>()); break;
    case 3: f(std::integral_constant<int, 3>()); break;
    case 4: f(std::integral_constant<int, 4>()); break;
    case 5: f(std::integral_constant<int, 5>()); break;
    case 6: f(std::integral_constant<int, 6>()); break;
    case 7: f(std::integral_constant<int, 7>()); break;
    default: f(std::integral_constant<int, 8>());
    }
}

// widest near group: its panel piece leaves room for two CTAs an SM
int near_columns(const MeshData &m)
{
    int nc = 8;
    while (nc > 1 && (size_t)m.max_panel_w * nc * 8 > 100 * 1024) nc >>= 1;
    return nc;
}

}  // namespace

// Y = A X with the FP64 operator (all parts); the workspaces are those of the FP64 apply
void apply_fixed(const MeshData &m, OpData &op, const double *X, double *Y, int nrhs, int64_t ld, cudaStream_t st,
                 const int *skip, ApplyDot *dot)
{
    if (dot) dot->n = nrhs == 1 ? m.kt.nleaf * cdiv(m.max_leaf_size, 16) : 0;
    if (dot && !dot->n) dot = nullptr;
    if (!skip && !dot && apply_tensor_fits(m, op, nrhs)) return apply_tensor(m, op, X, Y, nrhs, ld, st);
    FaWhen when;
    when.skip = skip;
    // the node sums inside the gathers pay for few columns and short spans (sums inside / of their own:
    // 3 columns at 27361 DoFs 432 / 395 us, 16129 182 / 171, 3721 61 / 59; 2 columns at 27361 258 / 270,
    // 10267 138 / 160, 3997 51 / 58)
    const bool summed = nrhs >= 3 || m.kt.L - m.far_lmin > 7, far = m.nfar > 0;
    // far groups: of 8, the remainder in one group of the next power of two
    auto far_groups = [&](auto f) {
        int c0 = 0;
        auto go = [&](int n, int ng) {
            with_columns(n, [&](auto NC) {
                if constexpr ((NC & (NC - 1)) == 0) f(NC, c0, ng);
            });
            c0 += n * ng;
        };
        if (nrhs / 8) go(8, nrhs / 8);
        if (c0 < nrhs) {
            int r = 1;
            while (r < nrhs - c0) r <<= 1;
            go(r, 1);
        }
    };
    if (far) {
        VFD_CUDA(cudaEventRecord(op.ev_fork, st));
        VFD_CUDA(cudaStreamWaitEvent(op.side, op.ev_fork, 0));
        far_groups([&](auto NC, int c0, int ng) { far_group<NC>(m, op, X, c0, ng, nrhs, ld, summed, skip); });
    }
    const int nc = near_columns(m);
    auto near = [&](int n, int c0, int ng) {
        with_columns(n, [&](auto NC) {
            near_group<NC>(m, op, X, Y, c0, ng, nrhs, ld, st, when, dot && !far ? dot->part : nullptr);
        });
    };
    if (nc == 1)
        for (int c = 0; c < nrhs; ++c) near(1, c, 1);
    else if (nrhs / nc)
        near(nc, 0, nrhs / nc);
    if (nc > 1 && nrhs % nc) near(nrhs % nc, nrhs / nc * nc, 1);
    if (far) {
        VFD_CUDA(cudaEventRecord(op.ev_join, op.side));
        VFD_CUDA(cudaStreamWaitEvent(st, op.ev_join, 0));
        far_groups([&](auto NC, int c0, int ng) { expand_group<NC>(m, op, X, Y, c0, ng, nrhs, ld, summed, st, when, dot); });
    }
}

// the kernels above with the sums as kernels of their own, on st, for what the many-column apply
// leaves to them
void apply_fixed_redo(FaStep step, const MeshData &m, OpData &op, const double *X, double *Y, int c0, int ng, int nrhs,
                      int64_t ld, cudaStream_t st, const FaWhen &when)
{
    FaFar P = fa_far_view(m, op);
    P.nrhs = nrhs;
    P.c0 = c0;
    // (grids of a size at which a launch with nothing to do costs a few microseconds)
    const int nc = near_columns(m);
    if (step == FA_PROJ)
        k_fa_proj<8><<<dim3(std::min(m.kt.nleaf, 64), cdiv(P.nlev * m.k, 128), ng), 128, (size_t)m.max_leaf_size * 64, st>>>(
            P, X, ld, op.P64.p, when);
    else if (step == FA_COUPLE)
        k_fa_couple<8><<<dim3(std::min(cdiv(m.nfar, FC_WARPS), 608), ng), 32 * FC_WARPS, 0, st>>>(P, op.P64.p, op.xhat.p,
                                                                                                op.ye64.p, when);
    else if (step == FA_EXPAND)
        expand_group<8>(m, op, X, Y, c0, ng, nrhs, ld, true, st, when, nullptr);
    else
        with_columns(nc, [&](auto NC) {
            const int cols = std::min(nrhs - c0, 8 * ng);
            if constexpr (NC == 1)
                for (int c = c0; c < c0 + cols; ++c) near_group<1>(m, op, X, Y, c, 1, nrhs, ld, st, when, nullptr);
            else
                near_group<NC>(m, op, X, Y, c0, cdiv(cols, (int)NC), nrhs, ld, st, when, nullptr);
        });
    VFD_CUDA(cudaGetLastError());
}

}  // namespace vfd
