// Fixed-point numbers and views of the operator shared by the fixed-point applies
// (the scheme is described in apply_fixed.cu).
#pragma once

#include "device_common.cuh"

namespace vfd {

typedef long long i64;
typedef unsigned long long u64;

constexpr int FA_LO = 30, FA_TOP = 40;

// exponent key of a value: 0 for zero, else its biased exponent (denormals 1)
__device__ __forceinline__ unsigned fa_key(double v)
{
    // the exponent field is masked after the shift: a mask of the sign bit alone becomes
    // an FP64 absolute value, which leaves the sign of a NaN
    const unsigned h = (unsigned)__double2hiint(v);
    return (h << 1 | (unsigned)__double2loint(v)) == 0 ? 0u : max(1u, (h >> 20) & 0x7ffu);
}
// keys of a piece that the fixed-point products cannot take
__device__ __forceinline__ bool fa_slow(unsigned key) { return key == 0x7ffu || (key && key < 128u); }

// v 2^(60 - E) rounded, E = key - 1022 with key the largest of the piece
__device__ __forceinline__ i64 fa_round(double v, int key)
{
    const u64 b = (u64)__double_as_longlong(v);
    const int e = (int)((b >> 52) & 0x7ff), s = e - key + 7;
    const u64 m = (b & 0xfffffffffffffULL) | (e ? 1ULL << 52 : 0ULL);
    const u64 r = s >= 0 ? m << s : (s > -64 ? (m + (1ULL << (-s - 1))) >> -s : 0ULL);
    return (i64)b < 0 ? -(i64)r : (i64)r;
}
__device__ __forceinline__ int2 fa_split(i64 v)
{
    const int lo = (int)((unsigned)v << (32 - FA_LO)) >> (32 - FA_LO);
    return make_int2(lo, (int)((v - lo) >> FA_LO));
}
// 2^k as FP64, -1022 <= k <= 1023
__device__ __forceinline__ double fa_pow2(int k) { return __longlong_as_double((i64)(k + 1023) << 52); }
// scale of a piece: 2^(E - 30), E = key - 1022 (any for a piece of zeros)
__device__ __forceinline__ double fa_scale(unsigned key) { return fa_pow2(key ? (int)key - 1022 - 30 : 0); }
// sums of products: carry() after every fourth mac at most (seven fit)
struct FaAcc {
    i64 hh = 0, mid = 0;
    int th = 0, tm = 0;   // what hh and mid have passed on, weight 2^FA_TOP
    __device__ __forceinline__ void mac(int2 a, int2 x)
    {
        hh += (i64)a.y * x.y;
        mid += (i64)a.y * x.x;
        mid += (i64)a.x * x.y;
    }
    __device__ __forceinline__ void carry()
    {
        th += (int)(hh >> FA_TOP);
        hh &= (1LL << FA_TOP) - 1;
        tm += (int)(mid >> FA_TOP);
        mid &= (1LL << FA_TOP) - 1;
    }
    // after carry: hh takes mid, rounded (the sum is th 2^FA_TOP + hh in units of 2^60)
    __device__ __forceinline__ void fold()
    {
        hh += ((mid + (1LL << (FA_LO - 1))) >> FA_LO) + ((i64)tm << (FA_TOP - FA_LO));
    }
    __device__ __forceinline__ double value() const { return fma((double)th, 1099511627776.0, (double)hh); }
};

// Which of a kernel's items run: none where *skip is set; with a mask those whose bit of this
// group of columns is set (item 0 of near), or all where *err is set
struct FaWhen {
    const int *skip = nullptr;
    const unsigned *mask = nullptr;
    const int *any = nullptr;   // 0: no item's bit is set
    const int *err = nullptr;
    int c0 = 0;   // first column of the mask's bit 0
};
// nothing to do at all; nothing for this item
__device__ __forceinline__ bool fa_none(const FaWhen &w)
{
    return (w.skip && *w.skip) || (w.mask && !*w.any && !*w.err);
}
__device__ __forceinline__ bool fa_off(const FaWhen &w, int item, int r0)
{
    return w.mask && !*w.err && !(w.mask[item] >> ((r0 - w.c0) >> 3) & 1u);
}

// sum over the 8 lanes of a row; every lane ends with one column, returned, and its sum in s[0]
template <int NC>
__device__ __forceinline__ int fa_sum8d(double *s, int l8)
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
                    const double send = up ? s[q] : s[q + n], keep = up ? s[q + n] : s[q];
                    s[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
            col += up ? n : 0;
        } else {
            s[0] += __shfl_xor_sync(0xffffffffu, s[0], o);
        }
    }
    return col;
}

struct FaFar {
    int fl, nleaf, lmin, L, nlev, k, nnode, nfar, nrhs, c0;   // c0: first column of this launch
    int kp, wp;   // row strides of a coupling block and of the bases (even: 16-byte rows)
    const int *kb, *ke, *fptr, *fcol;
    const int2 *U, *S;
    const int *ue;
    const short *se;         // exponents of a block's rows
    const unsigned char *hard;   // blocks that stay FP64
    const int *row;          // row node of a block
    const double *Ud, *Sd;   // FP64: [level][N][k], blocks
    int N;
};

struct FaNear {
    int fl, NR, nrhs, c0;
    const int *kb, *ke, *pw, *gcol, *goff, *rowptr, *colidx;
    const int64_t *poff;
    const double *val;   // B + M
    const double *val8;  // B + M plus the panel entries at its positions, which D leaves out
    const int2 *D;
    const int *re;
    const double *Dd;    // FP64 panels
};

inline FaFar fa_far_view(const MeshData &m, const OpData &op)
{
    FaFar P{};
    P.fl = m.kt.first_leaf();
    P.nleaf = m.kt.nleaf;
    P.lmin = m.far_lmin;
    P.L = m.kt.L;
    P.nlev = m.nfar > 0 ? m.kt.L - m.far_lmin + 1 : 0;
    P.k = m.k;
    P.kp = (m.k + 1) & ~1;
    P.wp = (P.nlev * m.k + 1) & ~1;
    P.nnode = m.kt.nnode;
    P.nfar = m.nfar;
    P.nrhs = 1;
    P.kb = m.kt_begin.p;
    P.ke = m.kt_end.p;
    P.fptr = m.far_ptr.p;
    P.fcol = m.far_col.p;
    P.U = (const int2 *)m.fa_U.p;
    P.S = (const int2 *)op.fa_S.p;
    P.ue = m.fa_ue.p;
    P.se = op.fa_se.p;
    P.hard = op.fa_hard.p;
    P.row = op.fa_row.p;
    P.Ud = m.Ul64.p;
    P.Sd = op.S64.p;
    P.N = m.N;
    return P;
}

inline FaNear fa_near_view(const MeshData &m, const OpData &op)
{
    FaNear R{};
    R.fl = m.kt.first_leaf();
    R.nrhs = 1;
    R.kb = m.kt_begin.p;
    R.ke = m.kt_end.p;
    R.pw = m.panel_w.p;
    R.gcol = m.gcol.p;
    R.goff = m.gcol_off.p;
    R.rowptr = m.rowptr.p;
    R.colidx = m.colidx.p;
    R.poff = m.panel_off.p;
    R.val = op.valBM.p;
    R.val8 = op.fa_val.p;
    R.D = (const int2 *)op.fa_D.p;
    R.re = op.fa_re.p;
    R.Dd = op.D64.p;
    return R;
}

}  // namespace vfd
