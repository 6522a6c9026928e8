// The kernel gamma in 64-bit fixed point.
//
// One FP64 instruction takes a warp 16 cycles of an SM on this part (2 lanes a
// cycle), a 32-bit integer multiply-add half a cycle to one.  A kernel
// evaluation exp2(A - B ln r^2) in FP64 costs about 30 FP64 instructions; here
// it is 32 x 32 -> 64 bit products and carries only: table-driven logarithm
// and exponential (P. T. P. Tang, ACM TOMS 15(2) 1989 and 16(4) 1990) on
// fixed-point operands.  Rates and errors, this path and FP64, are given at the
// end of the comment.
//
// Formats (Qn: an integer v stands for v 2^-n):
//   coordinates  X = (x - o) 2^62 / W, |X| <= 2^61, W = 2^w above the diagonal
//                of the mesh's box and o its centre: |X - X'| < 2^62 per axis
//                and r^2 < W^2
//   b            b / ln 2 of a point, Q61, b = s/2 + d/4 in [0, 2 ln 2)
//   a            base-2 exponent of a point, Q53: log2(kappa)/2 - 2 w b (plus the
//                log of a quadrature weight where it is folded in)
//   N            -ln(r^2 / W^2) >= 0, Q56
//   gamma        2^(a_x + a_y + (b_x + b_y) N), rounded to FP64
// The error of N is below 2^-56, so that of the exponent is below 2^-53: FP64
// arithmetic carries the rounding of an exponent of size 10 to 40 instead.
// What the formats cannot hold (s outside the range of b, extreme kappa, meshes
// with cells below 2^-16 of the box, where the rounding of X matters) stays
// on the FP64 path: MeshData::fx_ok and OpData::fx say which applies.
//
// Measured (points of [-1,1]^2 at distances 2^-10 to 1, s in [0.05, 0.9], against
// 113-bit arithmetic): relative error 1.0e-15 rms and 4.8e-15 at most, FP64
// 1.6e-15 and 1.2e-14; 163 G evaluations/s with all SMs busy, FP64 16.2 G/s.
#pragma once

#include "vfd_internal.h"

namespace vfd {

typedef unsigned long long u64;
typedef long long i64;

// table in 64-bit words: FX_LOGN pairs (c_j, T_j), c_j = ceil(2^31 / F_j) (Q31),
// F_j = 1 + j/1024, T_j = -ln c_j (Q56); then 2^(j/2048), j < 2048 (Q63, with
// 7/16 of a unit of the final rounding added)
constexpr int FX_LOGN = 1024, FX_EXPN = 2048, FX_WORDS = 2 * FX_LOGN + FX_EXPN;
constexpr size_t FX_BYTES = FX_WORDS * sizeof(u64);

struct FxTab {
    const ulonglong2 *lg;
    const u64 *ex;
};

// copy the table to shared memory (16-byte aligned); the caller synchronises
__device__ __forceinline__ FxTab fx_stage(const u64 *__restrict__ g, u64 *sh)
{
    const ulonglong2 *s = (const ulonglong2 *)g;
    ulonglong2 *t = (ulonglong2 *)sh;
    for (int i = threadIdx.x; i < FX_WORDS / 2; i += blockDim.x) t[i] = __ldg(s + i);
    return {t, sh + 2 * FX_LOGN};
}

__device__ __forceinline__ u64 fx_wide(unsigned a, unsigned b) { return (u64)a * b; }

// r^2 / W^2 = M 2^(-K), M in [1, 2) as Q63, from the coordinate differences
// (one's complement in place of the absolute value: off by one unit, 2^-62 W)
template <int D>
__device__ __forceinline__ void fx_r2(const i64 *x, const i64 *y, u64 &M, int &K)
{
    unsigned hi[D], lo[D], h = 0;
#pragma unroll
    for (int c = 0; c < D; ++c) {
        const u64 t = (u64)(x[c] - y[c]);
        const unsigned th = (unsigned)(t >> 32), sg = (unsigned)((int)th >> 31);
        hi[c] = th ^ sg;
        lo[c] = (unsigned)t ^ sg;
        h |= hi[c];
    }
    const int s = __clz(h) - 1;   // the largest difference gets its leading bit at 62
    u64 S = 0;
#pragma unroll
    for (int c = 0; c < D; ++c) {
        const unsigned a = __funnelshift_l(lo[c], hi[c], s), b = lo[c] << (s & 31);
        S += fx_wide(a, a) + (fx_wide(a, b) >> 31);
    }
    const int z = __clz((unsigned)(S >> 32));
    M = S << (z & 31);
    K = 2 * s + z - 3;
}

// the same of a positive normal FP64 number times 2^(-2w)
__device__ __forceinline__ void fx_r2(double r2, int w, u64 &M, int &K)
{
    const u64 b = (u64)__double_as_longlong(r2);
    M = (b << 11) | 0x8000000000000000ULL;
    K = 1023 + 2 * w - (int)(b >> 52);
}

// N = -ln(M 2^-K) in Q56; ln(1 + r) = r - r^2/2 + r^3 (1/3 - r/4 + r^2/5), r < 2^-10
// (the next term is below 2^-62)
__device__ __forceinline__ u64 fx_neglog(const FxTab &t, u64 M, int K)
{
    const unsigned mh = (unsigned)(M >> 32), ml = (unsigned)M;
    const ulonglong2 e = t.lg[(mh >> 21) & (FX_LOGN - 1)];
    const unsigned c = (unsigned)e.x;
    const u64 r = fx_wide(mh, c) + (fx_wide(ml, c) >> 32) - (1ULL << 62);   // Q62
    const unsigned rh = (unsigned)(r >> 20), rl = (unsigned)r << 12;        // r = (rh + rl 2^-32) 2^-42
    const u64 r2 = fx_wide(rh, rh) + (fx_wide(rh, rl) >> 31);               // Q84
    const unsigned r3 = __umulhi((unsigned)(r2 >> 32), rh);                 // Q62
    const unsigned p = 0x55555555u - __umulhi(rh, (1u << 20) - __umulhi(rh, 819u));
    const u64 v = r - (r2 >> 23) + __umulhi(r3, p);                         // ln(1 + r), Q62
    // K ln 2: Q56 and the 32 bits below
    const u64 kl = (u64)(i64)K * 0xB17217F7D1CF79ULL + (fx_wide((unsigned)K, 0xABC9E3B4u) >> 32);
    return kl - e.y - (v >> 6);
}

// 2^(A + B N) as FP64
__device__ __forceinline__ double fx_exp(const FxTab &t, i64 A, u64 B, u64 N)
{
    const unsigned bh = (unsigned)(B >> 32), bl = (unsigned)B, nh = (unsigned)(N >> 32), nl = (unsigned)N;
    const u64 mid = fx_wide(bl, nh) + fx_wide(bh, nl);
    const u64 E = (u64)A + fx_wide(bh, nh) + (mid >> 32);   // Q53
    const unsigned eh = (unsigned)(E >> 32), el = (unsigned)E;
    const u64 T = t.ex[(eh >> 10) & (FX_EXPN - 1)];
    // 2^g - 1 = g ln 2 + g^2 (c2 + g (c3 + g c4)), g < 2^-11 as (gh + gl 2^-32) 2^-43
    const unsigned gh = __funnelshift_l(el, eh, 22), gl = el << 22;
    const u64 p1 = fx_wide(gh, 0xB17217F7u) + __umulhi(gh, 0xD1CF79ABu) + __umulhi(gl, 0xB17217F7u);   // Q75
    const unsigned q = 4127059954u + __umulhi(gh, 465603u + __umulhi(gh, 39u));                        // Q34
    const u64 p = p1 + (fx_wide(gh, __umulhi(gh, q)) >> 13);
    const unsigned th = (unsigned)(T >> 32), tl = (unsigned)T, ph = (unsigned)(p >> 32), pl = (unsigned)p;
    const u64 tp = fx_wide(th, ph) + __umulhi(th, pl) + __umulhi(tl, ph);   // T p, Q74
    const u64 m = T + (tp >> 11);
    const u64 bits = (m >> 11) + ((u64)(unsigned)(((int)eh >> 21) + 1022) << 52);
    return __longlong_as_double((i64)bits);
}

// exponent terms (a, b) of a point with field values s, log kappa; false (and
// zeros) where they do not fit the formats
__device__ __forceinline__ bool fx_terms(int d, int w, double s, double lk, i64 &A, i64 &B)
{
    A = B = 0;
    if (!(s >= -0.5 * d && 0.5 * s + 0.25 * d < 1.38 && fabs(lk) < 100.0)) return false;
    const i64 b = __double2ll_rn(s * 2305843009213693952.0) + ((i64)d << 60);   // Q62: s 2^61 and d 2^60
    B = (i64)__umul64hi((u64)b, 0xB8AA3B295C17F0BCULL);                          // times 1/ln 2 (Q63): Q61
    const i64 l = __mul64hi(__double2ll_rn(lk * 72057594037927936.0), 0x5C551D94AE0BF85ELL);   // Q56 x 1/(2 ln 2) (Q63)
    A = ((l + 2) >> 2) - (((b >> 6) * (2 * w)) >> 3);
    return true;
}

// the same for the sums of s and of log kappa over two points that fit (2D)
__device__ __forceinline__ void fx_sums(int w, double s, double lk, i64 &A, u64 &B)
{
    const u64 b = (u64)__double2ll_rn(s * 2305843009213693952.0) + (1ULL << 62);   // Q62, below 2^64
    B = __umul64hi(b, 0xB8AA3B295C17F0BCULL);
    const i64 l = __mul64hi(__double2ll_rn(lk * 36028797018963968.0), 0x5C551D94AE0BF85ELL);   // Q55 x Q63
    A = ((l + 1) >> 1) - (((i64)(b >> 6) * (2 * w)) >> 3);
}

template <int D>
__device__ __forceinline__ double fx_gamma(const FxTab &t, const i64 *x, const i64 *y, i64 A, u64 B)
{
    u64 M;
    int K;
    fx_r2<D>(x, y, M, K);
    return fx_exp(t, A, B, fx_neglog(t, M, K));
}

}  // namespace vfd
