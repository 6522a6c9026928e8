// The FP64 operator apply of many columns on the tensor cores, in exact integer digits.
//
// The fixed-point products of apply_fixed.cu cost three 32-bit multiply-adds each,
// about 5 cycles of an SM and warp with their carries.  Here an entry (62 bits: the
// fixed-point integer times 4) is cut into eight digits of base 2^8 in [-128, 127],
// exact in FP16, and the digits of the two factors are multiplied by tcgen05.mma
// (kind::f16, FP32 accumulators in tensor memory):
//   a x = sum_{i, j} 2^(8 (i + j)) a_i x_j,
// the 36 products with i + j >= 7.  Products of equal i + j share an accumulator, 8 of
// them, and after 160 products at most they move to 96-bit integers in registers: 6 pairs
// of 160 stay below 2^24 and are exact; of the two lowest accumulators (8 and 7 pairs) a
// sum above 2^24 is rounded by less than the dropped pairs add up to.  So the result is
// that of integer arithmetic up to the dropped pairs, about 2^-62 of the two scales a product.
//
// Scales.  A row of the operator has one (near panel rows, rows of a coupling block, bases of
// a leaf), and so has a leaf's or node's piece of the columns of a tile; the cutting warps
// shift the entries of a piece to the largest scale of the sum.  The diagonal and the other
// entries at B + M's positions, 2^5 to 2^8 above the next, are left out of the near
// panels and summed in FP64 (k_td_csr).  Sums that a scale would still cost precision are
// found before they are used and done without digits ("What the digits cannot hold").
//
// A CTA computes 128 rows (two halves of 64: sibling leaves, sibling nodes) of a tile
// of NC columns.  The digit planes of the vector lie one after the other along N, so
// one instruction multiplies plane i of the operator by planes 7 - i .. 7 of the vector
// into neighbouring accumulators: N = NC (i + 1).  Sibling rows share most of their
// partners, and a partner's vector digits serve both halves (records built with the
// mesh: build_tensor_lists); a half without the partner multiplies zeros.
//
//   k_td_max, k_td_digits   x -> digits per leaf, in the order the instruction reads
//   k_td_csr, k_td_near     Y = B + M and the large entries, FP64; rows that stay FP64
//   k_td<PROJ>              projections, then the node sums (apply.cu), digits per node
//   k_td<COUPLE>            coupling blocks summed per node, digits per node
//   k_td<ROWS>              near panel rows and the expansion of a leaf, added to Y
//
// Warp roles of k_td, per step of 16 rows of a partner:
//   warps 0-15 copy the operator's integers (apply_fixed.cu) two steps ahead and cut them
//              into digit planes in shared memory; after every 10 steps at most they move
//              the accumulators on
//   warp 16    lane 0 issues the products (it waits where the tensor cores are behind, so
//              it cannot also cut); the warp owns the tensor memory
//   warp 17    lane 0 copies the vector's digits of the step (cp.async.bulk)
// Every wait is bounded by a count of cycles; a CTA whose wait expires raises err, waits
// (bounded again) for its copies and products, and returns.  What the digits of such a
// launch should have given is then redone by the kernels of apply_fixed.cu.
//
// What bounds it: 36 products of 128 x 64 x 16 (12 instructions) are 1152 cycles of the
// tensor cores, cutting a step 800 to 1100 cycles of 16 warps beside them, and a move of the
// accumulators (64 K conversions at 16 a cycle, 64-bit sums) about 6000 cycles in which
// the tensor cores wait.  64 normal columns at 27361 DoFs and rank 64: 1.42 ms (fixed point 5.27,
// FP64 kernels 11.88): rows 458, coupling 362, projections 148, node sums 77, digits and
// their scales 150, B + M 85, checks and alignment 60 us.  (With one scale a column for the
// whole mesh and one a row with the diagonal in it, which lost up to 20 bits, 1.15 ms.)
// The same digits with mma.sync m16n8k16 (600 TFLOP/s against 2.2 PFLOP/s) took 2664 us.
// Errors in units of |A||x| (meshes of 800 to 1000 DoFs, against extended precision), FP64
// kernels and here: normal columns 6.4e-17 and 4.7e-17 rms, 3.2e-16 and 3.6e-16 at most;
// columns over six decades 8.8e-17 and 9.3e-17; falling by 14 decades across the mesh
// 5.4e-17 and 4.7e-17; columns of the operator agree to 9e-16.
#include <cuda_fp16.h>

#include <algorithm>

#include "apply_common.cuh"
#include "apply_fixed.cuh"

namespace vfd {

namespace {

constexpr int TD_D = 8;                     // digits
constexpr int TD_G = 8;                     // accumulators: i + j = 7 .. 14
constexpr int TD_COLS = 64;                 // columns of a pass
constexpr int TD_NST = 4;                   // stages
constexpr int TD_MOVE = 10;                 // steps between two moves of the accumulators at most
constexpr int TD_LAG = 3;                   // steps cut ahead of a move of the accumulators
constexpr int TD_CW = 16;                   // cutting warps
constexpr int TD_AHEAD = 2;                 // steps whose entries are on their way
constexpr int TD_RAW = TD_CW * 32 * 32;     // bytes of a step's entries
constexpr int TD_THREADS = 32 * (TD_CW + 2);
constexpr int TD_A = 128 * 16 * TD_D * 2;   // bytes of the operator's digits of a step
constexpr int TD_SMS = 152;                // CTAs of a launch and tile: one an SM
constexpr double TD_HZ = 2e9;               // SM cycles a second, about
constexpr long long TD_WAIT = (long long)TD_HZ;   // of an aborted CTA's waits, and the default of the others
enum { TD_PROJ, TD_COUPLE, TD_ROWS };

// bytes of the vector's digits of a step: [digit][column / 8][row / 8][column % 8][row % 8],
// i.e. core matrices of 8 columns x 16 bytes
__host__ __device__ constexpr int td_step(int nc) { return nc * 16 * TD_D * 2; }

struct TdVec {          // a set of pieces of a matrix of columns
    const double *v;
    size_t ld, base;    // column stride; offset of piece 0 (nodes)
    int npiece, ns, len;                 // ns: steps of a piece; len: rows of a piece (nodes)
    const int *kb, *ke;                  // rows of a piece (leaves), or null
    int nrhs, c0, nc;                    // columns c0 .. min(c0 + 64, nrhs) in tiles of nc
    int node0, lmin, nlev;               // nodes: the first, its level; keys of nlev levels (1: one for all)
    unsigned *key, *piece;               // largest keys: per level and column of the pass; per piece and column
    int *w;                              // [tile][piece]: exponent of a piece's scale less the columns'
    unsigned char *out;                  // [tile][piece][step]
    float *n1;                           // sum of a piece's |x| in units of its scale, [piece][64]
};

__device__ __forceinline__ void td_range(const TdVec &P, int p, size_t &b, int &n)
{
    b = P.kb ? (size_t)P.kb[p] : P.base + (size_t)p * P.len;
    n = P.kb ? P.ke[p] - (int)b : P.len;
}

// largest key of every piece and column, and of every column (over a level's pieces); CTA per
// piece, a warp per column
__global__ void __launch_bounds__(256) k_td_max(TdVec P)
{
    const int p = blockIdx.x, lane = threadIdx.x & 31;
    size_t b;
    int n;
    td_range(P, p, b, n);
    unsigned *key = P.key + (P.nlev > 1 ? 31 - __clz(P.node0 + p + 1) - P.lmin : 0) * TD_COLS;
    double v[8][2];
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int h = 0; h < 2; ++h) {   // a piece has at most 64 rows
            const int c = (threadIdx.x >> 5) + 8 * u, i = lane + 32 * h;
            v[u][h] = P.c0 + c < P.nrhs && i < n ? P.v[(size_t)(P.c0 + c) * P.ld + b + i] : 0.0;
        }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int c = (threadIdx.x >> 5) + 8 * u;
        const unsigned mk = __reduce_max_sync(0xffffffffu, max(fa_key(v[u][0]), fa_key(v[u][1])));
        if (lane == 0) {
            P.piece[(size_t)p * TD_COLS + c] = mk;
            if (mk > key[c]) atomicMax(key + c, mk);
        }
    }
}

// digits of piece blockIdx.x for tile blockIdx.y; a thread takes 8 rows of a column.  A piece has
// one scale for the tile's columns: where they are all small in it (a solution where its
// equation is stiff, a vector that is local) the bits are not spent on zeros.  (A column that
// does not fit gets zeros; its sums are redone.)
// (A program's 64 solutions for random loads at 27k DoFs, s from 0.1 to 0.9: 1645 us an apply,
// with scales in steps of 2^4 3616, because 36% of the nodes are redone.)
constexpr int TD_WMIN = -60;
__global__ void __launch_bounds__(256) k_td_digits(TdVec P)
{
    __shared__ float red[2 * ((KMAX + 15) / 16)][TD_COLS];
    __shared__ int w;
    const int p = blockIdx.x;
    size_t b;
    int n;
    td_range(P, p, b, n);
    const unsigned *keys = P.key + (P.nlev > 1 ? 31 - __clz(P.node0 + p + 1) - P.lmin : 0) * TD_COLS;
    unsigned char *out = P.out + ((size_t)blockIdx.y * P.npiece + p) * P.ns * td_step(P.nc);
    if (threadIdx.x == 0) w = TD_WMIN;
    __syncthreads();
    if ((int)threadIdx.x < P.nc) {
        const int r = blockIdx.y * P.nc + threadIdx.x;
        const unsigned key = keys[r], own = P.piece[(size_t)p * TD_COLS + r];
        if (P.c0 + r < P.nrhs && own && !fa_slow(key)) atomicMax(&w, (int)own - (int)key);
    }
    __syncthreads();
    if (threadIdx.x == 0) P.w[(size_t)blockIdx.y * P.npiece + p] = w;
    for (int t = threadIdx.x; t < P.nc * 2 * P.ns; t += 256) {
        const int ch = t / P.nc, col = t % P.nc, r = blockIdx.y * P.nc + col;
        const bool on = P.c0 + r < P.nrhs;
        const unsigned key = on ? keys[r] : 0u;
        const bool fits = on && !fa_slow(key);
        const double *v = P.v + (size_t)(P.c0 + r) * P.ld + b;
        u64 d[8];
        float sum = 0.0f;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int i = ch * 8 + q;
            const double y = fits && i < n ? v[i] : 0.0;
            const i64 x = fa_round(y, (int)key + w);
            sum += y != 0.0 ? fmaxf((float)llabs(x) * 0x1p-60f, 1e-30f) : 0.0f;   // an entry that rounds to zero counts
            d[q] = (u64)(x << 2) + 0x8080808080808080ULL;   // digits plus 128
        }
        red[ch][col] = sum;
        unsigned char *o = out + (size_t)(ch >> 1) * td_step(P.nc) + (ch & 1) * 128 + (col & 7) * 16;
#pragma unroll
        for (int i = 0; i < TD_D; ++i) {
            half2 h[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const unsigned u = (unsigned)(d[2 * q] >> (8 * i)) & 255u, w_ = (unsigned)(d[2 * q + 1] >> (8 * i)) & 255u;
                h[q] = __halves2half2(__int2half_rn((int)u - 128), __int2half_rn((int)w_ - 128));
            }
            *(uint4 *)(o + (size_t)(i * (P.nc >> 3) + (col >> 3)) * 256) = *(const uint4 *)h;
        }
    }
    __syncthreads();
    if ((int)threadIdx.x < P.nc) {
        float t = 0.0f;
        for (int ch = 0; ch < 2 * P.ns; ++ch) t += red[ch][threadIdx.x];
        P.n1[(size_t)p * TD_COLS + blockIdx.y * P.nc + threadIdx.x] = t;
    }
}

struct TdP {
    FaFar F;
    FaNear R;
    int nrhs, c0, nsl, nsn, node0, nnodes;   // steps of a leaf and of a node; nodes node0 .. node0 + nnodes
    const unsigned char *dx, *dh;            // digits of the leaves' x; of the nodes' xhat or yhat
    const unsigned *kx, *kh;                 // their column keys (COUPLE: kh per level)
    const int *wx;                           // PROJ: exponents of the leaves' scales, [tile][leaf]
    const short *er, *ef;                    // ROWS: exponents of near rows, [tile][N], and expansions, [tile][leaf]
    const uchar2 *shr;                       // ROWS: shifts of a record's halves to them, [tile][record]
    int nrec;
    const short *ec;                         // COUPLE: exponents of a node's rows, [tile][node][k]
    const unsigned char *sh;                 // COUPLE: shifts of a block's rows to them, [tile][block][k]
    const int *bin;                          // items of a CTA (build_tensor_lists)
    const int4 *items;
    const TdRec *rec;
    int *err;
    long long wait;                          // cycles after which a wait gives up
};

__device__ __forceinline__ unsigned td_sa(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

// SM cycles (reading the global timer instead takes about a microsecond)
__device__ __forceinline__ u64 td_timer() { return (u64)clock64(); }

__device__ __forceinline__ bool td_wait(unsigned bar, unsigned parity, u64 deadline)
{
    while (true) {
        unsigned done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if (td_timer() > deadline) return false;
    }
}
__device__ __forceinline__ void td_arrive(unsigned bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void td_commit(unsigned bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}

// K-major operand without swizzle: core matrices of 8 rows x 16 bytes, the two of a
// step's 16 rows 128 bytes apart, groups of 8 rows 256 bytes apart
__device__ __forceinline__ u64 td_desc(unsigned a)
{
    return (u64)((a & 0x3FFFF) >> 4) | (u64)(128 >> 4) << 16 | (u64)(256 >> 4) << 32 | (u64)1 << 46;
}
// FP32 accumulator, FP16 operands, both K-major, M = 128
__device__ __forceinline__ void td_mma(unsigned d, unsigned a, unsigned b, int n, bool acc)
{
    const unsigned idesc = (1u << 4) | ((unsigned)(n >> 3) << 17) | ((128u >> 4) << 24);
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
                 "l"(td_desc(a)), "l"(td_desc(b)), "r"(idesc), "r"((unsigned)acc));
}

// (h 2^32 + l) 2^(56 + e) rounded to FP64 with integers (two conversions, a multiply-add
// and a scaling in FP64 would be 80 cycles of the SM a warp), but for results that are not normal
__device__ __forceinline__ double td_value(i64 h, unsigned l, int e)
{
    const i64 h0 = h;
    const unsigned l0 = l;
    const bool neg = h < 0;
    if (neg) {
        h = ~h + (l == 0);
        l = 0u - l;
    }
    const bool big = (u64)h >> 32 != 0;
    const u64 a = big ? (u64)h : (u64)h << 32 | l;
    const int z = __clzll(a);
    const u64 t = z == 64 ? 0 : a << z | (big ? l >> (32 - z) : 0u);   // leading one at 63
    const int b = 1023 + 56 + 95 - z - (big ? 0 : 32) + e;
    if (t != 0 && (b < 2 || b > 2045)) return scalbn(fma((double)h0, 4294967296.0, (double)l0), 56 + e);
    const u64 r = (((t >> 1) + 512) >> 10) + ((u64)(b - 1) << 52);
    return __longlong_as_double(t ? (i64)(r | (neg ? 1ULL << 63 : 0ULL)) : 0LL);
}

// a b + c, kept a multiply-add (as shifts and 64-bit adds it takes four instructions)
__device__ __forceinline__ i64 td_mad(int a, int b, i64 c)
{
    i64 r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}

// exponent of a sum of digit products: entries below 2^ea, a column with this key
__device__ __forceinline__ int td_exp(int ea, unsigned key) { return ea + (key ? (int)key - 1022 : 0) - 2 * 62; }

// where a role stands: piece q of an item, its partner, rows and the half's offset
struct TdIt {
    int i, item, q, q1, q2, col, n, nrow, W;   // i: of the CTA's items
    i64 off;
    uchar2 sh;
};

template <int NC, int MODE>
__global__ void __launch_bounds__(TD_THREADS, 1)
k_td(TdP P, int nitem, const double *__restrict__ X, int64_t ld, double *__restrict__ out)
{
    extern __shared__ __align__(1024) unsigned char td_sm[];
    constexpr int STAGE = TD_A + td_step(NC), NH = NC / 4;
    u64 *bars = (u64 *)(td_sm + TD_NST * STAGE + TD_AHEAD * TD_RAW);   // A full, B full, empty [stages each], moved, drained
    unsigned *tslot = (unsigned *)(bars + 3 * TD_NST + 2);
    volatile int *abort_f = (volatile int *)(tslot + 1);
    unsigned *skey = tslot + 2;   // column keys of the tile: leaves, nodes
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tile = blockIdx.y;
    const unsigned bar0 = td_sa(bars), base = td_sa(td_sm);
    auto fullA = [&](int s) { return bar0 + 8u * s; };
    auto fullB = [&](int s) { return bar0 + 8u * (TD_NST + s); };
    auto empty = [&](int s) { return bar0 + 8u * (2 * TD_NST + s); };
    const unsigned moved = bar0 + 24u * TD_NST, drained = moved + 8u;
    if (threadIdx.x == 0) {
        for (int s = 0; s < TD_NST; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(fullA(s)), "r"(TD_CW));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(fullB(s)), "r"(1));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(empty(s)), "r"(1));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(moved), "r"(1));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(drained), "r"(TD_CW));
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        *abort_f = 0;
    }
    if (warp == TD_CW) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(td_sa(tslot)), "n"(TD_G * NC));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    if (threadIdx.x < 2 * NC) {
        const unsigned *key = threadIdx.x < NC ? P.kx : P.kh;
        skey[threadIdx.x] = key ? key[tile * NC + (int)threadIdx.x % NC] : 0u;
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const unsigned taddr = *tslot;
    const u64 deadline = td_timer() + P.wait;

    // Items: pairs of leaves (ROWS), of nodes (COUPLE), 128 columns of a leaf's bases (PROJ).
    // An item's records q .. q2, the first section up to q1 (ROWS: near, then far).
    const int k = P.F.k, half = warp >> 3 & 1, nz = (P.F.nlev * k + 127) >> 7;
    const int ibeg = MODE == TD_PROJ ? (int)((i64)nitem * blockIdx.x / gridDim.x) : P.bin[blockIdx.x];
    const int iend = MODE == TD_PROJ ? (int)((i64)nitem * (blockIdx.x + 1) / gridDim.x) : P.bin[blockIdx.x + 1];
    auto record = [&](TdIt &I) {
        if (MODE == TD_PROJ) return;
        const TdRec r = P.rec[I.q];
        I.col = r.col;
        I.n = r.n;
        I.off = r.off[half];
        if (MODE == TD_ROWS) I.sh = P.shr[(size_t)tile * P.nrec + I.q];
    };
    auto start = [&](TdIt &I) {   // first piece of item I.i; false: no more items
        I.n = 0;
        if (I.i >= iend) return false;
        if (MODE == TD_PROJ) {
            const int leaf = I.i / nz, c0 = (I.i - leaf * nz) * 128 + half * 64;
            const int b = P.F.kb[P.F.fl + leaf], n = P.F.ke[P.F.fl + leaf] - b;
            I.item = I.i;
            I.q = 0;
            I.q1 = I.q2 = 1;
            I.col = leaf;
            I.n = max(n, 1);
            I.off = n > 0 ? (i64)b * P.F.wp + c0 : -1;
            I.nrow = max(0, min(64, P.F.nlev * k - c0));
        } else {
            const int4 v = P.items[I.i];
            I.q = v.x;
            I.q1 = v.y;
            I.q2 = v.z;
            I.item = v.w;
            I.nrow = k;
        }
        if (MODE == TD_ROWS) {
            const int leaf = 2 * I.item + half;
            I.nrow = leaf < P.F.nleaf ? P.R.ke[P.R.fl + leaf] - P.R.kb[P.R.fl + leaf] : 0;
            I.W = leaf < P.F.nleaf ? P.R.pw[leaf] : 0;
        }
        record(I);
        return true;
    };
    auto next = [&](TdIt &I) {
        if (++I.q < I.q2) {
            record(I);
            return true;
        }
        ++I.i;
        return start(I);
    };
    // 0: nothing after this step; 1: move the accumulators; 2, 3: and end the first, second section
    int since = 0;
    auto code_of = [&](int end, bool last) {
        const int c = last ? end : 0;
        since = c || since == TD_MOVE - 1 ? 0 : since + 1;
        return c ? c : (since == 0 ? 1 : 0);
    };
    TdIt I{};
    I.i = ibeg;
    bool have = start(I), ok = true;
    int issued = 0, moves = 0;   // steps of the products, of the copies; moves of the accumulators
    if (warp < TD_CW) {
        // cutting: 8 rows a warp; a lane takes 4 neighbouring entries of a row
        const int g = lane >> 1 & 7, tt = 8 * (lane >> 4) + 4 * (lane & 1);   // row, first entry
        const int mrow = (warp & 7) * 8 + g;   // this lane's row in the half
        // reading the accumulators: row of the tile, columns
        const int orow = 32 * (warp & 3) + lane, ohalf = orow >> 6, om = orow & 63, oc = (warp >> 2) * NH;
        i64 sh[NH];   // sums in units of 2^56: sh 2^32 + sl
        unsigned sl[NH];
#pragma unroll
        for (int c = 0; c < NH; ++c) sh[c] = sl[c] = 0;
        int m8 = 256, m16 = 65536, m24 = 16777216;
        asm("" : "+r"(m8), "+r"(m16), "+r"(m24));   // in registers: not shifts
        int ei = ibeg;   // the item that ends next
        auto emit = [&](int code) {
            int ri = 0, e = 0;   // row of out
            bool on = false;
            size_t os = (size_t)ld;   // column stride
            const int item = MODE == TD_PROJ ? ei : P.items[ei].w;
            if (MODE != TD_ROWS || code == 3 || P.F.nlev == 0) ++ei;
            if (MODE == TD_PROJ) {
                const int leaf = item / nz, c = (item - leaf * nz) * 128 + orow, lv = c / k;
                on = c < P.F.nlev * k;
                ri = (lv * P.F.nleaf + leaf) * k + c - lv * k;
                e = P.F.ue[leaf] + P.wx[tile * P.F.nleaf + leaf];
                os = (size_t)P.F.nlev * P.F.nleaf * k;
            }
            if (MODE == TD_ROWS) {
                const int leaf = 2 * item + ohalf;
                if (leaf < P.F.nleaf) {
                    const int b = P.R.kb[P.R.fl + leaf];
                    ri = b + om;
                    on = om < P.R.ke[P.R.fl + leaf] - b;
                    if (on) e = code == 2 ? P.er[(size_t)tile * P.F.N + ri] : P.ef[tile * P.F.nleaf + leaf];
                }
            }
            if (MODE == TD_COUPLE) {
                const int node = P.node0 + 2 * item + ohalf;
                on = node < P.F.nnode && om < k;
                ri = node * k + om;
                if (on) e = P.ec[((size_t)tile * P.nnodes + node - P.node0) * k + om];
                os = (size_t)P.F.nnode * k;
            }
            const unsigned *key = skey + oc + (MODE == TD_PROJ || (MODE == TD_ROWS && code == 2) ? 0 : NC);
            if (MODE == TD_COUPLE)   // the pair's level
                key = P.kh + (31 - __clz(P.node0 + 2 * item + 1) - P.F.lmin) * TD_COLS + tile * NC + oc;
            double *o = out + ri;
            const int r0 = P.c0 + tile * NC + oc, nr = on ? P.nrhs - r0 : 0;   // columns 0 .. nr of this thread
            o += (size_t)r0 * os;
#pragma unroll
            for (int c0 = 0; c0 < NH; c0 += 2) {
                double v[2], y[2];
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    v[j] = td_value(sh[c0 + j], sl[c0 + j], td_exp(e, key[c0 + j]));
                    sh[c0 + j] = sl[c0 + j] = 0;
                    if (MODE == TD_ROWS) y[j] = c0 + j < nr ? o[(c0 + j) * os] : 0.0;
                }
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    if (MODE == TD_ROWS) v[j] += y[j];
                    if (c0 + j < nr) o[(c0 + j) * os] = v[j];
                }
            }
        };
        auto move = [&](int code) {
            if (!td_wait(moved, moves & 1, deadline)) return false;
            ++moves;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
#pragma unroll
            for (int c = 0; c < NH; c += 2) {
                unsigned f[TD_G][2];
#pragma unroll
                for (int q = 0; q < TD_G; ++q)
                    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];\n"
                                 : "=r"(f[q][0]), "=r"(f[q][1])
                                 : "r"(taddr + ((unsigned)(32 * (warp & 3)) << 16) + (unsigned)(q * NC + oc + c)));
                asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    int v[TD_G];
#pragma unroll
                    for (int q = 0; q < TD_G; ++q) v[q] = __float2int_rn(__uint_as_float(f[q][j]));
                    i64 lo = td_mad(v[1], m8, (i64)v[0]);
                    lo = td_mad(v[3], m24, td_mad(v[2], m16, lo));
                    i64 hi = td_mad(v[5], m8, (lo >> 32) + v[4]);
                    hi = td_mad(v[7], m24, td_mad(v[6], m16, hi));
                    const u64 x = (u64)sl[c + j] + (unsigned)lo;
                    sl[c + j] = (unsigned)x;
                    sh[c + j] += hi + (i64)(x >> 32);
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) td_arrive(drained);
            if (code > 1) emit(code);
            return true;
        };
        auto matrix = [&](const TdIt &J, int &sm, int &sk) {
            const bool far = MODE == TD_ROWS && J.q >= J.q1;
            sm = MODE == TD_ROWS ? (far ? P.F.wp : J.W) : 1;
            sk = MODE == TD_ROWS ? 1 : (MODE == TD_COUPLE ? P.F.kp : P.F.wp);
            if (MODE == TD_COUPLE) return P.F.S + J.off * (k * sk);   // off: the block
            return (MODE == TD_PROJ || far ? P.F.U : P.R.D) + J.off;
        };
        // copies the entries of the next step to the lane's place, and puts its code to hist
        int2 *const raw = (int2 *)(td_sm + TD_NST * STAGE) + warp * 128 + lane;
        const int2 *p = nullptr;
        int left = 0, steps = 0, np = 0, end = 0, pulled = 0;   // of the piece: rows and steps that are left
        int shift = 0;   // of the piece's entries, to the scale of the sum
        unsigned hist = 0;
        auto pull = [&]() {
            if (steps == 0) {
                if (!have) {
                    hist <<= 2;
                    asm volatile("cp.async.commit_group;" ::: "memory");
                    return false;
                }
                int sm, sk;
                p = matrix(I, sm, sk);   // sets the strides
                p += mrow * sm + tt * sk;
                left = I.off >= 0 && mrow < I.nrow ? I.n - tt : 0;
                if (MODE == TD_COUPLE) shift = left > 0 ? P.sh[((size_t)tile * P.F.nfar + I.off) * k + mrow] : 0;
                if (MODE == TD_ROWS) shift = half ? I.sh.y : I.sh.x;
                np = I.n;
                steps = (np + 15) >> 4;
                end = I.q + 1 == I.q1 ? 2 : (I.q + 1 == I.q2 ? 3 : 0);
                have = next(I);   // I: the piece after this one
            }
            const int sk = MODE == TD_ROWS ? 1 : (MODE == TD_COUPLE ? P.F.kp : P.F.wp);
#pragma unroll
            for (int j = 0; j < 4; ++j)   // zeros outside (nothing is read)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(
                                 td_sa(raw + (pulled % TD_AHEAD) * (TD_RAW / 8) + 32 * j)),
                             "l"(j < left ? p + j * sk : (const int2 *)P.F.U), "r"(j < left ? 8 : 0)
                             : "memory");
            asm volatile("cp.async.commit_group;" ::: "memory");
            p += 16 * sk;
            left -= 16;
            ++pulled;
            --steps;
            hist = hist << 2 | (unsigned)code_of(end, steps == 0);
            if (have && steps + 2 == (np + 15) >> 4) {
                // in the piece's second step (its record has come): the warp's entries of the next piece to L2
                int sm, sq;
                const int2 *A = matrix(I, sm, sq);
                const int m = (warp & 7) * 8;
                if (MODE == TD_ROWS) {   // 8 rows of 64 entries
                    if (I.off >= 0 && m + (lane >> 2) < I.nrow && 16 * (lane & 3) < I.n)
                        asm volatile("prefetch.global.L2 [%0];\n" ::"l"(A + ((m + (lane >> 2)) * sm + 16 * (lane & 3))));
                } else {                 // 8 entries of 64 rows
#pragma unroll
                    for (int h = 0; h < 64; h += 32)
                        if (I.off >= 0 && m < I.nrow && h + lane < I.n)
                            asm volatile("prefetch.global.L2 [%0];\n" ::"l"(A + (m + (h + lane) * sq)));
                }
            }
            return true;
        };
        static_assert(TD_AHEAD == 2, "v0, v1");
        bool v0 = pull();
        int s0 = shift;
        bool v1 = pull();
        int s1 = shift;
        int cut = 0;   // steps cut
#pragma unroll 1
        for (int t = 0; v0 || t < cut + TD_LAG; ++t) {
            const bool now = v0;
            unsigned wl[4], wh[4];   // low and high words of the digits plus 128
            asm volatile("cp.async.wait_group %0;" ::"n"(TD_AHEAD - 1) : "memory");
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int2 a = raw[(t % TD_AHEAD) * (TD_RAW / 8) + 32 * j];
                u64 v = ((u64)(unsigned)a.y << 32) + (u64)((i64)a.x << 2);
                if (MODE == TD_COUPLE || (MODE == TD_ROWS && s0)) v = (u64)(((i64)v + ((1LL << s0) >> 1)) >> s0);
                v += 0x8080808080808080ULL;
                wl[j] = (unsigned)v;
                wh[j] = (unsigned)(v >> 32);
            }
            v0 = v1;
            s0 = s1;
            v1 = pull();
            s1 = shift;
            if (now) {
                const int st = t % TD_NST;
                if (t >= TD_NST && !td_wait(empty(st), (t / TD_NST - 1) & 1, deadline)) {
                    ok = false;
                    break;
                }
                unsigned char *sa = td_sm + st * STAGE + warp * 256 + lane * 8;
#pragma unroll
                for (int i = 0; i < TD_D; i += 2) {
                    const unsigned *w = i < 4 ? wl : wh;
                    unsigned d[2][2];   // [digit i, i + 1][pair of entries]
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        // digits i (bytes 0, 1) and i + 1 (bytes 2, 3) of two entries
                        const unsigned b = __byte_perm(w[2 * j], w[2 * j + 1], i & 2 ? 0x7362 : 0x5140);
                        // 0x64dd is 1024 + dd in FP16; less 1152
                        const unsigned h0 = __byte_perm(b, 0x64646464u, 0x4140), h1 = __byte_perm(b, 0x64646464u, 0x4342);
                        const half2 off2 = __half2half2(__ushort_as_half(0x6480));
                        const half2 d0 = __hsub2(*(const half2 *)&h0, off2), d1 = __hsub2(*(const half2 *)&h1, off2);
                        d[0][j] = *(const unsigned *)&d0;
                        d[1][j] = *(const unsigned *)&d1;
                    }
                    *(uint2 *)(sa + i * 4096) = make_uint2(d[0][0], d[0][1]);
                    *(uint2 *)(sa + i * 4096 + 4096) = make_uint2(d[1][0], d[1][1]);
                }
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
                __syncwarp();
                if (lane == 0) td_arrive(fullA(st));
                ++cut;
            }
            const int c = (hist >> (2 * (TD_AHEAD + TD_LAG))) & 3;   // of step t - LAG
            if (c && !move(c)) {
                ok = false;
                break;
            }
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
    } else if (lane == 0) {
        bool first = true;
        while (have && ok) {
            TdIt J = I;   // its record comes while this piece is worked on
            const bool more = next(J);
            const int ns = (I.n + 15) >> 4, end = I.q + 1 == I.q1 ? 2 : (I.q + 1 == I.q2 ? 3 : 0);
            const bool leaf = MODE == TD_PROJ || (MODE == TD_ROWS && I.q < I.q1);
            const unsigned char *src = leaf ? P.dx + ((size_t)tile * P.F.nleaf + I.col) * P.nsl * td_step(NC)
                                            : P.dh + ((size_t)tile * P.nnodes + I.col) * P.nsn * td_step(NC);
            for (int s = 0; s < ns && ok; ++s) {
                const int st = issued % TD_NST;
                const unsigned par = (issued / TD_NST) & 1;
                if (warp == TD_CW) {
                    // ---- products
                    if (!td_wait(fullA(st), par, deadline) || !td_wait(fullB(st), par, deadline)) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                    const unsigned sa = base + st * STAGE, sb = sa + TD_A;
#pragma unroll
                    for (int i = TD_D - 1; i >= 0; --i) {
                        // accumulators 0 .. i, in instructions of at most 256 columns; i = 7 first: it clears all
                        constexpr int GM = 256 / NC < 8 ? 256 / NC : 8;
#pragma unroll
                        for (int g0 = 0; g0 <= i; g0 += GM) {
                            const int ng = i + 1 - g0 < GM ? i + 1 - g0 : GM;
                            td_mma(taddr + g0 * NC, sa + i * 4096, sb + (7 - i + g0) * (NC * 32), ng * NC, !(first && i == 7));
                        }
                    }
                    td_commit(empty(st));
                    ++issued;
                    first = false;
                    if (code_of(end, s + 1 == ns)) {
                        td_commit(moved);
                        ok = td_wait(drained, moves & 1, deadline);
                        ++moves;
                        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                        first = true;
                    }
                } else {
                    // ---- the vector's digits
                    if (issued >= TD_NST && !td_wait(empty(st), par ^ 1, deadline)) {
                        ok = false;
                        break;
                    }
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(fullB(st)), "r"(td_step(NC))
                                 : "memory");
                    asm volatile(
                        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                            base + st * STAGE + TD_A),
                        "l"(src + (size_t)s * td_step(NC)), "r"(td_step(NC)), "r"(fullB(st))
                        : "memory");
                    ++issued;
                }
            }
            I = J;
            have = more;
        }
    }
    if (!ok) *abort_f = 1;
    __syncwarp();
    __syncthreads();
    if (*abort_f) {
        // wait for what is in flight: the copies, then the products and the arrival after them
        const u64 dl = td_timer() + TD_WAIT;
        if (warp >= TD_CW && lane == 0)
            for (int i = max(0, issued - TD_NST); i < issued; ++i)
                td_wait(warp == TD_CW ? empty(i % TD_NST) : fullB(i % TD_NST), (i / TD_NST) & 1, dl);
        if (warp == TD_CW && lane == 0 && moves) td_wait(moved, (moves - 1) & 1, dl);
        if (threadIdx.x == 0) atomicOr(P.err, 1);
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == TD_CW)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(taddr), "n"(TD_G * NC));
}

// ---------------------------------------------------------------------------
// What the digits cannot hold.  A piece of the vector has one scale for a tile's columns and a
// row of the operator one for a piece (xhat) or a section (near rows), so a sum's error is
// about sqrt(products) 2^-62 of the largest product of scales, whatever the sum's own terms
// are.  Before the sums are used, each is compared with a lower bound of its sum of absolute
// values; where the error could be above 2^-54 (near; 2^-53 far, a part of the row) of it,
// FP64 products or the kernels of apply_fixed.cu, whose scales are of a column's leaf or
// node, do that sum.
// ---------------------------------------------------------------------------
constexpr int TDC_CH = 512;   // columns of a panel in shared memory at a time

// |v| 2^(1022 - key) for v below 2^(key - 1022), cut to 20 bits and to zero below 2^-126: the
// conversion without FP64 instructions, and a lower bound
__device__ __forceinline__ float td_float(double v, int key)
{
    return __int_as_float(max((__double2hiint(v) & 0x7fffffff) - ((key - 126) << 20), 0) << 3);
}

// Y = (B + M and the panel entries at its positions) X in FP64, a thread per row and 4 columns;
// rows for which 2^-54 of the absolute values of these terms, its largest, is below the
// digits' error for its others are marked (rowmask, 64 bits a leaf and tile) for k_td_near.
// least: the smallest such sum of the rows, its log2 in units of 2^-8 (a lower bound).
// grid (leaf, group of 8 columns).
__global__ void __launch_bounds__(128)
k_td_csr(FaNear R, int nleaf, int nc, const int *__restrict__ nptr, const int *__restrict__ ncol,
         const double *__restrict__ X, int64_t ld, double *__restrict__ Y, const unsigned *__restrict__ kx,
         const int *__restrict__ wx, int *__restrict__ wnear, unsigned *__restrict__ rowmask, int *__restrict__ least)
{
    __shared__ unsigned nz;   // columns with x in the panel
    __shared__ int low[4][4];
    constexpr int NONE = 0x7fffffff;
    const int lf = blockIdx.x, g = blockIdx.y, r0 = R.c0 + 8 * g, b = R.kb[R.fl + lf], e = R.ke[R.fl + lf], W = R.pw[lf];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // the scale of the partners' pieces, for the tile
    const int tile = 8 * g / nc;
    int w = TD_WMIN;
    for (int q = nptr[lf] + lane; q < nptr[lf + 1]; q += 32) w = max(w, wx[tile * nleaf + ncol[q]]);
    w = __reduce_max_sync(0xffffffffu, w);
    if (threadIdx.x == 0) {
        wnear[tile * nleaf + lf] = w;
        nz = 0;
    }
    const double *x0 = X + (size_t)r0 * ld;
    const int i = b + (threadIdx.x & 63), c0 = 4 * (threadIdx.x >> 6), nr = i < e ? min(4, R.nrhs - r0 - c0) : 0;
    double v[4] = {};
    float s[4] = {};
    int t[4];
    unsigned redo = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) t[c] = NONE;
    if (nr > 0) {
        const double *x = x0 + (size_t)c0 * ld;
        int key[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) key[c] = c < nr ? (int)kx[8 * g + c0 + c] : 0;
        int ka = 1;   // the scale of the row: its largest term's
        for (int q = R.rowptr[i]; q < R.rowptr[i + 1]; ++q) ka = max(ka, (int)fa_key(R.val8[q]));
        double d = 0.0;
#pragma unroll 2
        for (int q = R.rowptr[i]; q < R.rowptr[i + 1]; ++q) {   // (16 loads of x ahead: 120 us instead of 85)
            const int j = R.colidx[q];
            const double a = R.val8[q], o = j == i ? 0.0 : a;
            const float fa = td_float(a, ka);
            if (j == i) d = a;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const double y = c < nr ? x[(size_t)c * ld + j] : 0.0;
                v[c] = fma(o, y, v[c]);
                s[c] = fmaf(fa, td_float(y, key[c]), s[c]);
            }
        }
        const float unit = sqrtf((float)W);
        const int up = R.re[i] + w - (ka - 1022) - 8;   // digits' scale over this row's, less 8 bits
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            v[c] = fma(d, c < nr ? x[(size_t)c * ld + i] : 0.0, v[c]);   // the diagonal's product, the largest, rounds the sum once
            if (key[c] && (fa_slow(key[c]) || up > 100 || !(s[c] >= scalbnf(unit, up)))) redo |= 1u << c;
            if (c < nr) t[c] = s[c] > 0.0f ? (__float_as_int(s[c]) >> 15) - (127 << 8) + ((ka + key[c] - 2 * 1022) << 8) : -NONE;
        }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        t[c] = __reduce_min_sync(0xffffffffu, t[c]);
        if (lane == c) low[warp][c] = t[c];
    }
    if (__syncthreads_or(redo != 0)) {
        // columns without any x in the panel have exact zeros
        const int *gc = R.gcol + R.goff[lf];
        unsigned m = 0;
        for (int q = threadIdx.x; q < W; q += 128) {
            const int j = gc[q];
            for (int c = 0; c < 8 && j >= 0 && r0 + c < R.nrhs; ++c) m |= x0[(size_t)c * ld + j] != 0.0 ? 1u << c : 0u;
        }
        m = __reduce_or_sync(0xffffffffu, m);
        if (lane == 0 && m) atomicOr(&nz, m);
        __syncthreads();
        const unsigned rows = __ballot_sync(0xffffffffu, redo & nz >> c0);
        if (lane == 0 && rows) atomicOr(rowmask + ((size_t)tile * nleaf + lf) * 2 + (warp & 1), rows);
    }
    if (threadIdx.x < 8) {
        const int h = threadIdx.x >> 2, c = threadIdx.x & 3;
        least[(size_t)lf * TD_COLS + 8 * g + threadIdx.x] = min(low[2 * h][c], low[2 * h + 1][c]);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
        if (c < nr) Y[(size_t)(r0 + c0 + c) * ld + i] = v[c];
}

// the marked near rows in FP64, 8 lanes a row and 16 rows at a time, and the exponents of the others'
// digit sums (marked rows: so small that the sums vanish).  grid (leaf, group of 8 columns)
constexpr int TD_NONE = -4000;
__global__ void __launch_bounds__(128)
k_td_near(FaNear R, int N, int nleaf, int nc, const double *__restrict__ X, int64_t ld, double *__restrict__ Y,
          const int *__restrict__ wnear, const unsigned *__restrict__ rowmask, short *__restrict__ er, int *__restrict__ count)
{
    extern __shared__ __align__(16) double td_xs[];   // [pair of columns][entry]
    const int lf = blockIdx.x, g = blockIdx.y, r0 = R.c0 + 8 * g, b = R.kb[R.fl + lf], e = R.ke[R.fl + lf], W = R.pw[lf];
    const int tile = 8 * g / nc, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, l8 = lane & 7;
    const unsigned bad[2] = {rowmask[((size_t)tile * nleaf + lf) * 2], rowmask[((size_t)tile * nleaf + lf) * 2 + 1]};
    if (8 * g % nc == 0 && b + (int)threadIdx.x < e) {
        const int i = b + threadIdx.x;
        er[(size_t)tile * N + i] = (short)((bad[threadIdx.x >> 5 & 1] >> lane & 1u) ? TD_NONE : R.re[i] + wnear[tile * nleaf + lf]);
    }
    if (!(bad[0] | bad[1])) return;
    if (threadIdx.x == 0) atomicAdd(count, __popc(bad[0]) + __popc(bad[1]));
    const double *x0 = X + (size_t)r0 * ld;
    const int *gc = R.gcol + R.goff[lf];
    for (int s = 0; s < 64 && b + s < e; s += 16) {
        if (!((s < 32 ? bad[0] : bad[1]) >> (s & 31) & 0xffffu)) continue;
        const int ro = s + 4 * warp + (lane >> 3), i = b + ro;
        const bool any = (s < 32 ? bad[0] : bad[1]) >> (ro & 31) & 1u;
        const double *D = R.Dd + R.poff[lf] + (size_t)ro * W;
        double a[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) a[c] = 0.0;
        for (int j0 = 0; j0 < W; j0 += TDC_CH) {
            const int n = min(TDC_CH, W - j0);
            __syncthreads();
            for (int q = threadIdx.x; q < n; q += 128) {
                const int j = gc[j0 + q];
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    td_xs[(c >> 1) * 2 * TDC_CH + 2 * q + (c & 1)] = j >= 0 && r0 + c < R.nrhs ? x0[(size_t)c * ld + j] : 0.0;
            }
            __syncthreads();
            if (any)
                for (int j = l8; j < n; j += 8) {
                    const double d = D[j0 + j];
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        const double2 x = *(const double2 *)(td_xs + p * 2 * TDC_CH + 2 * j);
                        a[2 * p] = fma(d, x.x, a[2 * p]);
                        a[2 * p + 1] = fma(d, x.y, a[2 * p + 1]);
                    }
                }
        }
        if (any)
            for (int q = R.rowptr[i] + l8; q < R.rowptr[i + 1]; q += 8) {
                const double d = R.val[q], *x = x0 + R.colidx[q];
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    if (r0 + c < R.nrhs) a[c] = fma(d, x[(size_t)c * ld], a[c]);
            }
        const int c = fa_sum8d<8>(a, l8);
        if (any && r0 + c < R.nrhs) Y[(size_t)(r0 + c) * ld + i] = a[0];
    }
}

// shifts of the rows' records to the scales of their sums; a warp per item.  grid (items, tile)
__global__ void __launch_bounds__(32)
k_td_shift(const int4 *__restrict__ items, const TdRec *__restrict__ rec, int nrec, int nleaf, int nnodes,
           const int *__restrict__ wx, const int *__restrict__ wh, const int *__restrict__ wnear, const int *__restrict__ wfar,
           uchar2 *__restrict__ shr)
{
    const int4 v = items[blockIdx.x];
    const int tile = blockIdx.y, l0 = 2 * v.w, l1 = min(l0 + 1, nleaf - 1);
    for (int q = v.x + (int)threadIdx.x; q < v.z; q += 32) {
        const bool near = q < v.y;
        const int w = near ? wx[tile * nleaf + rec[q].col] : wh[tile * nnodes + rec[q].col], *to = near ? wnear : wfar;
        const int a = to[tile * nleaf + l0] - w, c = to[tile * nleaf + l1] - w;   // (negative where the half has no such partner)
        shr[(size_t)tile * nrec + q] = make_uchar2(min(max(a, 0), 63), min(max(c, 0), 63));
    }
}

// bits of the groups of 8 columns in which a thread of the first 64 says yes
__device__ __forceinline__ unsigned td_groups(bool yes, unsigned *sh)
{
    const unsigned b = __ballot_sync(0xffffffffu, yes);
    if ((threadIdx.x & 31) == 0) {
        unsigned m = 0;
        for (int g = 0; g < 4; ++g) m |= (b >> (8 * g) & 255u) ? 1u << g : 0u;
        sh[threadIdx.x >> 5] = m;
    }
    __syncthreads();
    return sh[0] | sh[1] << 4;
}

// leaves whose projections are redone: their x is small in its column (n1: sum of a leaf's |x| in
// units of the column's scale).  A projection's error goes to k entries of xhat and from there
// through a block's entries, which differ by a few bits.
__global__ void __launch_bounds__(64)
k_td_check_x(int k, int nrow, int cols, const unsigned *__restrict__ kx, const float *__restrict__ n1,
             const float *__restrict__ umin, unsigned *mask, int *count)
{
    __shared__ unsigned sh[2];
    const int lf = blockIdx.x, c = threadIdx.x;
    const float n = c < cols ? n1[(size_t)lf * TD_COLS + c] : 0.0f;
    const bool redo = c < cols && (fa_slow(kx[c]) || (n > 0.0f && !(256.0f * umin[lf] * n >= 2.0f * sqrtf((float)nrow * k))));
    const unsigned m = td_groups(redo, sh);
    if (c == 0) {
        mask[lf] = m;
        if (m) atomicAdd(count, __popc(m));
    }
}

// exponents of a node's rows (the largest product of a block row's and its partner's scales) and
// the shifts of the blocks' rows to them.  grid (node, tile)
__global__ void __launch_bounds__(128)
k_td_align(FaFar P, int node0, int nnodes, const int *__restrict__ wh, short *__restrict__ ec, unsigned char *__restrict__ sh)
{
    __shared__ int top[KMAX];
    const int t = node0 + blockIdx.x, tile = blockIdx.y, k = P.k, e0 = P.fptr[t], e1 = P.fptr[t + 1];
    wh += (size_t)tile * nnodes - node0;
    sh += (size_t)tile * P.nfar * k;
    if ((int)threadIdx.x < k) {
        int m = -900;   // (below it: rows of zeros)
#pragma unroll 4
        for (int e = e0; e < e1; ++e) m = max(m, P.se[(size_t)e * k + threadIdx.x] + wh[P.fcol[e]]);
        top[threadIdx.x] = m;
        ec[((size_t)tile * nnodes + blockIdx.x) * k + threadIdx.x] = (short)m;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < (e1 - e0) * k; i += 128) {
        const int e = e0 + i / k, a = i % k;
        sh[(size_t)e0 * k + i] = (unsigned char)min(top[a] - max(P.se[(size_t)e0 * k + i] + wh[P.fcol[e]], -900), 63);
    }
}

// nodes whose sum over their blocks is redone, and a lower bound of sum |S||xhat| of a node's rows.
// CTA per node, 64 columns x 4 groups of rows: low 2^-shift |xhat| of a row and block is at most
// its sum of absolute values
__global__ void __launch_bounds__(256)
k_td_check_couple(FaFar P, int node0, int nnodes, int cols, int nc, const unsigned *__restrict__ kh, const int *__restrict__ wh,
                  const float *__restrict__ n1, const double *__restrict__ least, const float *__restrict__ low,
                  const unsigned char *__restrict__ shift, double *__restrict__ sum, unsigned *mask, int *count, const int *err)
{
    constexpr int CH = 8;   // blocks at a time
    __shared__ float rows[4][TD_COLS], u[CH][KMAX];
    const int t = node0 + blockIdx.x, c = threadIdx.x & 63, g = threadIdx.x >> 6, l = 31 - __clz(t + 1), k = P.k;
    const int e0 = P.fptr[t], e1 = P.fptr[t + 1], tile = c < cols ? c / nc : 0;
    const unsigned key = kh[(l - P.lmin) * TD_COLS + c];
    float r = INFINITY;
    for (int tl = 0; tl < (cols + nc - 1) / nc; ++tl) {
        float v[KMAX / 4];
#pragma unroll
        for (int q = 0; q < KMAX / 4; ++q) v[q] = 0.0f;
        for (int b = e0; b < e1; b += CH) {
            __syncthreads();
            for (int i = threadIdx.x; i < min(CH, e1 - b) * k; i += 256) {
                const size_t j = (size_t)b * k + i;
                u[i / k][i % k] = low[j] * __uint_as_float((127u - shift[(size_t)tl * P.nfar * k + j]) << 23);
            }
            __syncthreads();
            if (tl != tile) continue;
#pragma unroll 4
            for (int e = b; e < min(b + CH, e1); ++e) {
                const float x = n1[(size_t)(P.fcol[e] - node0) * TD_COLS + c];
#pragma unroll
                for (int q = 0; q < KMAX / 4; ++q)
                    if (g + 4 * q < k) v[q] = fmaf(u[e - b][g + 4 * q], x, v[q]);
            }
        }
        if (tl == tile)
#pragma unroll
            for (int q = 0; q < KMAX / 4; ++q)
                if (g + 4 * q < k) r = fminf(r, v[q]);
    }
    rows[g][c] = r;
    __syncthreads();
    if (g) return;
    r = fminf(fminf(rows[0][c], rows[1][c]), fminf(rows[2][c], rows[3][c]));
    double s = 0.0;
    float n = 0.0f;
    for (int e = e0; e < e1; ++e) {
        const int f = P.fcol[e] - node0;
        const float x = c < cols ? n1[(size_t)f * TD_COLS + c] : 0.0f;
        n += x;
        s = fma(least[e], scalbn((double)x, wh[(size_t)tile * nnodes + f]), s);
    }
    const bool redo = c < cols && e1 > e0 &&
                      (*err || fa_slow(key) || (n > 0.0f && !(512.0f * r >= sqrtf((float)(e1 - e0) * k))));
    const unsigned b = __ballot_sync(0xffffffffu, redo);
    if ((c & 31) == 0) {
        unsigned m = 0;
        for (int q = 0; q < 4; ++q) m |= (b >> (8 * q) & 255u) ? 1u << (4 * (c >> 5) + q) : 0u;
        if (m) {
            atomicOr(mask + t, m);
            atomicAdd(count, __popc(m));
        }
    }
    sum[(size_t)blockIdx.x * TD_COLS + c] = n > 0.0f ? fmax(scalbn(s, (int)key - 1022), 1e-300) : 0.0;
}

// yhat of the nodes that are redone: the sum over their blocks
__global__ void __launch_bounds__(256)
k_td_couple_sum(FaFar P, int node0, int c0, const double *__restrict__ ye, double *__restrict__ yhat, FaWhen when)
{
    if (fa_none(when)) return;
    const int k = P.k, r = c0 + blockIdx.y;
    for (int t = node0 * k + blockIdx.x * 256 + threadIdx.x; t < P.nnode * k; t += gridDim.x * 256) {
        const int node = t / k, a = t - node * k;
        if (fa_off(when, node, r)) continue;
        double s = 0.0;
        for (int e = P.fptr[node]; e < P.fptr[node + 1]; ++e) s += ye[((size_t)r * P.nfar + e) * k + a];
        yhat[(size_t)r * P.nnode * k + t] = s;
    }
}

// leaves whose expansion is redone: the bound of a row's far sum (sum, umin) and of its near terms
// (least, the smallest of the leaf's rows) against the digits' error; wfar: the scale of the
// ancestors' pieces
__global__ void __launch_bounds__(64)
k_td_check_expand(FaFar P, int node0, int nnodes, int cols, int nc, const unsigned *__restrict__ ky,
                  const int *__restrict__ wh, int *__restrict__ wfar, short *__restrict__ ef, const double *__restrict__ sum,
                  const float *__restrict__ umin, const int *__restrict__ least, unsigned *mask, int *count, const int *err)
{
    __shared__ unsigned sh[2];
    const int lf = blockIdx.x, c = threadIdx.x, tile = c < cols ? c / nc : 0;
    double s = 0.0;
    int w = TD_WMIN;
    for (int lv = 0; lv < P.nlev; ++lv) {
        const int f = ((P.fl + lf + 1) >> (P.nlev - 1 - lv)) - 1 - node0;
        s += sum[(size_t)f * TD_COLS + c];
        w = max(w, wh[(size_t)tile * nnodes + f]);
    }
    const unsigned key = ky[c];
    const double have = 512.0 * umin[lf] * s + scalbn(1.0, max((least[(size_t)lf * TD_COLS + c] >> 8) + 8 - P.ue[lf], -2000));
    const bool redo = c < cols && (*err || fa_slow(key) ||
                                   (key && s > 0.0 && !(have >= scalbn((double)sqrtf((float)(P.nlev * P.k)), (int)key + w - 1022))));
    unsigned m = td_groups(redo, sh);
    // all groups of a tile together: its sums are left out (an exponent so small that they vanish)
    const unsigned tm = nc == 64 ? 255u : (1u << (nc >> 3)) - 1u;
    unsigned all = 0;
    for (int q = 0; q < 8; q += nc >> 3)
        if (m >> q & tm) all |= tm << q;
    m = all & ((1u << ((cols + 7) >> 3)) - 1u);
    if (c < cols && c % nc == 0) {
        wfar[tile * P.nleaf + lf] = w;
        ef[tile * P.nleaf + lf] = (short)(all >> (c >> 3) & 1u ? TD_NONE : P.ue[lf] + w);
    }
    if (c == 0) {
        mask[lf] = m;
        if (m) atomicAdd(count, __popc(m));
    }
}

template <int NC, int MODE>
void launch_td(const TdP &P, int nitem, int nt, const double *X, int64_t ld, double *out, cudaStream_t st)
{
    constexpr int shm = TD_NST * (TD_A + td_step(NC)) + TD_AHEAD * TD_RAW + (3 * TD_NST + 2) * 8 + 8 + 2 * NC * 4;
    VFD_CUDA(cudaFuncSetAttribute(k_td<NC, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, shm));
    k_td<NC, MODE><<<dim3(std::min(nitem, TD_SMS), nt), TD_THREADS, shm, st>>>(P, nitem, X, ld, out);
    VFD_CUDA(cudaGetLastError());
}
template <int MODE>
void launch_td(int nc, const TdP &P, int nitem, int nt, const double *X, int64_t ld, double *out, cudaStream_t st)
{
    if (nc == 16) launch_td<16, MODE>(P, nitem, nt, X, ld, out, st);
    else if (nc == 32) launch_td<32, MODE>(P, nitem, nt, X, ld, out, st);
    else launch_td<64, MODE>(P, nitem, nt, X, ld, out, st);
}

}  // namespace

// Records of k_td, geometry only (end of the mesh setup).  A record: partner (leaf, or node
// less the first far node), its rows (> 0), offsets of the two halves' entries (-1: none).
// td_rows: pairs of leaves (2 p, 2 p + 1): near partners (offsets in the panels), then the
// ancestors of the far levels (offsets in the flattened bases).
// td_couple: pairs of nodes from the first far node on (offsets: the coupling blocks).
// Items (first record, second section, end, pair) in the order of the CTAs that take them.
static void build_lists(MeshData &m)
{
    if (m.max_leaf_size > 64 || !m.nnear || (m.nfar > 0 && m.far_lmin < 1)) return;   // (pairs of nodes share a level)
    const int nleaf = m.kt.nleaf, fl = m.kt.first_leaf(), nlev = m.nfar > 0 ? m.kt.L - m.far_lmin + 1 : 0;
    const int k = m.k, wp = (nlev * k + 1) & ~1, node0 = nlev ? (1 << m.far_lmin) - 1 : 0;
    std::vector<TdRec> rec;
    std::vector<int4> items;
    auto add = [&](int col, int n, int64_t a, int64_t b) { if (n > 0) rec.push_back({col, n, {a, b}}); };
    // merge of two sorted lists [a0, a1) and [b0, b1) of partners
    auto merge = [&](const std::vector<int> &list, int a0, int a1, int b0, int b1, auto f) {
        while (a0 < a1 || b0 < b1) {
            const int c = std::min(a0 < a1 ? list[a0] : list[b0], b0 < b1 ? list[b0] : list[a0]);
            const int ea = a0 < a1 && list[a0] == c ? a0++ : -1, eb = b0 < b1 && list[b0] == c ? b0++ : -1;
            f(c, ea, eb);
        }
    };
    // the largest items first, each to the CTA with the fewest steps so far
    auto upload = [&](DBuf<TdRec> &dr, DBuf<int4> &di, DBuf<int> &db) {
        const int n = (int)items.size(), nb = std::min(n, TD_SMS);
        std::vector<int64_t> steps(n, 2), load(nb, 0);   // and 2 for an item's end
        std::vector<int> ord(n), bin(1, 0);
        std::vector<std::vector<int>> of(nb);
        for (int i = 0; i < n; ++i) {
            ord[i] = i;
            for (int q = items[i].x; q < items[i].z; ++q) steps[i] += (rec[q].n + 15) >> 4;
        }
        std::stable_sort(ord.begin(), ord.end(), [&](int a, int b) { return steps[a] > steps[b]; });
        for (int i : ord) {
            const int b = (int)(std::min_element(load.begin(), load.end()) - load.begin());
            load[b] += steps[i];
            of[b].push_back(i);
        }
        std::vector<int4> out;
        for (auto &l : of) {
            for (int i : l) out.push_back(items[i]);
            bin.push_back((int)out.size());
        }
        dr.upload(rec);
        di.upload(out);
        db.upload(bin);
        rec.clear();
        items.clear();
    };
    for (int a = 0; a < nleaf; a += 2) {
        const int b = a + 1 < nleaf ? a + 1 : -1, q0 = (int)rec.size();
        merge(m.near_col_h, m.near_ptr_h[a], m.near_ptr_h[a + 1], b < 0 ? 0 : m.near_ptr_h[b], b < 0 ? 0 : m.near_ptr_h[b + 1],
              [&](int c, int ea, int eb) {
                  add(c, m.kt.end[fl + c] - m.kt.begin[fl + c], ea < 0 ? -1 : m.near_off_h[ea], eb < 0 ? -1 : m.near_off_h[eb]);
              });
        const int q1 = (int)rec.size();
        for (int lv = 0; lv < nlev; ++lv) {
            const int na = ((fl + a + 1) >> (nlev - 1 - lv)) - 1, nb = b < 0 ? -1 : ((fl + b + 1) >> (nlev - 1 - lv)) - 1;
            const int64_t oa = (int64_t)m.kt.begin[fl + a] * wp + lv * k;
            const int64_t ob = b < 0 ? -1 : (int64_t)m.kt.begin[fl + b] * wp + lv * k;
            if (na == nb || b < 0) {
                add(na - node0, k, oa, ob);
            } else {
                add(na - node0, k, oa, -1);
                add(nb - node0, k, -1, ob);
            }
        }
        if (q0 < (int)rec.size()) items.push_back({q0, q1, (int)rec.size(), a / 2});
    }
    upload(m.td_rows, m.td_rows_item, m.td_rows_bin);
    if (!nlev) return;
    for (int a = node0; a < m.kt.nnode; a += 2) {
        const bool two = a + 1 < m.kt.nnode;
        const int q0 = (int)rec.size();
        merge(m.far_col_h, m.far_ptr_h[a], m.far_ptr_h[a + 1], two ? m.far_ptr_h[a + 1] : 0, two ? m.far_ptr_h[a + 2] : 0,
              [&](int c, int ea, int eb) { add(c - node0, k, ea, eb); });
        if (q0 == (int)rec.size()) add(0, k, -1, -1);   // no blocks: zeros
        items.push_back({q0, (int)rec.size(), (int)rec.size(), (a - node0) / 2});
    }
    upload(m.td_couple, m.td_couple_item, m.td_couple_bin);
}
void build_tensor_lists(MeshData &m)
{
    if (!if_memory([&] { build_lists(m); })) m.td_rows.release();   // (no digits then)
}

// Where the digits pay.  The kernels of few columns take groups of 8, the digits up to 64 columns
// a pass, and a pass costs 240 to 700 us however few they are, so the columns of one pass count
// (817 DoFs, 256 columns in 4 passes: 369 us in groups of 8, 966 with digits).  Measured,
// 10^6 entries x groups of a pass: groups / digits in us: 9 (9025 DoFs, rank 16, 8 columns)
// 186 / 284, 18 (16) 288 / 294, 27 (24) 566 / 337; 19 (10267 DoFs, rank 36, 8) 282 / 399, 38
// (12) 580 / 408; 18 (3997 DoFs, rank 64, 16) 222 / 364, 28 (24) 367 / 386, 37 (32) 411 / 386;
// 24 (16129 DoFs, rank 16, 5) 338 / 312; 97 (27361 DoFs, rank 64, 5) 719 / 718, (8) 896 / 724.
// Up to 4 columns go as one narrow group (97: 437 / 712).
bool apply_tensor_fits(const MeshData &m, const OpData &op, int nrhs)
{
    if (!m.td_rows.n || op.td_off) return false;
    if (op.td_min > 0) return nrhs >= op.td_min;
    const int nlev = m.nfar > 0 ? m.kt.L - m.far_lmin + 1 : 0;
    const double entries = (double)m.near_entries + (double)m.nfar * m.k * m.k + 2.0 * nlev * m.k * m.N;
    return nrhs >= 5 && entries * cdiv(std::min(nrhs, TD_COLS), 8) >= 2.2e7;
}

// Columns of a tile: the time of a wave of CTAs is 1, 1.07 and 1.6 for 16, 32 and 64
// columns (27361 DoFs: 625, 685 and 996 us for 16 columns; 817 DoFs: 171, 183, 255)
static int td_tile(const MeshData &m, int cols)
{
    const double cost[3] = {1.0, 1.07, 1.6};
    int best = 0;
    double tb = 0;
    for (int i = 0; i < 3; ++i) {
        const double t = cost[i] * std::max(1.0, (double)m.td_rows_item.n * cdiv(cols, 16 << i) / TD_SMS);
        if (i == 0 || t < tb) {
            best = i;
            tb = t;
        }
    }
    return 16 << best;
}

namespace {
constexpr int TD_TILES = TD_COLS / 16;   // tiles of a pass at most
// td_key: keys of x, of yhat, of xhat per level, of the pieces; td_mask: a zero, the nodes, the leaves (projections, expansion)
constexpr int TK_X = 0, TK_Y = TD_COLS, TK_H = 2 * TD_COLS, TK_N = TK_H + 32 * TD_COLS;
// td_flag: an expired wait; what was redone: near rows, projections, nodes, leaves (in groups of 8 columns)
enum { TF_ERR, TF_ROWS, TF_PROJ, TF_NODES, TF_LEAVES, TF_N };
}  // namespace

// workspace: the digits of 64 columns per leaf and per node, column keys, masks and flags
void apply_tensor_alloc(const MeshData &m, OpData &op)
{
    if (op.td_mem.p) return;
    const int node0 = m.nfar > 0 ? (1 << m.far_lmin) - 1 : m.kt.nnode;
    const size_t nodes = m.kt.nnode - node0, leaves = m.kt.nleaf;
    size_t total = 0;
    auto part = [&](auto &v, size_t n) {   // sizes, then (with the memory) places
        v.n = n;
        if (op.td_mem.p) v.p = (decltype(v.p))(op.td_mem.p + total);
        total += (v.bytes() + 1023) & ~(size_t)1023;
    };
    auto parts = [&] {
        total = 0;
        part(op.td_x, leaves * ((m.max_leaf_size + 15) >> 4) * td_step(TD_COLS));
        part(op.td_h, nodes * ((m.k + 15) >> 4) * td_step(TD_COLS));
        part(op.td_key, TK_N + std::max(leaves, nodes) * TD_COLS);
        part(op.td_w, TD_TILES * (3 * leaves + nodes));
        part(op.td_exp, TD_TILES * (nodes * m.k + m.N + leaves));
        part(op.td_shift, (size_t)TD_TILES * (2 * m.td_rows.n + (size_t)m.nfar * m.k));
        part(op.td_mask, 1 + m.kt.nnode + (2 + 2 * TD_TILES) * leaves);
        part(op.td_n1, (nodes + leaves) * TD_COLS);
        part(op.td_sum, nodes * TD_COLS);
        part(op.td_least, leaves * TD_COLS);
        part(op.td_flag, TF_N);
    };
    parts();
    op.td_off = !if_memory([&] { op.td_mem.alloc(total); });   // the kernels of few columns do without
    if (!op.td_off) parts();
}

// Y = A X for all columns
void apply_tensor(const MeshData &m, OpData &op, const double *X, double *Y, int nrhs, int64_t ld, cudaStream_t st)
{
    op.td_cols = nrhs;
    const bool far = m.nfar > 0;
    const int k = m.k, nleaf = m.kt.nleaf, node0 = far ? (1 << m.far_lmin) - 1 : m.kt.nnode, nnodes = m.kt.nnode - node0;
    TdP P{};
    P.F = fa_far_view(m, op);
    P.R = fa_near_view(m, op);
    P.nrhs = P.R.nrhs = nrhs;
    P.nsl = (m.max_leaf_size + 15) >> 4;
    P.nsn = (k + 15) >> 4;
    P.node0 = node0;
    P.nnodes = nnodes;
    int *flag = op.td_flag.p, *err = flag + TF_ERR;
    unsigned *key = op.td_key.p, *zero = op.td_mask.p, *nodemask = zero + 1, *leafmask = nodemask + m.kt.nnode, *projmask = leafmask + nleaf, *rowmask = projmask + nleaf;
    int *wx = op.td_w.p, *wnear = wx + TD_TILES * nleaf, *wfar = wnear + TD_TILES * nleaf, *wh = wfar + TD_TILES * nleaf;
    float *n1x = op.td_n1.p, *n1h = n1x + (size_t)nleaf * TD_COLS;
    int *least = op.td_least.p;
    double *sum = op.td_sum.p;
    VFD_CUDA(cudaMemsetAsync(flag, 0, op.td_flag.bytes(), st));
    P.err = err;
    P.wait = (long long)(op.td_wait * TD_HZ);
    P.dx = op.td_x.p;
    P.dh = op.td_h.p;
    P.kx = key + TK_X;
    short *er = op.td_exp.p, *ef = er + (size_t)TD_TILES * m.N, *ec = ef + (size_t)TD_TILES * nleaf;
    uchar2 *shr = (uchar2 *)op.td_shift.p;
    unsigned char *shc = op.td_shift.p + (size_t)TD_TILES * 2 * m.td_rows.n;
    P.wx = wx;
    P.er = er;
    P.ef = ef;
    P.ec = ec;
    P.shr = shr;
    P.nrec = (int)m.td_rows.n;
    P.sh = shc;
    const size_t hs = (size_t)m.kt.nnode * k;
    for (int c0 = 0; c0 < nrhs; c0 += TD_COLS) {
        const int cols = std::min(TD_COLS, nrhs - c0), ng = cdiv(cols, 8);
        const int nc = td_tile(m, cols), nt = cdiv(cols, nc);
        auto digits = [&](const double *v, size_t vld, size_t base, bool leaves, int nlev, unsigned *keys) {
            TdVec V{};
            V.v = v;
            V.ld = vld;
            V.base = base;
            V.npiece = leaves ? nleaf : nnodes;
            V.ns = leaves ? P.nsl : P.nsn;
            V.len = k;
            V.kb = leaves ? P.F.kb + P.F.fl : nullptr;
            V.ke = leaves ? P.F.ke + P.F.fl : nullptr;
            V.nrhs = nrhs;
            V.c0 = c0;
            V.nc = nc;
            V.node0 = node0;
            V.lmin = m.far_lmin;
            V.nlev = nlev;
            V.key = keys;
            V.piece = key + TK_N;
            V.w = leaves ? wx : wh;
            V.out = leaves ? op.td_x.p : op.td_h.p;
            V.n1 = leaves ? n1x : n1h;
            k_td_max<<<V.npiece, 256, 0, st>>>(V);
            k_td_digits<<<dim3(V.npiece, nt), 256, 0, st>>>(V);
            VFD_CUDA(cudaGetLastError());
        };
        auto when = [&](const unsigned *mask, int any) {
            FaWhen w;
            w.mask = mask;
            w.any = flag + any;
            w.err = err;
            w.c0 = c0;
            return w;
        };
        auto redo = [&](FaStep step, const FaWhen &w) { apply_fixed_redo(step, m, op, X, Y, c0, ng, nrhs, ld, st, w); };
        VFD_CUDA(cudaMemsetAsync(key, 0, TK_N * sizeof(unsigned), st));
        VFD_CUDA(cudaMemsetAsync(zero, 0, op.td_mask.bytes(), st));
        P.c0 = P.R.c0 = c0;
        digits(X, ld, 0, true, 1, key + TK_X);
        k_td_csr<<<dim3(nleaf, ng), 128, 0, st>>>(P.R, nleaf, nc, m.near_ptr.p, m.near_col.p, X, ld, Y, P.kx, wx, wnear, rowmask,
                                                  least);
        k_td_near<<<dim3(nleaf, ng), 128, TDC_CH * 64, st>>>(P.R, m.N, nleaf, nc, X, ld, Y, wnear, rowmask, er, flag + TF_ROWS);
        VFD_CUDA(cudaGetLastError());
        if (far) {
            k_td_check_x<<<nleaf, 64, 0, st>>>(k, m.max_leaf_size, cols, P.kx, n1x, m.fa_umin.p, projmask, flag + TF_PROJ);
            launch_td<TD_PROJ>(nc, P, nleaf * cdiv(P.F.nlev * k, 128), nt, X, ld, op.P64.p, st);
            redo(FA_PROJ, when(projmask, TF_PROJ));
            launch_far_sum(m, op, c0, cols, st, nullptr);
            digits(op.xhat.p, hs, (size_t)node0 * k, false, P.F.nlev, key + TK_H);
            k_td_align<<<dim3(nnodes, nt), 128, 0, st>>>(P.F, node0, nnodes, wh, ec, shc);
            P.kh = key + TK_H;
            P.items = m.td_couple_item.p;
            P.bin = m.td_couple_bin.p;
            P.rec = m.td_couple.p;
            launch_td<TD_COUPLE>(nc, P, (int)m.td_couple_item.n, nt, X, ld, op.yhat.p, st);
            k_td_check_couple<<<nnodes, 256, 0, st>>>(P.F, node0, nnodes, cols, nc, P.kh, wh, n1h, op.fa_min.p, op.fa_low.p, shc,
                                                      sum, nodemask, flag + TF_NODES, err);
            const FaWhen nodes = when(nodemask, TF_NODES);
            redo(FA_COUPLE, nodes);
            k_td_couple_sum<<<dim3(std::min(cdiv(hs, 256), 32), cols), 256, 0, st>>>(P.F, node0, c0, op.ye64.p, op.yhat.p, nodes);
            digits(op.yhat.p, hs, (size_t)node0 * k, false, 1, key + TK_Y);
            P.kh = key + TK_Y;
            k_td_check_expand<<<nleaf, 64, 0, st>>>(P.F, node0, nnodes, cols, nc, key + TK_Y, wh, wfar, ef, sum, m.fa_umin.p,
                                                    least, leafmask, flag + TF_LEAVES, err);
            VFD_CUDA(cudaGetLastError());
        }
        P.items = m.td_rows_item.p;
        P.bin = m.td_rows_bin.p;
        P.rec = m.td_rows.p;
        k_td_shift<<<dim3((int)m.td_rows_item.n, nt), 32, 0, st>>>(P.items, P.rec, P.nrec, nleaf, nnodes, wx, wh, wnear, wfar, shr);
        launch_td<TD_ROWS>(nc, P, (int)m.td_rows_item.n, nt, X, ld, Y, st);
        redo(FA_NEAR, when(zero, TF_ERR));
        if (far) redo(FA_EXPAND, when(leafmask, TF_LEAVES));
    }
}

// vfd_op_apply_stats; waits for the device
void apply_tensor_stats(const OpData &op, int64_t *out, int n)
{
    int h[1 + TF_N] = {op.td_cols};
    if (op.td_cols) {
        VFD_CUDA(cudaDeviceSynchronize());
        VFD_CUDA(cudaMemcpy(h + 1, op.td_flag.p, TF_N * sizeof(int), cudaMemcpyDeviceToHost));
    }
    for (int i = 0; i < n; ++i) out[i] = i <= TF_N ? h[i] : 0;
}

}  // namespace vfd
