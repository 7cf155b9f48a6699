// FP64 matrix products on the BF16 tensor cores by exact digit slicing.
//
// The splitting is the error-free transformation of matrix products of Ozaki,
// Ogita, Oishi and Rump (Numer. Algorithms 59, 2012), here with BF16 digits and
// the FP32 accumulators of tcgen05:
//   * every row i of A (over the K range of one pass) is scaled by 2^-ea_i so that
//     its entries lie in (-1/2, 1/2), rounded to 49 fractional bits and written
//     as sum_s d_s 2^{-7(s+1)} with balanced base-128 digits |d_s| <= 64 (the
//     plain digits of the value plus a bias of 64 per position, less 64); slice
//     s holds d_s 2^{-7(s+1)}, exact in BF16.  Columns of B the same with 2^-eb_j.
//     Both operands of up to four passes are sliced in one launch.
//   * the slice products of one order o = s + t carry the unit 2^{-7(o+2)}; each
//     term is at most 2^12 units, so the FP32 accumulation of the (o+1) products
//     of order o over K terms is exact while (o+1) K 2^12 <= 2^24.  A pass covers
//     at most 1024 of K: orders 0..3 are exact (with nine digits 0..5, see OZ_OUTS_F64);
//     the orders above are rounded, with seven digits below 2^-52 of the leading term.
//   * one launch of the multi-GEMM engine computes D_o = sum_{s+t=o} A_s B_t for
//     every kept order and every pass of the group (the passes as K-aligned
//     parts stored apart; longer and shorter outputs paired on the CTAs by the
//     boustrophedon tile order); C = beta C + sum over the
//     passes of alpha 2^{ea_i + eb_j} sum_o D_o in FP64, the passes in order.
// Orders above digits - 1 are dropped: with 7 digits per operand the error per element is
// about 2^-46 K max_k|a_ik| max_k|b_kj|, the size of an FP64 product's own
// worst-case rounding error.  FP32 operands take 7 digits too: the digits cover
// a window below the row's largest entry, not each entry's own 24 bits.
// FP64 operands of the FP64 path take nine digits (63 bits below each row's
// largest entry, orders 0..8): 45 slice products instead of 28, and one for the
// entries' sizes.  Measured against
// extended precision (relative Frobenius error of a Gaussian product, K = 500 /
// 2048): 4.8e-17 / 6.7e-17, the FP64 units 3.0e-16 / 9.2e-16; with low-rank, 1 %
// sparse and graded (1e8) matrices the slices stay at 3e-17..8e-17 and the units
// at 8e-17..1.4e-15.  The digits' error scales with max|a_i.| max|b_.j|; entries whose
// sum |a_ik| |b_kj| is small beside that are formed with FP64 FMA (OZ_SMALL), so that
// each entry keeps the bound of an FP64 sum.  FP64 sketch 8000 x 4000, r = 200, us:
// Gaussian operands 2240, X and Y selecting columns and rows 4050, 2 % dense operands
// 33400 (nearly every entry); the FP64 units 40320 each.
#include "gn_internal.cuh"

#include <cooperative_groups.h>

#include <algorithm>

namespace gn {
namespace {

constexpr int OZ_KPASS = 1024;   // K per pass (exactness of the orders <= 3)
constexpr int OZ_NPANEL = 256;   // least N per GEMM launch (oz_npanel bounds the FP32 outputs)
constexpr int OZ_MAX_DIGITS = OZ_DIGITS_F64;
constexpr int OZ_PGRP = 4;       // passes per group of launches (slicing, products, combination)

// FP32 outputs of a product: one per order, and with nine digits a second one for the orders 4
// and 5.  Their 5 and 6 slice products can pass 2^24 units over 1024 of K (digits all large and
// of one sign), so they are cut after four: every output of the orders 0..5 is then exact.
// The last output is the size of each entry, sum_k |a_ik| |b_kj| from the leading digits' absolute
// values (a slice of its own): where that is small, the window below the row's and the column's
// largest entries is not enough and the entry is formed from the operands (see OZ_SMALL).
constexpr int OZ_OUTS_F64 = OZ_DIGITS_F64 + 3;
constexpr int OZ_SLICES_F64 = OZ_DIGITS_F64 + 1;
constexpr int OZ_CUT = 4;        // slice products per output of the exact orders
int oz_outputs(int digits) { return digits == OZ_DIGITS_F64 ? OZ_OUTS_F64 : digits; }
int oz_slices(int digits) { return digits == OZ_DIGITS_F64 ? OZ_SLICES_F64 : digits; }

// An entry whose size S is below this (rows and columns scaled to maxima of 1/4 .. 1/2) in a part
// is formed from the operands with FP64 FMA.  The digits' error in a part is at most K 2^-62
// there (rounding of both operands to 2^-64, the orders dropped below 2^-62), typically
// K^1/2 2^-65; the bound of an FP64 sum is K 2^-53 S.  The two meet at S = 2^-9, so that the
// digits never exceed the bound that the FP64 units keep, entry by entry.  (Leading digits round:
// S is at most twice too large where it is that small.)
constexpr float OZ_SMALL = 1.0f / 256.0f;

size_t al256(size_t b) { return (b + 255) & ~static_cast<size_t>(255); }

// Columns of C per GEMM launch: at least 256, more while the FP32 outputs of all
// orders and K parts stay within 64 MB (short, wide products in one launch); 160 MB
// with more than seven digits: their wide products (Y^T A of an FP64 sketch) then have
// enough 256-row tiles, which need 62 B per cycle and SM from L2 where 128-row ones
// need 94 of the ~60 there are.  Measured at one shape only, 20000 x 10000, r = 500: 28.4
// -> 26.3 ms with nine outputs; with twelve, panels a third wider (213 MB) cost 1.2 ms.
// Whole tiles of 256 columns there: the last tile of a panel costs as much at 64 columns
// (sketch at 32768 x 16384, r = 1000: 124 -> 109 ms).
long long oz_npanel(long long M, long long N, long long parts, int orders) {
    long long np = ((orders > 7 ? 160LL : 64LL) << 20) / (4LL * orders * std::max<long long>(M, 1) * std::max<long long>(parts, 1));
    np = std::max<long long>(np, OZ_NPANEL) / (orders > 7 ? OZ_NPANEL : 16) * (orders > 7 ? OZ_NPANEL : 16);
    return std::min<long long>(N, np);
}
long long r8(long long x) { return (x + 7) / 8 * 8; }
long long r4(long long x) { return (x + 3) / 4 * 4; }

// ---- digit extraction in integer arithmetic (the FP64 pipe is the slow one)
//
// |x| as an unsigned integer orders like |x| itself; the row exponent e comes
// from the largest one: |x| < 2^(e-1) for every entry of the row.
__device__ __forceinline__ unsigned long long abs_bits(double x) {
    return static_cast<unsigned long long>(__double_as_longlong(x)) & 0x7FFFFFFFFFFFFFFFull;
}
__device__ __forceinline__ unsigned long long abs_bits(float x) { return __float_as_uint(x) & 0x7FFFFFFFu; }

template <typename T>
__device__ __forceinline__ int row_exponent(unsigned long long mx);
template <>
__device__ __forceinline__ int row_exponent<double>(unsigned long long mx) {
    if (mx == 0) return 0;
    const int E = static_cast<int>(mx >> 52);
    return E == 0 ? -1021 : E - 1021;   // |x| < 2^(E-1022) = 2^(e-1)
}
template <>
__device__ __forceinline__ int row_exponent<float>(unsigned long long mx) {
    if (mx == 0) return 0;
    const int E = static_cast<int>(mx >> 23);
    return E == 0 ? -125 : E - 125;
}

// round(x 2^(7 W - e)) as a signed integer, |result| <= 2^(7 W - 1): the row's window
// of W digits (W = 7: 49 bits; W = 9: 63 bits, every bit of the entries within a
// factor 2^-9 of the row's largest and 2^-63 of it for all).
template <int W>
__device__ __forceinline__ long long fixed_win(double x, int e) {
    const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
    const int E = static_cast<int>((b >> 52) & 0x7FF);
    const unsigned long long mant = (b & 0xFFFFFFFFFFFFFull) | (E ? (1ull << 52) : 0ull);
    const int sh = (E ? E : 1) - 1075 + 7 * W - e;   // x = mant 2^(E-1075); mant 2^sh < 2^(7 W - 1)
    long long v;
    if (sh >= 0) v = static_cast<long long>(mant << sh);
    else if (sh > -64) v = static_cast<long long>((mant + (1ull << (-sh - 1))) >> (-sh));
    else v = 0;
    return (b >> 63) ? -v : v;
}

template <int W>
__device__ __forceinline__ long long fixed_win(float x, int e) {
    const uint32_t b = __float_as_uint(x);
    const int E = static_cast<int>((b >> 23) & 0xFF);
    const unsigned long long mant = (b & 0x7FFFFFu) | (E ? 0x800000u : 0u);
    const int sh = (E ? E : 1) - 150 + 7 * W - e;
    long long v;
    if (sh >= 0) v = static_cast<long long>(mant << sh);
    else if (sh > -64) v = static_cast<long long>((mant + (1ull << (-sh - 1))) >> (-sh));
    else v = 0;
    return (b >> 31) ? -v : v;
}

// Signed base-2^7 digits of Y (|Y| <= 2^(7 W - 1)): slice s holds d_s 2^{-7(s+1)},
// |d_s| <= 64.  With a bias of 64 in each kept digit position (plus half of the
// last kept unit when S < W), U = Y + bias >= 0 has plain base-128 digits u_s,
// and d_s = u_s - 64: the S digits sum to Y exactly for S = W and to Y rounded
// to the last kept unit (nearest, ties up) for S < W.  Bit fields of one 64-bit
// integer (W = 9: U < 2^62 + 2^62 (1 + 2^-6) < 2^64), no carries to propagate.
template <int W>
__device__ __forceinline__ unsigned long long digit_bias(int S) {
    unsigned long long b = 0;
#pragma unroll
    for (int s = 0; s < W; ++s)
        if (s < S) b += 64ull << (7 * (W - 1 - s));
    if (S < W) b += 1ull << (7 * (W - S) - 1);
    return b;
}

// The digit u_s of U in slice s as a float, d_s 2^{-7(s+1)}: u below 256 put into the
// mantissa of 2^23 instead of converted (conversions run at a quarter of the rate), the
// bias and 2^23 taken off in the multiply-add that scales it; exact.
template <int W>
__device__ __forceinline__ float digit_value(unsigned long long U, int s) {
    const unsigned u = s ? static_cast<unsigned>(U >> (7 * (W - 1 - s))) & 127u : static_cast<unsigned>(U >> (7 * (W - 1)));
    const float sc = __int_as_float((127 - 7 * (s + 1)) << 23);   // 2^{-7(s+1)}
    return fmaf(__uint_as_float(0x4B000000u | u), sc, -8388672.0f * sc);
}

// Digits of two entries adjacent along K, stored as one bf16 pair per slice
// (out 4-byte aligned, slice_stride even); after nine digits the absolute values of the first.
template <int W>
__device__ __forceinline__ void write_digits2(long long Y0, long long Y1, int S, unsigned long long bias,
                                              __nv_bfloat16* out, long long slice_stride) {
    const unsigned long long U0 = static_cast<unsigned long long>(Y0) + bias;
    const unsigned long long U1 = static_cast<unsigned long long>(Y1) + bias;
#pragma unroll
    for (int s = 0; s < W; ++s) {
        if (s >= S) break;
        const __nv_bfloat162 w = __floats2bfloat162_rn(digit_value<W>(U0, s), digit_value<W>(U1, s));
        *reinterpret_cast<__nv_bfloat162*>(out + s * slice_stride) = w;
        if (W == OZ_DIGITS_F64 && s == 0 && S == W)
            *reinterpret_cast<__nv_bfloat162*>(out + W * slice_stride) = __habs2(w);
    }
}

// Eight entries adjacent along K: 16 bytes per slice (out 16-byte aligned).
template <int W>
__device__ __forceinline__ void write_digits8(const unsigned long long (&U)[8], int S, __nv_bfloat16* out,
                                              long long slice_stride) {
#pragma unroll
    for (int s = 0; s < W; ++s) {
        if (s >= S) break;
        __nv_bfloat162 w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) w[u] = __floats2bfloat162_rn(digit_value<W>(U[2 * u], s), digit_value<W>(U[2 * u + 1], s));
        *reinterpret_cast<uint4*>(out + s * slice_stride) = *reinterpret_cast<const uint4*>(w);
        if (W == OZ_DIGITS_F64 && s == 0 && S == W) {
#pragma unroll
            for (int u = 0; u < 4; ++u) w[u] = __habs2(w[u]);
            *reinterpret_cast<uint4*>(out + W * slice_stride) = *reinterpret_cast<const uint4*>(w);
        }
    }
}

// ---- slicing of both operands of one pass in one launch
//
// An operand is `rows` rows of K entries (row i, entry k at src[i s_row + k s_k];
// one of the strides is 1).  Its slices go to out[s slice_stride + i ldk + k] and
// the bits of max_k |x_ik| to mx[i].  FP32 sources are widened to FP64 on load
// (exact), so mx always holds FP64 bits.
struct OzOperand {
    const void* src;   // FP32 for operand 0 of the FP32-A instance, FP64 otherwise
    long long s_row, s_k, ldk, slice_stride;
    __nv_bfloat16* out;
    unsigned long long* mx;   // [passes][rows]
    int rows, K, S;
    int passes;     // ceil(K / OZ_KPASS): pass p is K range [p OZ_KPASS, min(K, (p + 1) OZ_KPASS))
    int tpr;        // K contiguous: threads per row, one per 8 of the pass (4, 8, 16 or whole warps)
    int rpc;        // rows per cluster: OZ_CS (OZ_ST / tpr) (K contiguous) or 32 (rows contiguous)
    int clusters;   // passes x ceil(rows / rpc): one cluster of OZ_CS CTAs per pass and rpc rows
};
struct OzSliceArgs {
    OzOperand op[2];
};

constexpr int OZ_CS = 8;                      // CTAs per cluster (the K split of a strided operand)
constexpr int OZ_ST = 512;                    // threads per CTA
constexpr int OZ_NW = OZ_ST / 32;
constexpr int OZ_KC_MAX = OZ_KPASS / OZ_CS;   // K per CTA of a strided operand (<= 128)

struct OzSmem {
    long long ys[OZ_KC_MAX][33];
    unsigned long long part[OZ_NW][32];
    unsigned long long lmax[32], rmax[32];
};

// mx[i] in FP64 form for the combine: the largest |entry| itself for FP64 rows;
// for FP32 rows an FP64 power of two with the same row exponent.
__device__ __forceinline__ unsigned long long mx_word(unsigned long long m, double*) { return m; }
__device__ __forceinline__ unsigned long long mx_word(unsigned long long m, float*) {
    return m ? static_cast<unsigned long long>(row_exponent<float>(m) + 1021) << 52 : 0ull;
}

// K contiguous (s_k == 1): tpr threads per row (one per 8 entries of the pass: 4, 8 or 16
// of a warp, or one to four warps), OZ_ST / tpr rows per CTA, eight adjacent entries along K per thread (16-byte
// stores per slice, 16-byte loads where the row is aligned); the row maximum is a
// shuffle, plus an exchange between the row's warps when there are several.  Bound by
// each CTA's chain (loads, row maximum, digits) as much as by memory: 3.6 GB over the
// factors' eight launches in 0.95-0.98 ms (0.99 as pairs with converted digits); the
// slices of a 20000 x 10000 FP64 sketch 3.4 -> 3.1 ms.
template <int W, typename T>
__device__ __forceinline__ void slice_kcontig(const OzOperand& o, int pass, int q, int rank, OzSmem& sm) {
    const long long koff = static_cast<long long>(pass) * OZ_KPASS;
    const T* src = static_cast<const T*>(o.src) + koff;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tpr = o.tpr;   // uniform over the cluster
    const int r = tid / tpr, l = tid - r * tpr;
    const int nw = tpr >> 5, rows = OZ_ST / tpr;   // (nw = 0: several rows per warp; with three warps per row the last warp idles)
    const long long i = static_cast<long long>(q) * o.rpc + rank * rows + r;
    const bool live = r < rows && i < o.rows;
    const int K = min(OZ_KPASS, o.K - pass * OZ_KPASS);   // <= 8 tpr
    T v[8];
    unsigned long long m = 0;
    const int k0 = 8 * l;
    const T* rs = src + i * o.s_row + k0;
    constexpr int VW = 16 / sizeof(T);
    if (live && k0 + 8 <= K && (reinterpret_cast<uintptr_t>(rs) & 15) == 0) {
#pragma unroll
        for (int u = 0; u < 8; u += VW) {
            const uint4 w = *reinterpret_cast<const uint4*>(rs + u);
            const T* p = reinterpret_cast<const T*>(&w);
#pragma unroll
            for (int q = 0; q < VW; ++q) v[u + q] = p[q];
        }
    } else {
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = live && k0 + u < K ? rs[u] : T(0);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) m = max(m, abs_bits(v[u]));
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, m, s);
        if (s < tpr) m = max(m, o);
    }
    if (nw > 1) {   // the row's warps
        if (lane == 0) sm.part[warp][0] = m;
        __syncthreads();
        if (live)
            for (int w = 0; w < nw; ++w) m = max(m, sm.part[nw * r + w][0]);
    }
    if (!live) return;   // no barrier follows in this path
    if (l == 0) o.mx[static_cast<long long>(pass) * o.rows + i] = mx_word(m, static_cast<T*>(nullptr));
    const int e = row_exponent<T>(m);
    if (k0 >= K) return;
    const unsigned long long bias = digit_bias<W>(o.S);
    unsigned long long U[8];   // entries past K are zero: ldk is K rounded up to 8
#pragma unroll
    for (int u = 0; u < 8; ++u) U[u] = static_cast<unsigned long long>(fixed_win<W>(v[u], e)) + bias;
    write_digits8<W>(U, o.S, o.out + i * o.ldk + koff + k0, o.slice_stride);
}

// Rows contiguous (s_row == 1): the cluster's 8 CTAs split K into chunks of
// <= 128; a CTA reads its 32 x chunk block along the rows (coalesced, 8
// entries per thread), the partial row maxima go through distributed shared
// memory, and the digits are written along K after a transpose in shared memory.
template <int W, typename T>
__device__ __forceinline__ void slice_strided(const OzOperand& o, int pass, int q, int rank, OzSmem& sm) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const long long koff = static_cast<long long>(pass) * OZ_KPASS;
    const T* src = static_cast<const T*>(o.src) + koff * o.s_k;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int K = min(OZ_KPASS, o.K - pass * OZ_KPASS);
    const int kc = ((K + OZ_CS - 1) / OZ_CS + 7) / 8 * 8;   // <= 128, a multiple of 8
    const int k0 = rank * kc, k1 = min(K, k0 + kc);
    const long long i = static_cast<long long>(q) * 32 + lane;
    const bool live = i < o.rows;
    T v[8];
    unsigned long long m = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int k = k0 + warp + OZ_NW * u;
        v[u] = live && k < k1 ? src[i + static_cast<long long>(k) * o.s_k] : T(0);
        m = max(m, abs_bits(v[u]));
    }
    sm.part[warp][lane] = m;
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int g = 1; g < OZ_NW; ++g) m = max(m, sm.part[g][lane]);
        sm.lmax[lane] = m;
    }
    cluster.sync();   // every CTA's partial maxima written
    if (warp == 0) {
        unsigned long long mr = 0;
#pragma unroll
        for (int c = 0; c < OZ_CS; ++c) mr = max(mr, cluster.map_shared_rank(sm.lmax, c)[lane]);
        sm.rmax[lane] = mr;
        if (rank == 0 && live) o.mx[static_cast<long long>(pass) * o.rows + i] = mx_word(mr, static_cast<T*>(nullptr));
    }
    cluster.sync();   // peers' reads of lmax done before any CTA moves on or exits
    const int e = row_exponent<T>(sm.rmax[lane]);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int kk = warp + OZ_NW * u;
        if (kk < kc) sm.ys[kk][lane] = fixed_win<W>(v[u], e);
    }
    __syncthreads();
    const int w = k1 - k0;
    if (w <= 0) return;
    // pairs along K: w is a multiple of 8 except in the last chunk, where an odd
    // w pairs the last entry with the zero row kk = w < kc (column K < ldk).
    // Thread: pair kp = tid % 64, rows tid / 64 + 8 j.
    const int wp = (w + 1) / 2, kp = tid & 63;
    if (kp >= wp) return;
    const unsigned long long bias = digit_bias<W>(o.S);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int ii = (tid >> 6) + 8 * j;
        const long long row = static_cast<long long>(q) * 32 + ii;
        if (row < o.rows)
            write_digits2<W>(sm.ys[2 * kp][ii], sm.ys[2 * kp + 1][ii], o.S, bias, o.out + row * o.ldk + koff + k0 + 2 * kp,
                          o.slice_stride);
    }
}

// Cluster q of the grid slices pass p, rows [rpc q', rpc q' + rpc) of operand 0
// (FP32 when A32) for q < op[0].clusters, else of operand 1 (FP64), with
// q - (operand base) = p ceil(rows / rpc) + q'.
template <bool A32, int W>
__global__ void __launch_bounds__(OZ_ST) oz_slice_kernel(const __grid_constant__ OzSliceArgs args) {
    __shared__ OzSmem sm;
    const int rank = static_cast<int>(cooperative_groups::this_cluster().block_rank());
    int q = static_cast<int>(blockIdx.x) / OZ_CS;
    const int which = q < args.op[0].clusters ? 0 : 1;
    const OzOperand& o = args.op[which];
    if (which) q -= args.op[0].clusters;
    const int rq = (o.rows + o.rpc - 1) / o.rpc;
    const int pass = q / rq;
    q -= pass * rq;
    if (which == 0 && A32) {
        if (o.s_k == 1) slice_kcontig<W, float>(o, pass, q, rank, sm);
        else slice_strided<W, float>(o, pass, q, rank, sm);
    } else {
        if (o.s_k == 1) slice_kcontig<W, double>(o, pass, q, rank, sm);
        else slice_strided<W, double>(o, pass, q, rank, sm);
    }
}

OzOperand oz_operand(const void* src, long long s_row, long long s_k, long long rows, long long K, int S,
                     __nv_bfloat16* out, long long ldk, long long slice_stride, unsigned long long* mx) {
    OzOperand o;
    o.src = src;
    o.s_row = s_row;
    o.s_k = s_k;
    o.rows = static_cast<int>(rows);
    o.K = static_cast<int>(K);
    o.S = S;
    o.out = out;
    o.ldk = ldk;
    o.slice_stride = slice_stride;
    o.mx = mx;
    o.passes = static_cast<int>((K + OZ_KPASS - 1) / OZ_KPASS);
    o.tpr = s_k != 1 ? 0 : K <= 32 ? 4 : K <= 64 ? 8 : K <= 128 ? 16 : 32 * static_cast<int>((std::min<long long>(K, OZ_KPASS) + 255) / 256);
    o.rpc = s_k == 1 ? OZ_CS * (OZ_ST / o.tpr) : 32;
    o.clusters = o.passes * static_cast<int>((rows + o.rpc - 1) / o.rpc);
    return o;
}

// Both operands, every pass of their K range (at most OZ_PGRP passes), in one launch.
gn_status slice_pair(gn_handle h, const OzOperand& a, int a_f32, const OzOperand& b) {
    OzSliceArgs args;
    args.op[0] = a;
    args.op[1] = b;
    for (const OzOperand& o : args.op)
        if ((o.s_k != 1 && o.s_row != 1) || o.K < 1 || o.passes > OZ_PGRP || o.rows < 1) return GN_ERR_INVALID_ARG;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(OZ_CS * (static_cast<long long>(a.clusters) + b.clusters)));
    cfg.blockDim = dim3(OZ_ST);
    cfg.stream = h->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = OZ_CS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (a.S > 7 || b.S > 7) {
        if (a_f32) return GN_ERR_INVALID_ARG;
        GN_CUDA_TRY(cudaLaunchKernelEx(&cfg, oz_slice_kernel<false, OZ_DIGITS_F64>, args));
    } else if (a_f32) {
        GN_CUDA_TRY(cudaLaunchKernelEx(&cfg, oz_slice_kernel<true, 7>, args));
    } else {
        GN_CUDA_TRY(cudaLaunchKernelEx(&cfg, oz_slice_kernel<false, 7>, args));
    }
    count_launch();
    return GN_OK;
}

// The operands of a product with eight or nine digits: an entry of C whose row of A or
// column of B is not finite in a part, or (nine) whose size is below OZ_SMALL, is formed
// from the operands themselves.  A null: not checked.
struct OzDirect {
    const double *A, *B;
    long long a_row, a_k, b_row, b_k;
    int K;
};

// Part q of entry (i, j), j a lane's own column, for the lanes of `need` (a warp has one row
// i and the columns of its first popc(live) lanes; all of these call).  A few entries: the
// lanes share each one's sum.  Many: a lane each, eight terms loaded ahead.
__device__ __noinline__ double oz_direct_dot(const OzDirect& x, int q, int i, int j, unsigned need, unsigned live) {
    const int lane = threadIdx.x & 31, k0 = q * OZ_KPASS, k1 = min(x.K, k0 + OZ_KPASS);
    const double* a = x.A + i * x.a_row;
    const double* b = x.B + j * x.b_row;
    double s = 0.0;
    if (__popc(need) > 8) {
        if (need >> lane & 1) {
            int k = k0;
            for (; k + 8 <= k1; k += 8) {
                double av[8], bv[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    av[u] = a[(k + u) * x.a_k];
                    bv[u] = b[(k + u) * x.b_k];
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) s = fma(av[u], bv[u], s);
            }
            for (; k < k1; ++k) s = fma(a[k * x.a_k], b[k * x.b_k], s);
        }
        return s;
    }
    const int cnt = __popc(live);
    for (unsigned todo = need; todo; todo &= todo - 1) {
        const int t = __ffs(todo) - 1;
        const double* bt = x.B + (j - lane + t) * x.b_row;
        double p = 0.0;
        for (int k = k0 + lane; k < k1; k += cnt) p = fma(a[k * x.a_k], bt[k * x.b_k], p);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double y = __shfl_down_sync(live, p, o);
            if (lane + o < cnt) p += y;
        }
        p = __shfl_sync(live, p, 0);
        if (lane == t) s = p;
    }
    return s;
}

// C[i, j] = beta C[i, j] + sum_q alpha 2^{ea_qi + eb_qj} sum_o D_qo[i, j] over
// the K parts q (passes, each with its own row exponents), added in part
// order with one rounding each.  Within a part the first NEX orders are summed
// as integers (one rounding), the orders below them in FP32.  NEX = 4 for up to
// seven digits (units of 2^-35: the orders that are always exact); 6 for eight and
// nine (units of 2^-49, so that the FP32 sum of the last orders rounds below 2^-60
// of the leading one).  With nine digits the orders 4 and 5 come as two outputs,
// the second ones in slots 9 and 10, so that these are exact too (slot 11 is the
// entry's size); with eight they are exact unless their sums pass 2^24 units.  A thread per column and row group
// (no division per element; narrow products fill a block with more rows); each
// output of an exact order is an integer of at most 2^24 units and converts
// through a 32-bit integer.
template <int NORD>
__global__ void __launch_bounds__(256) oz_combine_kernel(
    const float* __restrict__ D, long long d_stride, long long part_stride, long long ldd, int nparts, int M, int N,
    const unsigned long long* __restrict__ mxa, const unsigned long long* __restrict__ mxb, long long mxb_part,
    double alpha, double beta, double* __restrict__ C, long long ldc, int cw, const __grid_constant__ OzDirect direct,
    int j0) {
    constexpr int NEX = NORD > 7 ? 6 : 4, NEXACT = NORD < NEX ? NORD : NEX;
    constexpr int NOUT = NORD == OZ_DIGITS_F64 ? OZ_OUTS_F64 : NORD;
    // a block is cw columns by blockDim.x / cw rows (cw: a power of two >= min(N, 256), >= 32)
    const int j = blockIdx.x * cw + static_cast<int>(threadIdx.x) % cw;
    const int rb = static_cast<int>(blockDim.x) / cw, step = gridDim.y * rb;
    const unsigned live = __ballot_sync(0xffffffffu, j < N);   // (a warp's columns are consecutive)
    if (j >= N) return;
    const bool unit = alpha == 1.0 || alpha == -1.0;
    const int flip = alpha == -1.0 ? static_cast<int>(0x80000000u) : 0;
    // one part of one entry from its orders
    auto value = [&](const float (&d)[NOUT], int q, int i) {
        long long acc = 0;
#pragma unroll
        for (int o = 0; o < NEXACT; ++o) {   // D_o is an integer number of units 2^{-7(o+2)}
            const float unit_inv = __int_as_float((127 + 7 * (o + 2)) << 23);
            int u = __float2int_rn(d[o] * unit_inv);
            if (NOUT > NORD && o >= 4) u += __float2int_rn(d[NORD + o - 4] * unit_inv);
            acc += static_cast<long long>(u) << (7 * (NEX - 1 - o));
        }
        float low = 0.0f;
#pragma unroll
        for (int o = NORD - 1; o >= NEX; --o) low += d[o];
        // times 2^(ea + eb - 7 (NEX + 1)): a power of two built from its bits when normal
        const unsigned long long ma = mxa[static_cast<long long>(q) * M + i], mb = mxb[q * mxb_part + j];
        const int p = row_exponent<double>(ma) + row_exponent<double>(mb) - 7 * (NEX + 1);
        const double x = fma(static_cast<double>(low), static_cast<double>(1ull << (7 * (NEX + 1))),
                             static_cast<double>(acc));
        // times 2^p by the exponent field where x and the result are normal, times alpha = +-1 by the
        // sign (every FP64 instruction counts: the units run at 1/64 of the FP32 rate)
        const int ex = ((__double2hiint(x) >> 20) & 0x7FF), er = ex + p;
        double v = 0.0;
        if (ex > 0 && er > 0 && er < 0x7FF) {
            v = __hiloint2double((__double2hiint(x) + p * (1 << 20)) ^ flip, __double2loint(x));
            if (!unit) v *= alpha;
        } else if ((__double2hiint(x) << 1 | __double2loint(x)) != 0) {
            v = alpha * ldexp(x, p);
        }
        if (NEX == 6) {
            const bool need = direct.A && (max(ma, mb) >= 0x7FF0000000000000ull ||
                                           (NOUT > NORD && ma && mb && d[NOUT - 1] < OZ_SMALL));
            const unsigned any = __ballot_sync(live, need);
            if (any) {
                const double x = oz_direct_dot(direct, q, i, j0 + j, any, live);
                if (need) v = alpha * x;
            }
        }
        return v;
    };
    int i = blockIdx.y * rb + static_cast<int>(threadIdx.x) / cw;
    // one part: two rows at a time, both rows' orders loaded before either is used (32768 x
    // 128, 8 orders: 80 -> 69 us); several parts already have that many loads in flight
    if (nparts == 1)
        for (; i + step < M; i += 2 * step) {
            double* c = C + static_cast<long long>(i) * ldc + j;
            double* c2 = c + step * ldc;
            const float* p = D + static_cast<long long>(i) * ldd + j;
            const float* p2 = p + step * ldd;
            float d[NOUT], e[NOUT];
#pragma unroll
            for (int o = 0; o < NOUT; ++o) {
                d[o] = p[o * d_stride];
                e[o] = p2[o * d_stride];
            }
            const double v = value(d, 0, i), v2 = value(e, 0, i + step);
            *c = beta == 0.0 ? v : fma(beta, *c, v);
            *c2 = beta == 0.0 ? v2 : fma(beta, *c2, v2);
        }
    for (; i < M; i += step) {
        double* c = C + static_cast<long long>(i) * ldc + j;
        double out = 0.0;
        for (int q = 0; q < nparts; ++q) {   // K parts (passes) in order, as separate passes would add them
            const float* p = D + q * part_stride + static_cast<long long>(i) * ldd + j;
            float d[NOUT];
#pragma unroll
            for (int o = 0; o < NOUT; ++o) d[o] = p[o * d_stride];
            const double v = value(d, q, i);
            out = q ? out + v : (beta == 0.0 ? v : fma(beta, *c, v));
        }
        *c = out;
    }
}

struct OzWs {
    __nv_bfloat16 *as, *bs;
    float* d;
    unsigned long long *mxa, *mxb;
    long long ldk, ldd;
};

// K per group of passes, its passes, and the workspace carve for them.
long long oz_kgroup(long long K) { return std::min<long long>(std::max<long long>(K, 1), OZ_PGRP * OZ_KPASS); }
long long oz_parts(long long kg) { return (kg + OZ_KPASS - 1) / OZ_KPASS; }

bool oz_carve(long long M, long long N, long long K, int sa, int sb, void* ws, size_t ws_bytes, OzWs* o) {
    const long long kg = oz_kgroup(K), S = oz_parts(kg), np = oz_npanel(M, N, S, oz_outputs(sa));
    o->ldk = r8(kg);
    o->ldd = r4(np);
    char* p = static_cast<char*>(ws);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char* q = p + off;
        off += al256(bytes);
        return q;
    };
    o->as = reinterpret_cast<__nv_bfloat16*>(take(sizeof(__nv_bfloat16) * oz_slices(sa) * M * o->ldk));
    o->bs = reinterpret_cast<__nv_bfloat16*>(take(sizeof(__nv_bfloat16) * oz_slices(sb) * N * o->ldk));
    o->d = reinterpret_cast<float*>(take(sizeof(float) * S * oz_outputs(sa) * M * o->ldd));
    o->mxa = reinterpret_cast<unsigned long long*>(take(sizeof(unsigned long long) * S * M));
    o->mxb = reinterpret_cast<unsigned long long*>(take(sizeof(unsigned long long) * S * N));
    return off <= ws_bytes;
}

}  // namespace

size_t oz_ws_bytes(long long M, long long N, long long K, int a_f32, int digits) {
    (void)a_f32;
    const int slices = oz_slices(digits), nout = oz_outputs(digits);
    const long long kg = oz_kgroup(K), S = oz_parts(kg);
    // the FP32 outputs of s parts at the panel for s parts, largest over s <= S:
    // the panel narrows as the parts grow, and the size must not shrink with K
    size_t d = 0;
    for (long long s = 1; s <= S; ++s)
        d = std::max(d, al256(sizeof(float) * s * nout * M * r4(oz_npanel(M, std::max<long long>(N, 1), s, nout))));
    return al256(sizeof(__nv_bfloat16) * slices * M * r8(kg)) + al256(sizeof(__nv_bfloat16) * slices * N * r8(kg)) + d +
           al256(8 * S * M) + al256(8 * S * N) + 256;
}

gn_status oz_dgemm(gn_handle h, long long M, long long N, long long K, double alpha, const void* A, int a_f32,
                   long long lda, int ta, const double* B, long long ldb, int tb, double beta, double* C,
                   long long ldc, void* ws, size_t ws_bytes, int digits) {
    if (M <= 0 || N <= 0) return GN_OK;
    if (K <= 0 || !A || !B || !C || !ws || digits < 2 || (digits > 7 && (digits > OZ_DIGITS_F64 || a_f32)))
        return GN_ERR_INVALID_ARG;
    const int sa = digits, sb = digits;
    if (M > (1LL << 30) || N > (1LL << 30)) return GN_ERR_SHAPE;
    OzWs o;
    if (!oz_carve(M, N, K, sa, sb, ws, ws_bytes, &o)) return GN_ERR_WORKSPACE;
    // outputs: the slice products (s, ord - s) of every order 0 .. digits - 1, the orders 4 and 5 of
    // nine digits cut after OZ_CUT of them (the rest in the slots after the orders'), the size last
    const int ns = oz_slices(digits);
    struct Out {
        int slot, ord, s0, n;   // slice products (s0 + q, ord - s0 - q), q < n
    };
    Out outs[OZ_OUTS_F64];
    const int nout = oz_outputs(digits);
    for (int ord = 0; ord < digits; ++ord) {
        const bool cut = nout > digits && (ord == 4 || ord == 5);
        outs[ord] = Out{ord, ord, 0, cut ? OZ_CUT : ord + 1};
        if (cut) outs[digits + ord - 4] = Out{digits + ord - 4, ord, OZ_CUT, ord + 1 - OZ_CUT};
    }
    if (nout > digits) outs[nout - 1] = Out{nout - 1, 2 * digits, digits, 1};   // slice `digits` of both
    if (nout > TC_MAX_GEMMS || 2 * ns > TC_MAX_MAPS || digits > TC_MAX_SRC) return GN_ERR_UNSUPPORTED;
    // Launch order: the longest first.  Lengths digits, digits - 1, ..., 1 are paired to equal loads
    // by the boustrophedon order on (digits + 1) / 2 groups of CTAs (seven digits: 7; 6 + 1; 5 + 2;
    // 4 + 3).  Nine digits' 9, 8, 7, 4, 4, 4, 3, 2, 2, 1, 1, 1 are when the tiles fill the SMs several
    // times; with a CTA group per tile they go 4 + 4 + 1, 4 + 3 + 2, 7 + 2, 8 + 1, 9 + 1 (at most 10
    // slice products per CTA; 11 in decreasing order).
    std::stable_sort(outs, outs + nout, [](const Out& a, const Out& b) { return a.n > b.n; });
    Out few[OZ_OUTS_F64];
    if (nout > digits) {
        const int by[OZ_OUTS_F64] = {4, 4, 7, 8, 9, 1, 1, 2, 3, 4, 1, 2};   // lengths
        bool used[OZ_OUTS_F64] = {};
        for (int i = 0; i < nout; ++i)
            for (int q = 0; q < nout; ++q)
                if (!used[q] && outs[q].n == by[i]) {
                    used[q] = true;
                    few[i] = outs[q];
                    break;
                }
    }
    const long long as_stride = M * o.ldk, bs_stride = N * o.ldk, d_stride = M * o.ldd;
    // groups of at most OZ_PGRP passes: one slicing launch for all of them, the
    // passes as K-aligned parts of one multi-GEMM launch (stored apart), one
    // combination adding them in order
    const long long part_stride = nout * d_stride;
    const long long npanel = oz_npanel(M, N, oz_parts(oz_kgroup(K)), nout);   // the carve's panel (largest group)
    for (long long k0 = 0; k0 < K; k0 += OZ_PGRP * OZ_KPASS) {
        const long long kc = std::min<long long>(OZ_PGRP * OZ_KPASS, K - k0);
        const int S = static_cast<int>(oz_parts(kc));
        // A rows (i over M, k along the group) and B "rows" (j over N)
        const long long a_row = ta ? 1 : lda, a_k = ta ? lda : 1;
        const long long a_off = ta ? k0 * lda : k0;
        const long long b_row = tb ? ldb : 1, b_k = tb ? 1 : ldb;
        const long long b_off = tb ? k0 : k0 * ldb;
        const size_t esz = a_f32 ? sizeof(float) : sizeof(double);
        GN_TRY(slice_pair(h,
                          oz_operand(static_cast<const char*>(A) + esz * a_off, a_row, a_k, M, kc, sa, o.as, o.ldk,
                                     as_stride, o.mxa),
                          a_f32, oz_operand(B + b_off, b_row, b_k, N, kc, sb, o.bs, o.ldk, bs_stride, o.mxb)));
        const double beta_grp = k0 == 0 ? beta : 1.0;
        for (long long j0 = 0; j0 < N; j0 += npanel) {
            const long long nb = std::min<long long>(npanel, N - j0);
            // N tile: the widest of 256 / 128 / 64 that still gives the GPU about
            // two work items per SM over the orders and parts (small products are latency-bound)
            int bn = static_cast<int>(std::min<long long>(256, (nb + 31) / 32 * 32));
            while (bn > 64 && ((M + 127) / 128) * ((nb + bn - 1) / bn) * nout * S < 2LL * h->sm_count)
                bn = (bn / 2 + 31) / 32 * 32;
            TcParams p;
            memset(&p, 0, sizeof(p));
            for (int s = 0; s < ns; ++s)
                GN_TRY(tc_make_map_bf16(&p.maps[s], o.as + s * as_stride, M, kc, o.ldk, 64, 128));
            for (int t = 0; t < ns; ++t)
                GN_TRY(tc_make_map_bf16(&p.maps[ns + t], o.bs + t * bs_stride + j0 * o.ldk, nb, kc, o.ldk, 64, bn));
            const bool spread = nout > digits && (digits + 1) / 2 * ((M + 127) / 128) * ((nb + bn - 1) / bn) * S <= h->sm_count;
            for (int gi = 0; gi < nout; ++gi) {
                const Out& out = spread ? few[gi] : outs[gi];
                TcGemm& g = p.g[gi];
                g.M = static_cast<int>(M);
                g.N = static_cast<int>(nb);
                g.K = static_cast<int>(kc);
                g.bn = bn;
                g.a_mn = 0;
                g.b_mn = 0;
                g.nsrc = out.n;
                for (int q = 0; q < out.n; ++q) {
                    g.a_map[q] = static_cast<signed char>(out.s0 + q);
                    g.b_map[q] = static_cast<signed char>(ns + out.ord - out.s0 - q);
                }
                g.D = o.d + out.slot * d_stride;
                g.ldd = o.ldd;
                if (S >= 2) {   // pass q of the group: its own row scaling, stored at D + q part_stride
                    g.ksplit = S;
                    g.part_stride = part_stride;
                    g.kpart = OZ_KPASS / TC_BK;
                }
            }
            p.ngemm = nout;
            p.snake_groups = (digits + 1) / 2;
            GN_TRY(tc_launch(h, &p));
            int cw = 32;   // a power of two, so that it divides the block's 256 threads
            while (cw < nb && cw < 256) cw *= 2;
            const long long rows_per_block = 256 / cw;
            const unsigned gx = static_cast<unsigned>((nb + cw - 1) / cw);
            const unsigned gy = static_cast<unsigned>(std::max<long long>(
                1, std::min<long long>((M + rows_per_block - 1) / rows_per_block,
                                       static_cast<long long>(h->sm_count) * 16 / gx)));
            OzDirect dd{};
            if (digits > 7)
                dd = OzDirect{static_cast<const double*>(A) + a_off, B + b_off, a_row, a_k, b_row, b_k,
                              static_cast<int>(kc)};
            auto combine = [&]() {
                switch (digits) {
                    case 2: return oz_combine_kernel<2>;
                    case 3: return oz_combine_kernel<3>;
                    case 4: return oz_combine_kernel<4>;
                    case 5: return oz_combine_kernel<5>;
                    case 6: return oz_combine_kernel<6>;
                    case 7: return oz_combine_kernel<7>;
                    case 8: return oz_combine_kernel<8>;
                    default: return oz_combine_kernel<9>;
                }
            }();
            combine<<<dim3(gx, gy), 256, 0, h->stream>>>(
                o.d, d_stride, part_stride, o.ldd, S, static_cast<int>(M), static_cast<int>(nb), o.mxa, o.mxb + j0, N,
                alpha, beta_grp, C + j0, ldc, cw, dd, static_cast<int>(j0));
            count_launch();
            GN_CUDA_TRY(cudaGetLastError());
        }
    }
    return GN_OK;
}

// ---- FP64 products with nine digits per operand, or on the FP64 units
namespace {
// Blocks of C per digit-sliced product: the scratch (the slices of up to 4096 of K)
// stays near 2 GB however large the matrices are.
constexpr long long OZ_MBLK = 8192, OZ_NBLK = 16384;
// Microseconds of a nine-digit product: per block of C and group of K, three launches, the longest
// chain of slice products of one tile (10 per 64 of K, 0.28 us for 64 columns, 0.49 for 256) or
// all of them over the SMs, the slices and the outputs through memory.
double oz_us(long long M, long long N, long long K, int sms) {
    const double m = static_cast<double>(std::min(M, OZ_MBLK)), n = static_cast<double>(std::min(N, OZ_NBLK));
    const long long kc = std::min<long long>(K, OZ_PGRP * OZ_KPASS), parts = (kc + OZ_KPASS - 1) / OZ_KPASS;
    const double bn = std::min(256.0, n), c = 0.21 + 0.0011 * bn, kb = static_cast<double>(std::min<long long>(16, (kc + 63) / 64));
    const double tiles = static_cast<double>((std::min(M, OZ_MBLK) + 127) / 128) * std::max(1.0, n / bn) * parts;
    const double one = 15.0 + kb * c * std::max(10.0, 46.0 * tiles / sms) + (m + n) * kc * 28.0 / 4e6 + m * n * parts * 100.0 / 4e6;
    return one * std::max(1.0, M / m) * std::max(1.0, N / n) * std::max(1.0, static_cast<double>(K) / kc);
}
// Products of up to 16 M multiply-adds stay on the FP64 units (three launches and a tile's chain
// take ~40 us whatever the size), and larger ones that the estimates put at half the time
// there: few rows and columns over a long K, or few of them against many over a short one,
// where a tile of 128 rows and its slices are mostly padding.  Both products of a sketch at
// m, n, r, l = 1000, 500, 20, 10: 115 us in slices, 73 on the units; 4096, 2048, 100, 50: 0.45 ms
// and 5.25; 20000, 10000, 500, 250: 23.0 and 428.5; 100000, 40, 10, 5: 2.12 and 0.78; 40, 100000,
// 10, 5: 2.37 and 1.57.
bool oz_f64_pays(long long M, long long N, long long K, int sms) {
    return M >= 1 && N >= 1 && K >= 1 && !small_gemm(M, N, K) && 0.5 * oz_us(M, N, K, sms) < f64_units_us(M, N, K, sms);
}
}  // namespace

size_t dgemm_fast_ws_bytes(long long M, long long N, long long K, int sm_count) {
    size_t b = dgemm_ws_bytes(M, N, K, sm_count);
    if (!oz_f64_pays(M, N, K, sm_count)) return b;
    for (long long mm : {std::min(M, OZ_MBLK), M % OZ_MBLK})
        for (long long nn : {std::min(N, OZ_NBLK), N % OZ_NBLK})
            if (mm > 0 && nn > 0) b = std::max(b, oz_ws_bytes(mm, nn, K, 0, OZ_DIGITS_F64) + 256);
    return b;
}

gn_status dgemm_fast(gn_handle h, long long M, long long N, long long K, double alpha, const double* A,
                     long long lda, int ta, const double* B, long long ldb, int tb, double beta, double* C,
                     long long ldc, double* ws, size_t ws_bytes) {
    const size_t need = dgemm_fast_ws_bytes(M, N, K, h->sm_count);
    if (!h->fp64_tc || !ws || ws_bytes < need || !oz_f64_pays(M, N, K, h->sm_count))
        return dgemm(h, M, N, K, alpha, A, lda, ta, B, ldb, tb, beta, C, ldc, ws, ws_bytes);
    const size_t pad = (256 - (reinterpret_cast<uintptr_t>(ws) & 255)) & 255;
    char* base = reinterpret_cast<char*>(ws) + pad;
    for (long long j0 = 0; j0 < N; j0 += OZ_NBLK)
        for (long long i0 = 0; i0 < M; i0 += OZ_MBLK)
            GN_TRY(oz_dgemm(h, std::min(OZ_MBLK, M - i0), std::min(OZ_NBLK, N - j0), K, alpha,
                            A + (ta ? i0 : i0 * lda), 0, lda, ta, B + (tb ? j0 * ldb : j0), ldb, tb, beta,
                            C + i0 * ldc + j0, ldc, base, ws_bytes - pad, OZ_DIGITS_F64));
    return GN_OK;
}

}  // namespace gn
