// Batched generalized Nystrom: the sketches (Algorithm 2, step 2) and the core
// (C = Y^T A X, Householder QR, Section 5.1.1/5.1.2) of many independent
// problems of uneven m, n, r, in a fixed sequence of four launches:
//
//   1. one grouped tcgen05 launch computing AX and Y^T A of every problem (the
//      two products of a problem are adjacent in the tile order, so its A is
//      still in L2 when the second product streams it);
//   2. one launch splitting every Y^T A into three BF16 slices;
//   3. one grouped tcgen05 launch for the three slice products of every core;
//   4. one launch with a cluster of four CTAs per problem (large batches: one
//      CTA, see bc_pays): C = sum of the slice
//      products in FP64, Householder QR in shared memory, R and Q (formed in place), the
//      detector / truncation, and the second QR when the core is truncated.
//
// gn_batched_prepare builds every descriptor and TMA tensor map on the host and
// uploads them into the caller's workspace once; gn_batched_run only launches
// kernels on the handle's stream (no host synchronisation, no allocation).
#include "gn_internal.cuh"
#include "gn_push.cuh"
#include "gn_smem_core.cuh"

#include <cooperative_groups.h>
#include <string.h>

#include <algorithm>
#include <vector>

namespace gn {
namespace {
using namespace smemcore;

constexpr int DIAG_ITERS_B = 6;

struct ProblemDev {
    int m, n, r, l;
    const float* YtA;
    long long ld_yta;
    __nv_bfloat16* s[3];     // slices of Y^T A, (r+l) x lds
    long long lds;
    float* cpart[3];         // slice products, (r+l) x r
    double* Q;
    double* R;
    double* Q2;
    double* R2;
    int* k;
    double* diag;            // [3]: est ||R^{-1}||, est ||C||, eps used
    int* sgn;
};

size_t al(size_t b) { return (b + 255) & ~static_cast<size_t>(255); }
long long r8(long long x) { return (x + 7) / 8 * 8; }

// ----------------------------------------------------------------------------
// 2. split every Y^T A into hi / mid / lo BF16 slices (blockIdx.y = problem)
__global__ void batched_split3_kernel(const ProblemDev* __restrict__ P) {
    const ProblemDev& p = P[blockIdx.y];
    const long long rows = p.r + p.l, cols = p.n, total = rows * cols;
    for (long long e = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; e < total;
         e += static_cast<long long>(gridDim.x) * blockDim.x) {
        const long long i = e / cols, j = e % cols;
        const float x = p.YtA[i * p.ld_yta + j];
        const __nv_bfloat16 h = __float2bfloat16_rn(x);
        const float r1 = x - __bfloat162float(h);
        const __nv_bfloat16 m = __float2bfloat16_rn(r1);
        const float r2 = r1 - __bfloat162float(m);
        p.s[0][i * p.lds + j] = h;
        p.s[1][i * p.lds + j] = m;
        p.s[2][i * p.lds + j] = __float2bfloat16_rn(r2);
    }
}

// ----------------------------------------------------------------------------
// 4. per-problem core: a cluster of four CTAs per problem.
//
// The core's ~10 M multiply-adds (r = 128, l = 64) are 1.5 ms at one SM's FP64 rate and
// its columns a chain, so one CTA per core bounds a batch by its largest core (2.64 ms)
// while other SMs idle.  Here row i of the core lives in CTA i % 4 (in shared memory),
// warp (i / 4) % 8, so that every CTA has a share of the rows left at every column.  A
// column is one pass over the warp's rows (each row updated by the last reflector and
// at once summed for the next column's dots: a lane per column, no barrier between),
// the sums over the eight warps, one push exchange with the other CTAs, and the
// reflector's scalars.  The formation of Q runs the same way from the last column back.
// Three such CTAs share an SM, so one's chain overlaps another's passes.
// Whole batches, r in 16 .. 128, against one CTA per core: 1 problem 2556 -> 1215 us,
// 32: 2628 -> 1259, 128: 2860 -> 1808, 256: 3003 -> 2562; r in 16 .. 32: 1: 237 -> 143,
// 128: 408 -> 354, 400: 1023 -> 910.  The exchanges and the sums over the ranks are
// FP64 instructions too, so a batch bound by the SMs' total FP64 work keeps one CTA per
// core (400 problems of r in 16 .. 128: 3383 against 3698; 4b): see bc_pays.
namespace cg = cooperative_groups;
using namespace pushx;
constexpr int BC_CS = 4;
constexpr int BC_T = 256;
constexpr int BC_W = BC_T / 32;
constexpr int BC_L = (MMAX + BC_CS - 1) / BC_CS;   // rows per CTA
constexpr int BC_NG = NMAX / 32;

struct BcSmem {
    double S[BC_L * (NMAX + 1)];
    double red[BC_W * NMAX];
    double recv[2][BC_CS][NMAX];   // the CTAs' sums, pushed by them
    double rowj[2][NMAX];          // row j of the core, pushed by its owner
    double gs[NMAX];               // the update's coefficients
    double amb[NMAX], d[NMAX], beta[NMAX];
    double est, rn;                // read by the peers
    int k;
    unsigned long long bars[2];
};

struct BcState {
    int rank, step;
    bool dead;
    unsigned long long limit;
};

// One exchange: `cnt` sums per CTA (columns c0 .. c0 + cnt: red over the warps), with
// row j of its owner when owner >= 0.  Afterwards recv[par] and rowj[par] are filled.
// Returns par.  No CTA writes recv[par] again before every peer has read it: a peer's
// next push but one needs this CTA's next push, which follows the barrier after the reads.
__device__ __forceinline__ int bc_exchange(BcSmem& sm, BcState& st, int c0, int cnt, int owner, int lj, int ld) {
    const int tid = threadIdx.x, par = st.step & 1;
    const uint32_t bar = sm_u32(&sm.bars[par]);
    if (tid == 0 && !st.dead)
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                     "r"((BC_CS + (owner >= 0 ? 1 : 0)) * cnt * 8)
                     : "memory");
    __syncthreads();   // red complete (and every earlier read of the buffers)
    if (tid < NMAX) {
        if (tid < cnt) {
            const int c = c0 + tid;
            double s[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) s[q] = sm.red[q * NMAX + c] + sm.red[(q + 4) * NMAX + c];
            const double v = (s[0] + s[1]) + (s[2] + s[3]);
#pragma unroll
            for (int k = 0; k < BC_CS; ++k)
                push(map_rank(sm_u32(&sm.recv[par][st.rank][c]), k), v, map_rank(bar, k));
        }
    } else if (owner == st.rank && tid - NMAX < cnt) {
        const int c = c0 + tid - NMAX;
        const double v = sm.S[lj * ld + c];
#pragma unroll
        for (int k = 0; k < BC_CS; ++k) push(map_rank(sm_u32(&sm.rowj[par][c]), k), v, map_rank(bar, k));
    }
    if (!st.dead && !wait(bar, (st.step >> 1) & 1, st.limit)) st.dead = true;
    ++st.step;
    return par;
}

// Householder QR of the M x N core in place: R on and above the diagonal, the raw
// reflectors below (xt_j: amb_j in row j, the column as it was below it), and amb, d,
// beta per column, H_j = I + d_j xt_j xt_j^T (d_j = 0: no reflector).
__device__ void bc_qr(BcSmem& sm, BcState& st, int M, int N) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, ld = N + 1;
    const int L = (M - st.rank + BC_CS - 1) / BC_CS;   // own rows
    if (tid < NMAX) sm.gs[tid] = 0.0;
    double gq[BC_NG];
#pragma unroll
    for (int g = 0; g < BC_NG; ++g) gq[g] = 0.0;
    for (int j = 0; j < N; ++j) {
        // reflector j - 1 applied to rows j - 1 and below, and the dots of column j with
        // the columns from j on over the rows below j
        double acc[BC_NG];
#pragma unroll
        for (int g = 0; g < BC_NG; ++g) acc[g] = 0.0;
        const double ambp = j ? sm.amb[j - 1] : 0.0;
        const int gj = j >> 5, ja = max(0, j - 1);
        int li = ja <= st.rank ? 0 : (ja - st.rank + BC_CS - 1) / BC_CS;   // first own row >= ja
        li += (warp - li) & (BC_W - 1);                                     // ... of this warp
        for (; li < L; li += BC_W) {
            const int i = BC_CS * li + st.rank;
            double* row = sm.S + li * ld;
            const double x = j == 0 ? 0.0 : (i == j - 1 ? ambp : row[j - 1]);
            double v[BC_NG];
#pragma unroll
            for (int g = 0; g < BC_NG; ++g) {
                v[g] = 0.0;
                if (g < gj || 32 * g >= N) continue;   // warp-uniform
                const int q = 32 * g + lane;
                if (q < N) {
                    v[g] = row[q];
                    if (j) {
                        v[g] = fma(x, gq[g], v[g]);   // gq is 0 left of column j
                        row[q] = v[g];
                    }
                }
            }
            if (i <= j) continue;   // warp-uniform
            double y = 0.0;
#pragma unroll
            for (int g = 0; g < BC_NG; ++g)
                if (g == gj) y = __shfl_sync(0xffffffffu, v[g], j & 31);
#pragma unroll
            for (int g = 0; g < BC_NG; ++g)
                if (g >= gj && 32 * g < N) acc[g] = fma(y, v[g], acc[g]);
        }
#pragma unroll
        for (int g = 0; g < BC_NG; ++g)
            if (g >= gj && 32 * g < N) sm.red[warp * NMAX + 32 * g + lane] = acc[g];
        const int owner = j & (BC_CS - 1), lj = j / BC_CS;
        const int par = bc_exchange(sm, st, j, N - j, owner, lj, ld);
        // the sums over the CTAs, a lane per column; the scalars in column j's warp alone
        // (in all four they were as many FP64 instructions as half a pass)
        const bool live = tid < N && tid >= j;
        double sum = 0.0, row = 0.0;
        if (live) {
            sum = (sm.recv[par][0][tid] + sm.recv[par][1][tid]) + (sm.recv[par][2][tid] + sm.recv[par][3][tid]);
            row = sm.rowj[par][tid];
        }
        if (warp == gj) {
            const double tail = __shfl_sync(0xffffffffu, sum, j & 31), alpha = __shfl_sync(0xffffffffu, row, j & 31);
            double beta = alpha, amb = 0.0, d = 0.0;
            if ((__double2hiint(tail) << 1 | __double2loint(tail)) != 0) {   // tail != 0
                double nx, e;
                reflector_scalars(fma(alpha, alpha, tail), fabs(alpha), &nx, &e);
                beta = __double2hiint(alpha) < 0 ? nx : -nx;
                amb = alpha - beta;
                d = -e;   // 1 / (beta amb)
            }
            if (lane == 0) {
                sm.amb[j] = amb;
                sm.d[j] = d;
                sm.beta[j] = beta;
                if (owner == st.rank) sm.S[lj * ld + j] = beta;
            }
        }
        __syncthreads();
        if (live) sm.gs[tid] = tid > j ? sm.d[j] * fma(sm.amb[j], row, sum) : 0.0;
        __syncthreads();
#pragma unroll
        for (int g = 0; g < BC_NG; ++g) gq[g] = sm.gs[32 * g + lane];
    }
}

// Q in place of the reflectors (backward accumulation), S zero above the diagonal on
// entry: afterwards S[0:M, 0:N] is the thin Q before its sign normalisation.
__device__ void bc_form_q(BcSmem& sm, BcState& st, int M, int N) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, ld = N + 1;
    const int L = (M - st.rank + BC_CS - 1) / BC_CS;
    if (tid < NMAX) sm.gs[tid] = tid == N - 1 ? sm.d[N - 1] * sm.amb[N - 1] : 0.0;
    __syncthreads();
    for (int j = N - 1; j >= 0; --j) {
        // S[i, q] += xt_i h_q for q > j and column j = e_j + xt h_j, and the dots of
        // reflector j - 1 with the columns from j on
        double hq[BC_NG], acc[BC_NG];
        const int gj = j >> 5;
#pragma unroll
        for (int g = 0; g < BC_NG; ++g) {
            hq[g] = sm.gs[32 * g + lane];
            acc[g] = 0.0;
        }
        const double ambj = sm.amb[j];
        int li = j <= st.rank ? 0 : (j - st.rank + BC_CS - 1) / BC_CS;
        li += (warp - li) & (BC_W - 1);
        for (; li < L; li += BC_W) {
            const int i = BC_CS * li + st.rank;
            double* row = sm.S + li * ld;
            const double x = i == j ? ambj : row[j];
            const double y = j ? row[j - 1] : 0.0;
            __syncwarp();   // column j is read by every lane before its lane rewrites it
#pragma unroll
            for (int g = 0; g < BC_NG; ++g) {
                if (g < gj || 32 * g >= N) continue;   // warp-uniform
                const int q = 32 * g + lane;
                if (q >= j && q < N) {
                    const double v = fma(x, hq[g], q == j ? (i == j ? 1.0 : 0.0) : row[q]);
                    row[q] = v;
                    acc[g] = fma(y, v, acc[g]);
                }
            }
        }
        if (j == 0) break;
#pragma unroll
        for (int g = 0; g < BC_NG; ++g)
            if (g >= gj && 32 * g < N) sm.red[warp * NMAX + 32 * g + lane] = acc[g];
        const int par = bc_exchange(sm, st, j, N - j, -1, 0, ld);
        if (tid < NMAX) {
            const double d = sm.d[j - 1];
            double h = 0.0;
            if (tid >= j && tid < N)
                h = d * ((sm.recv[par][0][tid] + sm.recv[par][1][tid]) + (sm.recv[par][2][tid] + sm.recv[par][3][tid]));
            else if (tid == j - 1) h = d * sm.amb[j - 1];
            sm.gs[tid] = h;
        }
        __syncthreads();
    }
    __syncthreads();
}

// The factored core's R (N x N at Rg, ld ldr, diag >= 0), then Q (M x N at Qg, ld ldq)
// with the matching signs.
__device__ void bc_write(BcSmem& sm, BcState& st, int M, int N, double* Rg, int ldr, double* Qg, int ldq) {
    const int tid = threadIdx.x, ld = N + 1, L = (M - st.rank + BC_CS - 1) / BC_CS;
    for (int e = tid; e < L * N; e += BC_T) {
        const int li = e / N, q = e - li * N, i = BC_CS * li + st.rank;
        if (i < N) {
            Rg[static_cast<long long>(i) * ldr + q] = q < i ? 0.0 : (sm.beta[i] < 0.0 ? -sm.S[li * ld + q] : sm.S[li * ld + q]);
        }
        if (q > i) sm.S[li * ld + q] = 0.0;
    }
    __syncthreads();
    bc_form_q(sm, st, M, N);
    for (int e = tid; e < L * N; e += BC_T) {
        const int li = e / N, q = e - li * N, i = BC_CS * li + st.rank;
        Qg[static_cast<long long>(i) * ldq + q] = sm.beta[q] < 0.0 ? -sm.S[li * ld + q] : sm.S[li * ld + q];
    }
    __syncthreads();
}

// ||R||_2 by power iteration on R^T R from the all-ones vector (one CTA).
__device__ double bc_norm(BcSmem& sm, const double* R, int N) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    double *z = sm.recv[0][0], *y = sm.recv[0][1], *wv = sm.recv[0][2];
    double rn = 0.0;
    for (int i = tid; i < N; i += BC_T) z[i] = 1.0 / sqrt(static_cast<double>(N));
    __syncthreads();
    for (int it = 0; it < DIAG_ITERS_B; ++it) {
        for (int i = warp; i < N; i += BC_W) {   // y = R z: a warp per row, lanes over its columns
            double a = 0.0;
            for (int jj = i + lane; jj < N; jj += 32) a = fma(R[i * N + jj], z[jj], a);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if (lane == 0) y[i] = a;
        }
        __syncthreads();
        // w = R^T y: every column split into BC_T / N row parts, partials combined
        const int parts = min(BC_T / N, BC_W), jj = tid % N, part = tid / N;
        if (part < parts) {
            double a = 0.0;
            for (int i = part; i <= jj; i += parts) a = fma(R[i * N + jj], y[i], a);
            sm.red[part * NMAX + jj] = a;
        }
        __syncthreads();
        double ss = 0.0;
        for (int c = tid; c < N; c += BC_T) {
            double a = 0.0;
            for (int q = 0; q < parts; ++q) a += sm.red[q * NMAX + c];
            wv[c] = a;
            ss = fma(a, a, ss);
        }
        const double nw = sqrt(block_sum<BC_T>(ss, sm.red));
        if (nw == 0.0 || !isfinite(nw)) return nw;
        rn = sqrt(nw);
        const double inv = 1.0 / nw;
        for (int i = tid; i < N; i += BC_T) z[i] = wv[i] * inv;
        __syncthreads();
    }
    return rn;
}

// The power-method estimate of ||R^{-1}||_2 (one CTA; no zero pivot).
__device__ double bc_inverse_norm(BcSmem& sm, const double* R, int N) {
    const int tid = threadIdx.x;
    double* z = sm.recv[0][0];
    double est = 0.0;
    for (int i = tid; i < N; i += BC_T) z[i] = 1.0 / sqrt(static_cast<double>(N));
    __syncthreads();
    for (int it = 0; it < DIAG_ITERS_B; ++it) {
        smem_tri_solve<BC_T>(R, N, N, z, 1, sm.S);   // (S is free: Q is written)
        smem_tri_solve<BC_T>(R, N, N, z, 0, sm.S);
        double ss = 0.0;
        for (int i = tid; i < N; i += BC_T) ss = fma(z[i], z[i], ss);
        const double nw = sqrt(block_sum<BC_T>(ss, sm.red));
        if (!isfinite(nw)) return __longlong_as_double(0x7ff0000000000000LL);
        est = sqrt(nw);
        if (nw == 0.0) return est;
        const double inv = 1.0 / nw;
        for (int i = tid; i < N; i += BC_T) z[i] *= inv;
        __syncthreads();
    }
    return est;
}

__global__ void __launch_bounds__(BC_T, 3) batched_core_kernel(const ProblemDev* __restrict__ PP,
                                                              const int* __restrict__ order, double eps, int eps_rel,
                                                              int mode, int32_t* status, unsigned long long limit) {
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char bc_raw[];
    BcSmem& sm = *reinterpret_cast<BcSmem*>(bc_raw);
    const ProblemDev& p = PP[order[blockIdx.x / BC_CS]];   // largest cores first (longest-processing-time order)
    const int N = p.r, M = p.r + p.l, tid = threadIdx.x;
    BcState st{static_cast<int>(cluster.block_rank()), 0, false, limit};
    if (tid == 0) {
        for (int b = 0; b < 2; ++b)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sm_u32(&sm.bars[b])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        sm.k = N;
    }
    // own rows of C = sum of the three slice products, promoted to FP64
    {
        const int L = (M - st.rank + BC_CS - 1) / BC_CS;
        for (int e = tid; e < L * N; e += BC_T) {
            const int li = e / N, j = e - li * N;
            const long long o = static_cast<long long>(BC_CS * li + st.rank) * N + j;
            sm.S[li * (N + 1) + j] = static_cast<double>(p.cpart[0][o]) + static_cast<double>(p.cpart[1][o]) +
                                     static_cast<double>(p.cpart[2][o]);
        }
    }
    __syncthreads();
    cluster.sync();   // every CTA's mbarriers are ready
    bc_qr(sm, st, M, N);
    bc_write(sm, st, M, N, p.R, N, p.Q, N);

    // ---- Section 5.1.2 / 5.1.1 diagnostics (mode SGN / AUTO)
    int k = N, sgn = 0;
    double est = 0.0, rn = 0.0;
    if (mode != GN_MODE_PLAIN) {
        cluster.sync();   // every CTA's rows of R are written
        int zero = 0;
        for (int i = tid; i < N; i += BC_T)
            if (sm.beta[i] == 0.0) zero = 1;
        zero = __syncthreads_or(zero);
        if (st.rank == 0) {
            est = zero ? __longlong_as_double(0x7ff0000000000000LL) : bc_inverse_norm(sm, p.R, N);
            if (tid == 0) sm.est = est;
        } else if (st.rank == 1 && eps_rel) {
            rn = bc_norm(sm, p.R, N);
            if (tid == 0) sm.rn = rn;
        }
        cluster.sync();
        est = *cluster.map_shared_rank(&sm.est, 0);
        if (eps_rel) {
            rn = *cluster.map_shared_rank(&sm.rn, 1);
            eps = eps * rn;
        }
        // truncation rank: first |R_ii| <= eps
        for (int i = tid; i < N; i += BC_T)
            if (fabs(sm.beta[i]) <= eps) atomicMin(&sm.k, i);
        __syncthreads();
        sgn = (mode == GN_MODE_SGN) || (eps > 0.0 && est * eps >= 100.0);
        if (sgn) k = sm.k;
    }
    if (st.rank == 0 && tid == 0) {
        *p.k = k;
        *p.sgn = sgn;
        p.diag[0] = est;
        p.diag[1] = rn;
        p.diag[2] = eps;
    }
    if (sgn && k > 0 && k < N) {   // (the same in every CTA)
        // second QR: R_1^T (N x k) = Q2 R2
        const int L = (N - st.rank + BC_CS - 1) / BC_CS;
        __syncthreads();
        for (int e = tid; e < L * k; e += BC_T) {
            const int li = e / k, j = e - li * k;   // (R_1^T)[i][j] = R[j][i]
            sm.S[li * (k + 1) + j] = p.R[static_cast<long long>(j) * N + BC_CS * li + st.rank];
        }
        cluster.sync();   // no peer still reads est, rn or its vectors in recv
        bc_qr(sm, st, N, k);
        bc_write(sm, st, N, k, p.R2, N, p.Q2, N);
    }
    if (st.dead && (tid & 31) == 0) {
        if (atomicCAS(&status[GN_DEV_STATUS], 0, GN_ERR_TIMEOUT) == 0) status[GN_DEV_WHERE] = 31;
    }
    cluster.sync();   // no CTA leaves while a peer may still push to it or read it
}

size_t core_smem_bytes() { return sizeof(BcSmem); }

// Clusters while the batch's work, (r + l) r^2 summed, spread over the SMs stays below
// half its largest core's: then the largest core bounds the batch.  (Measured break-even
// for r in 16 .. 128 near 350 problems, 0.57.)  Cores of r <= 48 are bound by their
// chains at any count.
bool bc_pays(double total, double largest, int r_max, int sms) {
    return r_max <= 48 || total <= 0.5 * sms * largest;
}

// ----------------------------------------------------------------------------
// 4b. the same with one CTA per problem (shared-memory Householder routines:
// gn_smem_core.cuh), for batches that fill the SMs several times over.
__global__ void __launch_bounds__(BT) batched_core_cta_kernel(const ProblemDev* __restrict__ PP, const int* __restrict__ order,
                                                         double eps, int eps_rel, int mode) {
    const ProblemDev& p = PP[order[blockIdx.x]];   // largest cores first (longest-processing-time order)
    extern __shared__ double shm[];
    const int N = p.r, M = p.r + p.l, tid = threadIdx.x;
    Smem sm;
    sm.ld = N + 1;
    sm.S = shm;
    sm.red = sm.S + static_cast<size_t>(MMAX) * (NMAX + 1);
    sm.tau = sm.red + BW * NMAX;
    sm.dsum = sm.tau + NMAX;
    sm.wv = sm.dsum + NMAX;
    sm.scal = sm.wv + NMAX;
    double* z = sm.scal + 8;          // [NMAX]
    double* sgnv = z + NMAX;          // [NMAX]
    const int ld = sm.ld;

    // C = sum of the three slice products, promoted to FP64
    for (int e = tid; e < M * N; e += BT) {
        const int i = e / N, j = e - i * N;
        const long long o = static_cast<long long>(i) * N + j;
        sm.S[i * ld + j] = static_cast<double>(p.cpart[0][o]) + static_cast<double>(p.cpart[1][o]) +
                           static_cast<double>(p.cpart[2][o]);
    }
    __syncthreads();
    smem_qr(sm, M, N);
    // R with diag(R) >= 0 (rows flipped), then Q in place with matching column flips
    for (int i = tid; i < N; i += BT) sgnv[i] = sm.S[i * ld + i] < 0.0 ? -1.0 : 1.0;
    __syncthreads();
    for (int e = tid; e < N * N; e += BT) {
        const int i = e / N, j = e - i * N;
        p.R[e] = j >= i ? sgnv[i] * sm.S[i * ld + j] : 0.0;
    }
    __syncthreads();
    smem_form_q(sm, M, N);
    for (int e = tid; e < M * N; e += BT) {
        const int i = e / N, j = e - i * N;
        p.Q[e] = sgnv[j] * sm.S[i * ld + j];
    }
    __threadfence_block();
    __syncthreads();

    // ---- Section 5.1.2 / 5.1.1 diagnostics (mode SGN / AUTO)
    int k = N, sgn = 0;
    double est = 0.0, rn = 0.0;
    if (mode != GN_MODE_PLAIN) {
        const double inv = 1.0 / sqrt(static_cast<double>(N));
        if (eps_rel) {   // ||R||_2 by power iteration on R^T R
            for (int i = tid; i < N; i += BT) z[i] = inv;
            __syncthreads();
            for (int it = 0; it < DIAG_ITERS_B; ++it) {
                double* y = sm.dsum;
                // y = R z: a warp per row, lanes over its columns
                const int warp = tid >> 5, lane = tid & 31;
                for (int i = warp; i < N; i += BW) {
                    double a = 0.0;
                    for (int jj = i + lane; jj < N; jj += 32) a = fma(p.R[i * N + jj], z[jj], a);
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
                    if (lane == 0) y[i] = a;
                }
                __syncthreads();
                // w = R^T y: every column split into BT / N row parts, partials combined
                const int parts = min(BT / N, BW);   // sm.red holds BW rows of NMAX
                {
                    const int jj = tid % N, part = tid / N;
                    double a = 0.0;
                    if (part < parts)
                        for (int i = part; i <= jj; i += parts) a = fma(p.R[i * N + jj], y[i], a);
                    if (part < parts) sm.red[part * NMAX + jj] = a;
                }
                __syncthreads();
                double ss = 0.0;
                for (int jj = tid; jj < N; jj += BT) {
                    double a = 0.0;
                    for (int part = 0; part < parts; ++part) a += sm.red[part * NMAX + jj];
                    sm.wv[jj] = a;
                    ss = fma(a, a, ss);
                }
                const double nw = sqrt(block_sum(ss, sm.red));
                if (nw == 0.0 || !isfinite(nw)) {
                    rn = nw;
                    break;
                }
                rn = sqrt(nw);
                for (int i = tid; i < N; i += BT) z[i] = sm.wv[i] / nw;
                __syncthreads();
            }
            eps = eps * rn;
        }
        // truncation rank: first |R_ii| <= eps
        int kl = N, zero = 0;
        for (int i = tid; i < N; i += BT) {
            const double d = p.R[i * N + i];
            if (fabs(d) <= eps) kl = min(kl, i);
            if (d == 0.0) zero = 1;
        }
        __shared__ int s_k;
        if (tid == 0) s_k = N;
        __syncthreads();
        atomicMin(&s_k, kl);
        zero = __syncthreads_or(zero);
        const int kt = s_k;
        if (zero) {
            est = __longlong_as_double(0x7ff0000000000000LL);
        } else {
            for (int i = tid; i < N; i += BT) z[i] = inv;
            __syncthreads();
            for (int it = 0; it < DIAG_ITERS_B; ++it) {
                smem_tri_solve(p.R, N, N, z, 1, sm.red);
                smem_tri_solve(p.R, N, N, z, 0, sm.red);
                double ss = 0.0;
                for (int i = tid; i < N; i += BT) ss = fma(z[i], z[i], ss);
                const double nw = sqrt(block_sum(ss, sm.red));
                if (!isfinite(nw)) {
                    est = __longlong_as_double(0x7ff0000000000000LL);
                    break;
                }
                est = sqrt(nw);
                if (nw == 0.0) break;
                for (int i = tid; i < N; i += BT) z[i] /= nw;
                __syncthreads();
            }
        }
        sgn = (mode == GN_MODE_SGN) || (eps > 0.0 && est * eps >= 100.0);
        if (sgn) k = kt;
    }
    if (tid == 0) {
        *p.k = k;
        *p.sgn = sgn;
        p.diag[0] = est;
        p.diag[1] = rn;
        p.diag[2] = eps;
    }
    if (sgn && k > 0 && k < N) {
        // second QR: R_1^T (N x k) = Q2 R2
        __syncthreads();
        sm.ld = k + 1;
        const int ld2 = sm.ld;
        for (int e = tid; e < N * k; e += BT) {
            const int i = e / k, j = e - i * k;   // (R_1^T)[i][j] = R[j][i]
            sm.S[i * ld2 + j] = p.R[j * N + i];
        }
        __syncthreads();
        smem_qr(sm, N, k);
        for (int i = tid; i < k; i += BT) sgnv[i] = sm.S[i * ld2 + i] < 0.0 ? -1.0 : 1.0;
        __syncthreads();
        for (int e = tid; e < k * k; e += BT) {
            const int i = e / k, j = e - i * k;
            p.R2[i * N + j] = j >= i ? sgnv[i] * sm.S[i * ld2 + j] : 0.0;
        }
        __syncthreads();
        smem_form_q(sm, N, k);
        for (int e = tid; e < N * k; e += BT) {
            const int i = e / k, j = e - i * k;
            p.Q2[i * N + j] = sgnv[j] * sm.S[i * ld2 + j];
        }
    }
}

size_t core_cta_smem_bytes() {
    return sizeof(double) * (static_cast<size_t>(MMAX) * (NMAX + 1) + BW * NMAX + 3 * NMAX + 8 + 2 * NMAX);
}

// Layout of the prepared tables at the start of the workspace.
struct Layout {
    size_t maps, sk_gemms, c_gemms, probs, scratch, total;
    int n_maps, sk_tiles, c_tiles;
};

}  // namespace
}  // namespace gn

using namespace gn;

extern "C" {

gn_status gn_batched_workspace_size(int32_t count, const gn_problem* probs, size_t* bytes) {
    if (count <= 0 || !probs || !bytes) return GN_ERR_INVALID_ARG;
    size_t b = 4096;
    b += al(sizeof(CUtensorMap) * 7 * count);
    b += al(sizeof(TcGemm) * 2 * count) + al(sizeof(TcGemm) * 3 * count) + al(sizeof(ProblemDev) * count);
    b += al(sizeof(int) * count);
    for (int i = 0; i < count; ++i) {
        const long long n = probs[i].A.cols, r = probs[i].X.cols, rl = probs[i].Y.cols;
        b += 3 * al(sizeof(__nv_bfloat16) * rl * r8(n)) + 3 * al(sizeof(float) * rl * r) + al(8 * 4);
    }
    *bytes = b;
    return GN_OK;
}

gn_status gn_batched_prepare(gn_handle h, int32_t count, const gn_problem* probs, void* ws, size_t ws_bytes) {
    if (!h || count <= 0 || !probs || !ws) return GN_ERR_INVALID_ARG;
    size_t need = 0;
    GN_TRY(gn_batched_workspace_size(count, probs, &need));
    if (ws_bytes < need) return GN_ERR_WORKSPACE;
    char* base = static_cast<char*>(ws);
    size_t off = 256;   // header: counts
    const size_t o_maps = off;
    off += al(sizeof(CUtensorMap) * 7 * count);
    const size_t o_sk = off;
    off += al(sizeof(TcGemm) * 2 * count);
    const size_t o_c = off;
    off += al(sizeof(TcGemm) * 3 * count);
    const size_t o_p = off;
    off += al(sizeof(ProblemDev) * count);
    const size_t o_ord = off;
    off += al(sizeof(int) * count);

    std::vector<CUtensorMap> maps(7 * static_cast<size_t>(count));
    std::vector<TcGemm> sk(2 * static_cast<size_t>(count)), cg(3 * static_cast<size_t>(count));
    std::vector<ProblemDev> pd(count);
    int sk_tiles = 0, c_tiles = 0;
    const int policy = h->batched_policy;
    const int sk_mt = (policy & 16) ? 2 : 1;
    const int bn_yta = (policy & 3) == 1 ? 64 : ((policy & 3) == 2 ? 256 : 128);
    // position of each problem's two sketch GEMMs in the tile list
    std::vector<int> slot(count);
    {
        std::vector<int> ord(count);
        for (int i = 0; i < count; ++i) ord[i] = i;
        if (policy & 8) {
            std::stable_sort(ord.begin(), ord.end(), [&](int a, int b2) {
                const auto w = [&](int i) {
                    return double(probs[i].A.rows) * probs[i].A.cols * (2.0 * probs[i].X.cols + probs[i].Y.cols);
                };
                return w(a) > w(b2);
            });
        }
        for (int pos = 0; pos < count; ++pos) slot[ord[pos]] = pos;
    }
    for (int i = 0; i < count; ++i) {
        const gn_problem& q = probs[i];
        const long long m = q.A.rows, n = q.A.cols, r = q.X.cols, rl = q.Y.cols, l = rl - r;
        if (m <= 0 || n <= 0 || r < 1 || l < 1 || r > std::min(m, n) || rl > m) return GN_ERR_SHAPE;
        if (r > NMAX || rl > MMAX) return GN_ERR_UNSUPPORTED;   // the core must fit in shared memory
        if (q.X.rows != n || q.Y.rows != m || q.AX.rows != m || q.AX.cols != r || q.YtA.rows != rl ||
            q.YtA.cols != n)
            return GN_ERR_SHAPE;
        if (q.A.dtype != GN_BF16 || q.X.dtype != GN_BF16 || q.Y.dtype != GN_BF16 || q.AX.dtype != GN_F32 ||
            q.YtA.dtype != GN_F32)
            return GN_ERR_DTYPE;
        if (!q.A.data || !q.X.data || !q.Y.data || !q.AX.data || !q.YtA.data || !q.Q || !q.R || !q.Q2 ||
            !q.R2 || !q.k)
            return GN_ERR_INVALID_ARG;
        for (const gn_mat* mm : {&q.A, &q.X, &q.Y})
            if ((reinterpret_cast<uintptr_t>(mm->data) & 15) || mm->ld % 8) return GN_ERR_ALIGNMENT;
        CUtensorMap* mp = &maps[7 * static_cast<size_t>(i)];
        GN_TRY(tc_make_map_bf16(&mp[0], q.A.data, m, n, q.A.ld, 64, 128));
        GN_TRY(tc_make_map_bf16(&mp[1], q.A.data, m, n, q.A.ld, 64, 64));
        GN_TRY(tc_make_map_bf16(&mp[2], q.X.data, n, r, q.X.ld, 64, 64));
        GN_TRY(tc_make_map_bf16(&mp[3], q.Y.data, m, rl, q.Y.ld, 64, 64));
        // per-problem scratch
        ProblemDev& d = pd[i];
        d.m = static_cast<int>(m);
        d.n = static_cast<int>(n);
        d.r = static_cast<int>(r);
        d.l = static_cast<int>(l);
        d.YtA = static_cast<const float*>(q.YtA.data);
        d.ld_yta = q.YtA.ld;
        d.lds = r8(n);
        for (int s = 0; s < 3; ++s) {
            d.s[s] = reinterpret_cast<__nv_bfloat16*>(base + off);
            off += al(sizeof(__nv_bfloat16) * rl * d.lds);
        }
        for (int s = 0; s < 3; ++s) {
            d.cpart[s] = reinterpret_cast<float*>(base + off);
            off += al(sizeof(float) * rl * r);
        }
        d.diag = reinterpret_cast<double*>(base + off);
        d.sgn = reinterpret_cast<int*>(base + off + 24);
        off += al(8 * 4);
        d.Q = q.Q;
        d.R = q.R;
        d.Q2 = q.Q2;
        d.R2 = q.R2;
        d.k = q.k;
        for (int s = 0; s < 3; ++s) GN_TRY(tc_make_map_bf16(&mp[4 + s], d.s[s], rl, n, d.lds, 64, 128));
        // sketch GEMMs: AX (A K-major, X MN-major), Y^T A (Y MN-major, A MN-major)
        const int mi = 7 * i;
        TcGemm& g0 = sk[2 * slot[i]];
        memset(&g0, 0, sizeof(g0));
        g0.M = static_cast<int>(m);
        g0.N = static_cast<int>(r);
        g0.K = static_cast<int>(n);
        g0.bn = (policy & 4) && r > 64 ? 64 : static_cast<int>(std::min<long long>(256, (r + 63) / 64 * 64));
        g0.b_mn = 1;
        g0.nsrc = 1;
        g0.map_base = mi;
        g0.a_map[0] = 0;
        g0.b_map[0] = 2;
        g0.D = static_cast<float*>(q.AX.data);
        g0.ldd = q.AX.ld;
        TcGemm& g1 = sk[2 * slot[i] + 1];
        memset(&g1, 0, sizeof(g1));
        g1.M = static_cast<int>(rl);
        g1.N = static_cast<int>(n);
        g1.K = static_cast<int>(m);
        g1.bn = bn_yta;
        g1.a_mn = 1;
        g1.b_mn = 1;
        g1.nsrc = 1;
        g1.map_base = mi;
        g1.a_map[0] = 3;
        g1.b_map[0] = 1;
        g1.D = static_cast<float*>(q.YtA.data);
        g1.ldd = q.YtA.ld;
        for (int s = 0; s < 3; ++s) {
            TcGemm& g = cg[3 * i + s];
            memset(&g, 0, sizeof(g));
            g.M = static_cast<int>(rl);
            g.N = static_cast<int>(r);
            g.K = static_cast<int>(n);
            g.bn = static_cast<int>(std::min<long long>(256, (r + 63) / 64 * 64));
            g.b_mn = 1;
            g.nsrc = 1;
            g.map_base = mi;
            g.a_map[0] = static_cast<signed char>(4 + s);
            g.b_map[0] = 2;
            g.D = d.cpart[s];
            g.ldd = r;
            GN_TRY(tc_prepare_gemm(&g, c_tiles));
            c_tiles += g.tiles_m * g.tiles_n;
        }
    }
    for (int pos = 0; pos < 2 * count; ++pos) {   // tile bases in list order
        GN_TRY(tc_prepare_gemm(&sk[pos], sk_tiles, sk_mt));
        sk_tiles += sk[pos].tiles_m * sk[pos].tiles_n;
    }
    if (off > ws_bytes) return GN_ERR_WORKSPACE;
    int header[4] = {count, sk_tiles, c_tiles, 0};
    GN_CUDA_TRY(cudaMemcpy(base, header, sizeof(header), cudaMemcpyHostToDevice));
    GN_CUDA_TRY(cudaMemcpy(base + o_maps, maps.data(), sizeof(CUtensorMap) * maps.size(), cudaMemcpyHostToDevice));
    GN_CUDA_TRY(cudaMemcpy(base + o_sk, sk.data(), sizeof(TcGemm) * sk.size(), cudaMemcpyHostToDevice));
    GN_CUDA_TRY(cudaMemcpy(base + o_c, cg.data(), sizeof(TcGemm) * cg.size(), cudaMemcpyHostToDevice));
    GN_CUDA_TRY(cudaMemcpy(base + o_p, pd.data(), sizeof(ProblemDev) * pd.size(), cudaMemcpyHostToDevice));
    // core kernel order: decreasing (r + l) r^2, the FP64 work of a core
    std::vector<int> order(count);
    for (int i = 0; i < count; ++i) order[i] = i;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b2) {
        const double wa = double(pd[a].r + pd[a].l) * pd[a].r * pd[a].r;
        const double wb = double(pd[b2].r + pd[b2].l) * pd[b2].r * pd[b2].r;
        return wa > wb;
    });
    GN_CUDA_TRY(cudaMemcpy(base + o_ord, order.data(), sizeof(int) * count, cudaMemcpyHostToDevice));
    double total = 0.0, largest = 0.0;
    int r_max = 0;
    for (const ProblemDev& d : pd) {
        const double w = double(d.r + d.l) * d.r * d.r;
        total += w;
        largest = std::max(largest, w);
        r_max = std::max(r_max, d.r);
    }
    h->batched_cluster = bc_pays(total, largest, r_max, h->sm_count) ? 1 : 0;
    // keep the host-side counts in the header's host mirror (the run call re-reads them)
    h->batched_count = count;
    h->batched_sk_tiles = sk_tiles;
    h->batched_mt = sk_mt;
    h->batched_sk_bn = 0;
    for (const TcGemm& g : sk) h->batched_sk_bn = std::max(h->batched_sk_bn, g.bn);
    h->batched_c_tiles = c_tiles;
    h->batched_ws = ws;
    return GN_OK;
}

gn_status gn_batched_set_policy(gn_handle h, int32_t policy) {
    if (!h || policy < 0 || policy >= 32 || (policy & 3) == 3) return GN_ERR_INVALID_ARG;
    h->batched_policy = policy;
    return GN_OK;
}

gn_status gn_batched_tune(gn_handle h, int32_t count, const gn_problem* probs, void* ws, size_t ws_bytes,
                          double eps, int32_t mode, int32_t* best, double* best_ms) {
    if (!h || !best) return GN_ERR_INVALID_ARG;
    static const int kPolicies[GN_BATCHED_POLICIES] = {0,  1,  2,  4,  5,  6,  8,  9,  10, 12, 13, 14,
                                                       16, 17, 18, 20, 21, 22, 24, 25, 26, 28, 29, 30};
    cudaEvent_t e0, e1;
    GN_CUDA_TRY(cudaEventCreate(&e0));
    if (cudaEventCreate(&e1) != cudaSuccess) {
        cudaEventDestroy(e0);
        return GN_ERR_CUDA;
    }
    int best_p = -1;
    float best_t = 0.0f;
    gn_status st = GN_OK;
    for (int c = 0; c < GN_BATCHED_POLICIES && st == GN_OK; ++c) {
        h->batched_policy = kPolicies[c];
        st = gn_batched_prepare(h, count, probs, ws, ws_bytes);
        if (st == GN_OK) st = gn_batched_run(h, eps, mode, ws, ws_bytes);   // warm-up
        if (st != GN_OK) break;
        if (cudaEventRecord(e0, h->stream) != cudaSuccess) { st = GN_ERR_CUDA; break; }
        for (int rep = 0; rep < 3 && st == GN_OK; ++rep) st = gn_batched_run(h, eps, mode, ws, ws_bytes);
        if (st != GN_OK) break;
        float ms = 0.0f;
        if (cudaEventRecord(e1, h->stream) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess ||
            cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) {
            st = GN_ERR_CUDA;
            break;
        }
        if (best_p < 0 || ms < best_t) {
            best_p = kPolicies[c];
            best_t = ms;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (st != GN_OK) return st;
    h->batched_policy = best_p;
    GN_TRY(gn_batched_prepare(h, count, probs, ws, ws_bytes));
    *best = best_p;
    if (best_ms) *best_ms = best_t / 3.0;
    return GN_OK;
}

gn_status gn_batched_run(gn_handle h, double eps, int32_t mode, void* ws, size_t ws_bytes) {
    if (!h || !ws) return GN_ERR_INVALID_ARG;
    const int eps_rel = (mode & GN_EPS_RELATIVE) ? 1 : 0;
    mode &= ~GN_EPS_RELATIVE;
    if (mode < GN_MODE_PLAIN || mode > GN_MODE_AUTO || !(eps >= 0.0)) return GN_ERR_INVALID_ARG;
    if (ws != h->batched_ws || h->batched_count <= 0) return GN_ERR_INVALID_ARG;   // prepare first
    const int count = h->batched_count;
    char* base = static_cast<char*>(ws);
    const size_t o_maps = 256;
    const size_t o_sk = o_maps + al(sizeof(CUtensorMap) * 7 * count);
    const size_t o_c = o_sk + al(sizeof(TcGemm) * 2 * count);
    const size_t o_p = o_c + al(sizeof(TcGemm) * 3 * count);
    const size_t o_ord = o_p + al(sizeof(ProblemDev) * count);
    (void)ws_bytes;
    const CUtensorMap* maps = reinterpret_cast<const CUtensorMap*>(base + o_maps);
    GN_TRY(tc_launch_grouped(h, reinterpret_cast<const TcGemm*>(base + o_sk), 2 * count, maps, h->batched_sk_tiles,
                             h->batched_mt, h->batched_sk_bn));
    const ProblemDev* pd = reinterpret_cast<const ProblemDev*>(base + o_p);
    batched_split3_kernel<<<dim3(16, count), 256, 0, h->stream>>>(pd);
    count_launch();
    GN_CUDA_TRY(cudaGetLastError());
    GN_TRY(tc_launch_grouped(h, reinterpret_cast<const TcGemm*>(base + o_c), 3 * count, maps, h->batched_c_tiles, 1, NMAX));
    if (!h->batched_cluster) {
        static bool attr_cta = false;
        if (!attr_cta) {
            GN_CUDA_TRY(cudaFuncSetAttribute(batched_core_cta_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(core_cta_smem_bytes())));
            attr_cta = true;
        }
        batched_core_cta_kernel<<<count, BT, core_cta_smem_bytes(), h->stream>>>(
            pd, reinterpret_cast<const int*>(base + o_ord), eps, eps_rel, mode);
        count_launch();
        GN_CUDA_TRY(cudaGetLastError());
        return GN_OK;
    }
    static bool attr = false;
    if (!attr) {
        GN_CUDA_TRY(cudaFuncSetAttribute(batched_core_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(core_smem_bytes())));
        attr = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(BC_CS * count));
    cfg.blockDim = dim3(BC_T);
    cfg.dynamicSmemBytes = core_smem_bytes();
    cfg.stream = h->stream;
    cudaLaunchAttribute ca[1];
    ca[0].id = cudaLaunchAttributeClusterDimension;
    ca[0].val.clusterDim.x = BC_CS;
    ca[0].val.clusterDim.y = 1;
    ca[0].val.clusterDim.z = 1;
    cfg.attrs = ca;
    cfg.numAttrs = 1;
    GN_CUDA_TRY(cudaLaunchKernelEx(&cfg, batched_core_kernel, pd, reinterpret_cast<const int*>(base + o_ord), eps,
                                   eps_rel, mode, h->dstatus, static_cast<unsigned long long>(h->wait_limit_ns)));
    count_launch();
    return GN_OK;
}

}  // extern "C"
