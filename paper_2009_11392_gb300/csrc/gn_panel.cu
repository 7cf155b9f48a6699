// Householder panel factorization of the core (Algorithm 2, "Y^T A X = QR") for
// panels of up to 3072 rows: 32 columns over a cluster of 16 CTAs, the panel in
// registers, one push exchange per column.
//
// A column is a chain: dot products over the rows, their sum over the cluster, the
// reflector's scalars, the update.  On GB300 a warp's FP64 instruction takes ~64
// cycles of its sub-partition whatever its mask, so a CTA has four warps (one per
// sub-partition), a lane per column and the warp's rows in registers: per row and
// column one FMA for the update and one for the next column's dots, no shared
// memory and no barrier between them (a warp updates the rows it sums).  Lanes of
// finished columns sum x_c^T x_q, the Gram entries that T needs, in the same FMAs.
// The partial sums go straight into every peer's shared memory (st.async, counted
// on the peer's mbarrier), which takes one flight instead of a cluster barrier and
// a remote read (~3500 cycles together).
//
// With x = P[c:, c], alpha = x_0, beta = -sign(alpha) ||x||, amb = alpha - beta and
// d = 1 / (beta amb), the update is P_q += xt (d (x^T P_q - beta P_cq)) with xt = x
// below row c and xt_c = amb.  The sums run over the rows below c, so
//     x^T P_q - beta P_cq = sum_q + amb P_cq   (q > c),
//     xt_c^T xt_q         = sum_q + amb P_cq   (q < c: the Gram entry),
//     ||x||^2             = sum_c + alpha^2.
// Reflectors are normalised (v = xt / amb) once, after the last column.
//
// Per 32-column panel, against the panel in shared memory with a cluster barrier per
// column (qr_panel_cluster_kernel, which larger panels keep): 150 rows 127 -> 52 us,
// 1500 rows 152 -> 137 us.  Cycles per column at 150 / 1500 rows: push and flight 860
// / 900, sums over the ranks 630 / 650, scalars 1490 (13 FP64 instructions; 2150 with
// sqrt and a division), update 460 / 2500, dots 460 / 2340 (both at the FP64 rate:
// ~100 cycles per row of a warp with shuffles between).
#include "gn_internal.cuh"
#include "gn_push.cuh"

#include <cooperative_groups.h>

#include <algorithm>

namespace gn {
namespace {
namespace cg = cooperative_groups;
using namespace pushx;

constexpr int PN_JB = 32;         // panel columns (lanes)
constexpr int PN_WARPS = 4;
constexpr int PN_THREADS = 32 * PN_WARPS;
constexpr int PN_CS = 16;         // CTAs per cluster
constexpr int PN_MAX_RW = 48;     // rows per warp in registers

struct PanelArgs {
    double* W;
    double* V;
    double *tau, *T;
    long long ld, ldv;
    int M, j0, jb, rows_per;
    int32_t* status;
    unsigned long long limit;
};

// RW: rows per warp; warp w of rank k holds panel rows k rows_per + w + 4 i.
template <int RW>
__global__ void __launch_bounds__(PN_THREADS) qr_panel_push_kernel(const __grid_constant__ PanelArgs a) {
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = static_cast<int>(cluster.block_rank());
    __shared__ double recv[2][PN_CS][PN_JB];      // pushed by the peers: their rows' sums
    __shared__ double rowc[2][PN_JB];             // row c, pushed by its owner
    __shared__ double wsum[PN_WARPS][PN_JB];      // the warps' sums
    __shared__ double rsum[PN_WARPS][PN_JB];      // sums over four ranks
    __shared__ double gram[PN_JB][PN_JB + 1], Ts[PN_JB * PN_JB], Mt[PN_JB * PN_JB / 4];
    __shared__ double taus[PN_JB], scs[PN_JB];
    __shared__ alignas(8) unsigned long long bars[2];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int Mp = a.M - a.j0, r0 = rank * a.rows_per;
    const int nr = max(0, min(a.rows_per, Mp - r0));
    if (tid == 0) {
        for (int b = 0; b < 2; ++b)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sm_u32(&bars[b])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    double P[RW];
    int gi[RW];   // panel row of P[i]; -1: no row
#pragma unroll
    for (int i = 0; i < RW; ++i) {
        const int li = warp + PN_WARPS * i;
        gi[i] = li < nr ? r0 + li : -1;
        P[i] = li < nr && lane < a.jb ? a.W[static_cast<long long>(a.j0 + r0 + li) * a.ld + a.j0 + lane] : 0.0;
    }
    for (int e = tid; e < PN_JB * (PN_JB + 1); e += PN_THREADS) gram[e / (PN_JB + 1)][e % (PN_JB + 1)] = 0.0;
    cluster.sync();   // every CTA's mbarriers are ready

    double acc = 0.0, acc1 = 0.0;   // two partial sums: half the FMA chain
#pragma unroll
    for (int i = 0; i < RW; ++i) {
        const double x = __shfl_sync(0xffffffffu, P[i], 0);
        const double xe = gi[i] > 0 ? x : 0.0;
        if (i & 1) acc1 = fma(xe, P[i], acc1);
        else acc = fma(xe, P[i], acc);
    }
    double my_amb = 0.0, my_beta = 0.0, my_d = 0.0;   // lane c: column c's scalars (all 0: dropped)
    bool dead = false;
    for (int c = 0; c < a.jb; ++c) {
        const int par = c & 1;
        const uint32_t bar = sm_u32(&bars[par]);
        if (tid == 0 && !dead)   // (a phase that ran out is not armed again)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                         "r"((PN_CS + 1) * PN_JB * 8)
                         : "memory");
        wsum[warp][lane] = acc + acc1;
        __syncthreads();
        const double mine = (wsum[0][lane] + wsum[1][lane]) + (wsum[2][lane] + wsum[3][lane]);
#pragma unroll
        for (int q = 0; q < PN_CS / PN_WARPS; ++q) {
            const int peer = warp + PN_WARPS * q;
            push(map_rank(sm_u32(&recv[par][rank][lane]), peer), mine, map_rank(bar, peer));
        }
        const int owner = c / a.rows_per, lc = c - owner * a.rows_per;
        if (rank == owner && warp == lc % PN_WARPS) {   // this warp holds row c
            double rc = 0.0;
#pragma unroll
            for (int i = 0; i < RW; ++i)
                if (gi[i] == c) rc = P[i];
#pragma unroll 4
            for (int peer = 0; peer < PN_CS; ++peer)
                push(map_rank(sm_u32(&rowc[par][lane]), peer), rc, map_rank(bar, peer));
        }
        if (!dead && !wait(bar, (c >> 1) & 1, a.limit)) dead = true;
        rsum[warp][lane] = (recv[par][4 * warp][lane] + recv[par][4 * warp + 1][lane]) +
                           (recv[par][4 * warp + 2][lane] + recv[par][4 * warp + 3][lane]);
        const double row = rowc[par][lane];
        __syncthreads();
        // every warp takes the same decisions from the same numbers
        const double sum = (rsum[0][lane] + rsum[1][lane]) + (rsum[2][lane] + rsum[3][lane]);
        const double tail = __shfl_sync(0xffffffffu, sum, c), alpha = __shfl_sync(0xffffffffu, row, c);
        double beta = alpha, amb = 0.0, g = 0.0;
        if ((__double2hiint(tail) << 1 | __double2loint(tail)) != 0) {   // tail != 0
            double nx, e;
            reflector_scalars(fma(alpha, alpha, tail), fabs(alpha), &nx, &e);
            beta = __double2hiint(alpha) < 0 ? nx : -nx;
            amb = alpha - beta;
            const double d = -e;   // 1 / (beta amb)
            const double t = fma(amb, row, sum);
            g = lane > c ? d * t : 0.0;
            if (lane < c && warp == 0) gram[c][lane] = t;
            if (lane == c) {
                my_amb = amb;
                my_beta = beta;
                my_d = d;
            }
        }
        acc = acc1 = 0.0;
#pragma unroll
        for (int i = 0; i < RW; ++i) {
            const double x = __shfl_sync(0xffffffffu, P[i], c);
            P[i] = fma(gi[i] > c ? x : (gi[i] == c ? amb : 0.0), g, P[i]);
            if (gi[i] == c && lane == c) P[i] = beta;
        }
#pragma unroll
        for (int i = 0; i < RW; ++i) {   // (a loop of its own: shuffles keep their order, so each
                                         // would wait for the FMA before it)
            const double y = __shfl_sync(0xffffffffu, P[i], (c + 1) & 31);
            const double ye = gi[i] > c + 1 ? y : 0.0;
            if (i & 1) acc1 = fma(ye, P[i], acc1);
            else acc = fma(ye, P[i], acc);
        }
    }
    if (dead && lane == 0) {
        if (atomicCAS(&a.status[GN_DEV_STATUS], 0, GN_ERR_TIMEOUT) == 0) a.status[GN_DEV_WHERE] = 30;
    }

    const double my_tau = -my_amb * (my_amb * my_d);   // (beta - alpha) / beta
    const double my_sc = my_beta * my_d;               // 1 / amb

    // the panel back (R on and above the diagonal, v below) and the explicit reflectors
#pragma unroll
    for (int i = 0; i < RW; ++i)
        if (gi[i] >= 0 && lane < a.jb) {
            const double pv = gi[i] > lane ? P[i] * my_sc : P[i];
            const long long row = a.j0 + gi[i];
            a.W[row * a.ld + a.j0 + lane] = my_tau != 0.0 || gi[i] <= lane ? pv : P[i];
            a.V[row * a.ldv + a.j0 + lane] = gi[i] < lane ? 0.0 : gi[i] == lane ? 1.0 : my_tau != 0.0 ? pv : 0.0;
        }
    if (rank == PN_CS - 1) {   // the last rank has the fewest rows: it forms T
        if (warp == 0) {
            taus[lane] = my_tau;
            scs[lane] = my_sc;
            if (lane < a.jb) a.tau[a.j0 + lane] = my_tau;
        }
        __syncthreads();
        // Ts: the Gram in the strict lower triangle (zero for dropped reflectors and
        // padding), tau on the diagonal; T is built in the upper triangle.
        for (int e = tid; e < PN_JB * PN_JB; e += PN_THREADS) {
            const int q = e / PN_JB, q2 = e - q * PN_JB;
            Ts[e] = q2 < q ? (taus[q] == 0.0 || taus[q2] == 0.0 ? 0.0 : gram[q][q2] * (scs[q] * scs[q2]))
                           : (q2 == q ? taus[q] : 0.0);
        }
        __syncthreads();
        // T by recursive doubling: for adjacent diagonal blocks T1 (rows o..o+s) and
        // T2 (o+s..o+2s), the off-diagonal block is -T1 (V1^T V2) T2, where
        // (V1^T V2)[a][b] = g(o+s+b, o+a).  Mt holds (V1^T V2) T2 for every pair.
        for (int sz = 1; sz < PN_JB; sz <<= 1) {
            const int items = (PN_JB / (2 * sz)) * sz * sz;
            for (int e = tid; e < items; e += PN_THREADS) {
                const int pr = e / (sz * sz), rem = e - pr * sz * sz, x = rem / sz, b = rem - x * sz;
                const int o = pr * 2 * sz;
                double m = 0.0;
                for (int k = 0; k <= b; ++k)
                    m = fma(Ts[(o + sz + k) * PN_JB + o + x], Ts[(o + sz + k) * PN_JB + o + sz + b], m);
                Mt[e] = m;
            }
            __syncthreads();
            for (int e = tid; e < items; e += PN_THREADS) {
                const int pr = e / (sz * sz), rem = e - pr * sz * sz, x = rem / sz, b = rem - x * sz;
                const int o = pr * 2 * sz;
                double v = 0.0;
                for (int k = x; k < sz; ++k) v = fma(Ts[(o + x) * PN_JB + o + k], Mt[pr * sz * sz + k * sz + b], v);
                Ts[(o + x) * PN_JB + o + sz + b] = -v;
            }
            __syncthreads();
        }
        for (int e = tid; e < a.jb * a.jb; e += PN_THREADS) {
            const int x = e / a.jb, b = e - x * a.jb;
            a.T[e] = b >= x ? Ts[x * PN_JB + b] : 0.0;
        }
    }
    cluster.sync();   // no CTA leaves while a peer may still push to it
}

template <int RW>
cudaError_t launch_rw(const cudaLaunchConfig_t& cfg, const PanelArgs& a) {
    return cudaLaunchKernelEx(&cfg, qr_panel_push_kernel<RW>, a);
}

template <int RW>
bool usable_rw() {
    if (cudaFuncSetAttribute(qr_panel_push_kernel<RW>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
        return false;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(PN_CS);
    cfg.blockDim = dim3(PN_THREADS);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = PN_CS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    return cudaOccupancyMaxActiveClusters(&n, qr_panel_push_kernel<RW>, &cfg) == cudaSuccess && n >= 1;
}

}  // namespace

bool panel_push_usable(long long M) {
    static const bool ok = [] {
        const bool u = usable_rw<2>() && usable_rw<4>() && usable_rw<6>() && usable_rw<8>() && usable_rw<10>() &&
                       usable_rw<12>() && usable_rw<14>() && usable_rw<16>() && usable_rw<18>() && usable_rw<20>() &&
                       usable_rw<22>() && usable_rw<24>() && usable_rw<32>() && usable_rw<40>() && usable_rw<48>();
        cudaGetLastError();
        return u;
    }();
    return ok && M <= static_cast<long long>(PN_CS) * PN_WARPS * PN_MAX_RW;
}

gn_status launch_panel_push(gn_handle h, double* W, long long ld, long long M, long long j0, int jb, double* V,
                            long long ldv, double* tau, double* T) {
    PanelArgs a;
    a.W = W;
    a.V = V;
    a.tau = tau;
    a.T = T;
    a.ld = ld;
    a.ldv = ldv;
    a.M = static_cast<int>(M);
    a.j0 = static_cast<int>(j0);
    a.jb = jb;
    a.rows_per = static_cast<int>((M - j0 + PN_CS - 1) / PN_CS);
    a.status = h->dstatus;
    a.limit = h->wait_limit_ns;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(PN_CS);
    cfg.blockDim = dim3(PN_THREADS);
    cfg.stream = h->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = PN_CS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const int rw = (a.rows_per + PN_WARPS - 1) / PN_WARPS;
    cudaError_t e;
    if (rw <= 2) e = launch_rw<2>(cfg, a);
    else if (rw <= 4) e = launch_rw<4>(cfg, a);
    else if (rw <= 6) e = launch_rw<6>(cfg, a);
    else if (rw <= 8) e = launch_rw<8>(cfg, a);
    else if (rw <= 10) e = launch_rw<10>(cfg, a);
    else if (rw <= 12) e = launch_rw<12>(cfg, a);
    else if (rw <= 14) e = launch_rw<14>(cfg, a);
    else if (rw <= 16) e = launch_rw<16>(cfg, a);
    else if (rw <= 18) e = launch_rw<18>(cfg, a);
    else if (rw <= 20) e = launch_rw<20>(cfg, a);
    else if (rw <= 22) e = launch_rw<22>(cfg, a);
    else if (rw <= 24) e = launch_rw<24>(cfg, a);
    else if (rw <= 32) e = launch_rw<32>(cfg, a);
    else if (rw <= 40) e = launch_rw<40>(cfg, a);
    else if (rw <= PN_MAX_RW) e = launch_rw<48>(cfg, a);
    else return GN_ERR_UNSUPPORTED;
    GN_CUDA_TRY(e);
    count_launch();
    return GN_OK;
}

}  // namespace gn
