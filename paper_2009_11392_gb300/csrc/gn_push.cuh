// Exchanges between the CTAs of a cluster by pushing values into the peers' shared
// memory (st.async, counted on the peer's mbarrier), and the scalars of a Householder
// reflector: shared by the core's panels and the batched cores.
#pragma once

#include "gn_internal.cuh"

namespace gn {
namespace pushx {

__device__ __forceinline__ uint32_t sm_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ uint32_t map_rank(uint32_t addr, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}

// A double into a CTA of the cluster, its 8 bytes counted on that CTA's mbarrier.
__device__ __forceinline__ void push(uint32_t addr, double v, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(addr),
                 "l"(__double_as_longlong(v)), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ bool try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait: false once the limit has passed (the caller then stops waiting).
__device__ __forceinline__ bool wait(uint32_t bar, uint32_t parity, unsigned long long limit) {
    for (int i = 0; i < 64; ++i)
        if (try_wait(bar, parity)) return true;
    uint64_t t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    while (true) {
        for (int i = 0; i < 64; ++i)
            if (try_wait(bar, parity)) return true;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 > limit) return false;
    }
}

// x 2^-k as a float, truncated (x >= 0 normal; 0 below the float's range), and a
// positive normal float times 2^k as a double, both by their bits: conversions and
// compares of doubles go through the FP64 unit.
__device__ __forceinline__ float scaled_float(double x, int k) {
    const int hi = __double2hiint(x);
    const int f = ((hi >> 20) & 0x7FF) - 1023 + 127 - k;
    return f <= 0 ? 0.0f : __int_as_float((f << 23) | ((hi & 0xFFFFF) << 3) | (static_cast<unsigned>(__double2loint(x)) >> 29));
}
__device__ __forceinline__ double scaled_double(float x, int k) {
    const int b = __float_as_int(x);
    return __hiloint2double(((((b >> 23) & 0xFF) - 127 + 1023 + k) << 20) | ((b >> 3) & 0xFFFFF), b << 29);
}

// nx = ||x|| = sqrt(s) and e = 1 / (s + |alpha| nx), s = ||x||^2, the two scalars of a
// reflector (beta amb = -(s + |alpha| nx)).  Every FP64 instruction of the chain is
// ~76 cycles with the four warps busy, and sqrt and a division are about 20 of them:
// from FP32 estimates (22 bits) two Newton steps for the square root (the second
// leaves the rounding of its own last operations) and one third-order step, z (1 + q
// + q^2), for the reciprocal are 9.  Outside the range where every intermediate is
// normal (and for infinities and NaN): sqrt and /.
__device__ __forceinline__ void reflector_scalars(double s, double aa, double* nx, double* e) {
    const int E = (__double2hiint(s) >> 20) - 1023;   // sign bit set: far out of range
    if (E < -900 || E > 900) {
        *nx = sqrt(s);
        *e = 1.0 / fma(aa, *nx, s);
        return;
    }
    const int k = E >> 1;
    const float m = scaled_float(s, 2 * k);   // in [1, 4)
    float y, z;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(m));
    const float h = m * y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(z) : "f"(fmaf(scaled_float(aa, k), h, m)));   // |alpha| <= nx
    const double hy = scaled_double(y, -k - 1), z0 = scaled_double(z, -2 * k);
    const double n0 = s * scaled_double(y, -k);
    const double n1 = fma(fma(-n0, n0, s), hy, n0);
    const double n2 = fma(fma(-n1, n1, s), hy, n1);
    const double q = fma(-fma(aa, n2, s), z0, 1.0);
    *nx = n2;
    *e = fma(z0, fma(q, q, q), z0);
}

}  // namespace pushx
}  // namespace gn
