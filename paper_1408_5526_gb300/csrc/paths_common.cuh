// paths_common.cuh -- unit scheduling and the per-unit replication reduction shared by the
// fused path kernels.
//
// Work unit u = (replication m = u / tiles_per_m, tile = u % tiles_per_m): `tile`
// consecutive points i of replication m.  CTA c processes the contiguous unit range
// [c U / G, (c+1) U / G), so a grid of G = (SMs x resident CTAs) CTAs is balanced to
// within one unit.  Within a unit each warp accumulates its per-step payload in shared
// memory; at the end of the unit the warps' accumulators are added in double in warp
// order and written to partials[u][o].  No float atomics: the result is bit-identical
// from run to run, and independent of G where every unit ends so.  FP32 log-Euler caplets and the
// mortgage run kernel end only the last unit of a CTA's run in a replication (run_ends): their sums
// (compensated FP32, FP64) are grouped by G.  Caplets of 40 forwards, N = 65536, Sobol': a replication's
// theta in a plan of 7 and in one of 24 replications agrees to 1.7e-9 relative; mortgages, same bits.
#pragma once
#include "f32x2.cuh"
#include "rqmc_internal.h"

namespace rqmc {

__device__ __forceinline__ void unit_range(const RedParams &r, uint32_t &u0, uint32_t &u1) {
    u0 = (uint32_t)(((unsigned long long)blockIdx.x * r.units) / gridDim.x);
    u1 = (uint32_t)(((unsigned long long)(blockIdx.x + 1) * r.units) / gridDim.x);
}

// acc / cmp: [nwarps][nout] Kahan pairs (cmp unused in FP64 mode, kept zero).
template <typename T>
__device__ __forceinline__ void zero_acc(T *acc, T *cmp, int n) {
    for (int o = threadIdx.x; o < n; o += blockDim.x) {
        acc[o] = T(0);
        cmp[o] = T(0);
    }
}

template <typename T>
__device__ __forceinline__ void flush_unit(const RedParams &r, uint32_t u, T *acc, T *cmp) {
    __syncthreads();
    const int nw = blockDim.x >> 5, nout = r.nout;
    for (int o = threadIdx.x; o < nout; o += blockDim.x) {
        double s = 0.0;
        for (int w = 0; w < nw; ++w) {
            s += (double)acc[w * nout + o] - (double)cmp[w * nout + o];
            acc[w * nout + o] = T(0);
            cmp[w * nout + o] = T(0);
        }
        r.partials[(size_t)u * nout + o] = s;
    }
    __syncthreads();
}

// Kernels that accumulate over the CTA's consecutive units of one replication flush only at the
// last of them, into that unit's row; the theta kernel then reads those rows alone (launch_theta
// with the kernel's grid).  A flush costs a barrier and, per output and warp, four operations
// on the FP64 pipe (2 per SM and clock).  Done per unit, caplets of 10, 40 and 160 forwards took 6, 1.8
// and 0.4 % longer, mortgages 0.3 to 1 %.
__device__ __forceinline__ bool run_ends(const RedParams &r, uint32_t u, uint32_t u1) {
    return u + 1 == u1 || (u + 1) % r.tiles_per_m == 0;
}

// Lane 0 adds a warp total into the warp's accumulator slot o (Kahan in FP32).
template <typename T>
__device__ __forceinline__ void warp_accumulate(T v, T *acc, T *cmp, int o, int lane) {
    v = warp_sum(v);
    if (lane == 0) {
        T s = acc[o], c = cmp[o];
        kahan_add(s, c, v);
        acc[o] = s;
        cmp[o] = c;
    }
}

template <>
__device__ __forceinline__ void warp_accumulate<double>(double v, double *acc, double *, int o, int lane) {
    v = warp_sum(v);
    if (lane == 0) acc[o] += v;
}

// Asynchronous 4-byte global -> shared copies (waited for by the issuing thread only).
__device__ __forceinline__ void cp_async4(void *smem, const void *gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(sa), "l"(gmem) : "memory");
}
template <int BYTES>   // 4, 8 or 16 bytes, both addresses aligned to them
__device__ __forceinline__ void cp_async_n(void *smem, const void *gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(sa), "l"(gmem), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_cg16(void *smem, const void *gmem) {   // 16 bytes, past L1
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ float fmaT(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fmaT(double a, double b, double c) { return fma(a, b, c); }

// Normal z of dimension j for the current path.
template <typename T>
struct Draw;
template <>
struct Draw<float> {
    template <int SEQ>
    static __device__ __forceinline__ float normal(PathGen<SEQ> &pg, int j) { return ndtri32(pg.unif32(j)); }
};
template <>
struct Draw<double> {
    template <int SEQ>
    static __device__ __forceinline__ double normal(PathGen<SEQ> &pg, int j) { return ndtri64(pg.unif64(j)); }
};

// ------------------------------------------------------------------ lockstep generation
// P coordinates of one dimension at once (P paths of a thread, or P points of a stream):
// they share the dimension's constants and advance together through the digit or bit loop
// and the inverse-CDF polynomial, so each loop iteration carries P independent dependency
// chains.  Every value is bit-identical to the one-at-a-time routines.

// Halton/Rasrap: R and carry of the points lo0 + i[p] (see halton_R); sg = sigma of the dim.
template <int P>
__device__ __forceinline__ void halton_R_lockstep(const HaltonDim &h, const uint16_t *__restrict__ sg,
                                                  const uint32_t (&i)[P], uint32_t (&R)[P], uint32_t (&c)[P]) {
    uint32_t low[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        low[p] = h.lo0 + i[p];
        c[p] = low[p] >= h.pL ? 1u : 0u;
        low[p] -= c[p] ? h.pL : 0u;
        R[p] = 0u;
    }
    if (h.p == 2) {   // base 2: bit reversal, sigma the identity or the swap
        const uint32_t flip = sg[0] != 0 ? (1u << h.L) - 1u : 0u;
#pragma unroll
        for (int p = 0; p < P; ++p) R[p] = (__brev(low[p]) >> (32u - h.L)) ^ flip;
        return;
    }
    const uint32_t pb = h.p, mg = h.magic;
    for (uint32_t k = 0; k < h.L; ++k) {
#pragma unroll
        for (int p = 0; p < P; ++p) {
            uint32_t q = __umulhi(low[p], mg);
            uint32_t d = low[p] - q * pb;
            if ((int32_t)d < 0) {   // the rounded-up reciprocal overshot by one
                d += pb;
                q -= 1;
            }
            R[p] = R[p] * pb + (uint32_t)sg[d];
            low[p] = q;
        }
    }
}

// Sobol': x = shift ^ XOR of V_k over the set bits of n[p].  The construction is linear,
// x(n') = x(n) ^ (XOR of V_k over the set bits of n ^ n'): the first point runs the bit
// loop, the others (a fixed stride apart) differ from it in a few bits and cost a few XORs.
template <int P>
__device__ __forceinline__ void sobol_lockstep(const uint32_t *__restrict__ Vj, uint32_t shift,
                                               const uint32_t (&n)[P], int bits, uint32_t (&x)[P]) {
    uint32_t x0 = shift;
#pragma unroll 4
    for (int k = 0; k < bits; ++k) x0 ^= ((n[0] >> k) & 1u) ? Vj[k] : 0u;
    x[0] = x0;
#pragma unroll
    for (int p = 1; p < P; ++p) {
        uint32_t xp = x0;
        for (uint32_t d = n[p] ^ n[0]; d != 0u; d &= d - 1u) xp ^= Vj[__ffs(d) - 1];
        x[p] = xp;
    }
}

// Phi^-1 of P uniforms: the central polynomial for all of them in straight-line code, the
// tail branches only where some value needs them (about 0.3 % of the values).
template <int P>
__device__ __forceinline__ void ndtri32_lockstep(const Unif32 (&u)[P], float (&z)[P]) {
    float v[P], y[P], r[P];
    bool central = true;
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const float q = u[p].q;
        v[p] = ndtri32_v(q);
        y[p] = fmaf(-2.0f, q, 1.0f);
        central = central && v[p] > (float)RQMC_NDTRI_V_SPLIT;
        r[p] = erfinv_central32(v[p]);
    }
    if (!central) {
#pragma unroll
        for (int p = 0; p < P; ++p)
            if (!(v[p] > (float)RQMC_NDTRI_V_SPLIT)) r[p] = erfinv_tail32(v[p]);
    }
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const float x = y[p] * r[p];
        z[p] = u[p].lower ? -x : x;
    }
}

// |Phi^-1| of the lower-half values q of 2 NP points on packed pairs, bit-identical to ndtri32: 7
// issue slots a value for the central branch instead of 13 (the coefficients are loaded once
// for all pairs).
template <int NP>
__device__ __forceinline__ void ndtri32_pairs(const f32x2 (&q)[NP], f32x2 (&x)[NP]) {
    constexpr float V[] = RQMC_NDTRI_V;
    f32x2 v[NP], r[NP];
    float least = 0.0f;   // v = log2(q (1 - q)) <= -2
#pragma unroll
    for (int h = 0; h < NP; ++h) {
        const f32x2 w = mul2(q[h], fma2(q[h], dup2(-1.0f), dup2(1.0f)));
        v[h] = pack2(lg2_approx(lo2(w)), lg2_approx(hi2(w)));
        least = fminf(least, fminf(lo2(v[h]), hi2(v[h])));
        r[h] = dup2(V[RQMC_NDTRI_DEG_C]);
    }
#pragma unroll
    for (int k = RQMC_NDTRI_DEG_C - 1; k >= 0; --k) {
        const f32x2 c = dup2(V[k]);
#pragma unroll
        for (int h = 0; h < NP; ++h) r[h] = fma2(r[h], v[h], c);
    }
    if (!(least > (float)RQMC_NDTRI_V_SPLIT)) {   // some value in a tail
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            const float a = lo2(v[h]), b = hi2(v[h]);
            r[h] = pack2(a > (float)RQMC_NDTRI_V_SPLIT ? lo2(r[h]) : erfinv_tail32(a),
                         b > (float)RQMC_NDTRI_V_SPLIT ? hi2(r[h]) : erfinv_tail32(b));
        }
    }
#pragma unroll
    for (int h = 0; h < NP; ++h) x[h] = mul2(fma2(q[h], dup2(-2.0f), dup2(1.0f)), r[h]);
}

// Normals of P points (P even) from 32-bit words: q from min(x, ~x), the sign from the top bit.
template <int P>
__device__ __forceinline__ void normals_from_u32(const uint32_t (&x)[P], f32x2 (&z)[P / 2]) {
    f32x2 q[P / 2];
#pragma unroll
    for (int h = 0; h < P / 2; ++h) {
        const uint32_t a = x[2 * h], b = x[2 * h + 1];
        q[h] = fma2(pack2((float)min(a, ~a), (float)min(b, ~b)), dup2(2.3283064365386963e-10f),
                    dup2(1.1641532182693481e-10f));
    }
    ndtri32_pairs(q, z);
#pragma unroll
    for (int h = 0; h < P / 2; ++h)
        z[h] = pack2(__uint_as_float(__float_as_uint(lo2(z[h])) ^ (~x[2 * h] & 0x80000000u)),
                     __uint_as_float(__float_as_uint(hi2(z[h])) ^ (~x[2 * h + 1] & 0x80000000u)));
}

// FP32 normals of dimension j for the P lockstep paths of a thread (the values of P calls
// of Draw<float>::normal).  Eight paths take packed pairs; for two they were slower (20 forwards, Sobol',
// N = 1024, M = 8: 26 -> 32 us per caplet plan execute).
template <int SEQ, int P>
__device__ __forceinline__ void normals32(PathGen<SEQ> (&pg)[P], int j, float (&z)[P]) {
    const GenView &v = pg[0].v;   // every path of the thread shares the replication's view
    if constexpr (SEQ == kPhilox || SEQ == kSobolDS) {
        uint32_t x[P];
        if constexpr (SEQ == kPhilox) {
#pragma unroll
            for (int p = 0; p < P; ++p) x[p] = pg[p].philox_word(j);
        } else {
            uint32_t n[P];
#pragma unroll
            for (int p = 0; p < P; ++p) n[p] = (uint32_t)pg[p].n;
            sobol_lockstep<P>(v.V + 32 * j, v.shift[j], n, v.sob_bits, x);
        }
        if constexpr (P >= 8) {
            f32x2 y[P / 2];
            normals_from_u32<P>(x, y);
#pragma unroll
            for (int p = 0; p < P; ++p) z[p] = (p & 1) ? hi2(y[p / 2]) : lo2(y[p / 2]);
        } else {
            Unif32 u[P];
#pragma unroll
            for (int p = 0; p < P; ++p) u[p] = unif32_from_u32(x[p]);
            ndtri32_lockstep<P>(u, z);
        }
    } else {
        const HaltonDim &h = v.hd[j];
        Unif32 u[P];
        uint32_t i[P], R[P], c[P];
#pragma unroll
        for (int p = 0; p < P; ++p) i[p] = pg[p].i;
        halton_R_lockstep<P>(h, v.sig + h.sig_off, i, R, c);
#pragma unroll
        for (int p = 0; p < P; ++p) u[p] = unif32_halton(h, R[p], c[p]);
        if constexpr (P >= 8) {
            f32x2 q[P / 2], y[P / 2];
#pragma unroll
            for (int k = 0; k < P / 2; ++k) q[k] = pack2(u[2 * k].q, u[2 * k + 1].q);
            ndtri32_pairs(q, y);
#pragma unroll
            for (int p = 0; p < P; ++p) {
                const float a = (p & 1) ? hi2(y[p / 2]) : lo2(y[p / 2]);
                z[p] = u[p].lower ? -a : a;
            }
        } else {
            ndtri32_lockstep<P>(u, z);
        }
    }
}

template <typename T>
__device__ __forceinline__ T fast_rcp(T x);
template <>
__device__ __forceinline__ float fast_rcp<float>(float x) { return rcp_approx(x); }
template <>
__device__ __forceinline__ double fast_rcp<double>(double x) { return 1.0 / x; }

}  // namespace rqmc
