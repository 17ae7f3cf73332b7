// runs.cuh -- runs of 8 consecutive points in one dimension: the digit odometer of Halton/Rasrap
// (see k_points.cu for the derivation), and FP32 uniforms and normals of a run on packed pairs.
// Sobol' and Philox values, bases 2, 3 and 5, raw numerators and FP64 values are bit-identical to the
// point's own draw (PathGen); FP32 uniforms of bases p >= 7 come from another rounding of the same
// exact value (sigma / p + A, halton_run_q) and differ from it by 1 to 2 ulp.
#pragma once
#include "paths_common.cuh"

namespace rqmc {

constexpr int kRun = 8;

// sum_{k=1}^{L-1} sigma(d_k) p^(L-1-k) over the digits d_1, d_2, ... of q (least significant
// first), in Horner order.
__device__ __forceinline__ uint32_t halton_high(const HaltonDim &h, const uint16_t *__restrict__ sg, uint32_t q) {
    uint32_t r = 0;
    for (uint32_t k = 1; k < h.L; ++k) {
        uint32_t qq = __umulhi(q, h.magic);
        uint32_t d = q - qq * h.p;
        if ((int32_t)d < 0) {
            d += h.p;
            qq -= 1;
        }
        r = r * h.p + (uint32_t)sg[d];
        q = qq;
    }
    return r;
}

// halton_high of q (into *r0) and of q + 1 modulo p^(L-1) (into *r1) from one pass over the
// digits of q: the digits of q + 1 are those of q with a carry that runs through the low digits
// equal to p - 1.
__device__ __forceinline__ void halton_high2(const HaltonDim &h, const uint16_t *__restrict__ sg, uint32_t q,
                                             uint32_t *r0, uint32_t *r1) {
    uint32_t a = 0, b = 0, cy = 1;
    for (uint32_t k = 1; k < h.L; ++k) {
        uint32_t qq = __umulhi(q, h.magic);
        uint32_t d = q - qq * h.p;
        if ((int32_t)d < 0) {
            d += h.p;
            qq -= 1;
        }
        uint32_t e = d + cy;
        cy = e == h.p ? 1u : 0u;
        e = cy ? 0u : e;
        a = a * h.p + (uint32_t)sg[d];
        b = b * h.p + (uint32_t)sg[e];
        q = qq;
    }
    *r0 = a;
    *r1 = b;
}

// One Halton row's constants as scalars: the carry-dependent fields are picked with selects,
// so the row stays in registers (a HaltonDim indexed by the carry would live in local memory).
// HaltonRow32: what FP32 runs need.
struct HaltonRow32 {
    uint32_t pL, thr0, thr1;   // halton_lower(h, R, c) is R < thr_c
    float inv_pL, a0, a1, b0, b1;
    // the split R = sigma(d) p^(L-1) + R' of the FP32 runs (halton_run_q): thr_c = thi_c p^(L-1) + tlo_c
    uint32_t pLm1, thi0, tlo0, thi1, tlo1;
    float inv_p, pm1f;
    __device__ __forceinline__ explicit HaltonRow32(const HaltonDim &h)
        : pL(h.pL), thr0((h.pL >> 1) + (h.tie & 1u)), thr1((h.pL >> 1) + ((h.tie >> 1) & 1u)), inv_pL(h.inv_pL),
          a0(h.a[0]), a1(h.a[1]), b0(h.b[0]), b1(h.b[1]), pLm1(h.pL / h.p), thi0(thr0 / pLm1), tlo0(thr0 % pLm1),
          thi1(thr1 / pLm1), tlo1(thr1 % pLm1), inv_p(1.0f / (float)h.p), pm1f((float)(h.p - 1u)) {}
    // Run constants of the points with higher-digit sum R' and carry c: the point with lowest
    // digit sigma = sigma(d) has R = sigma p^(L-1) + R' and lies in the lower half exactly when
    // sigma < T (R < thr_c, R' < p^(L-1)); then u = sigma / p + A, else 1 - u with
    // 1 - u = (p - 1 - sigma) / p + B:  A = R' / p^L + a_c,  B = (p^(L-1) - 1 - R') / p^L + b_c.
    __device__ __forceinline__ void split(uint32_t Rp, uint32_t c, uint32_t &T, float &A, float &B) const {
        T = (c ? thi1 : thi0) + (Rp < (c ? tlo1 : tlo0) ? 1u : 0u);
        A = fmaf((float)Rp, inv_pL, c ? a1 : a0);
        B = fmaf((float)(pLm1 - 1u - Rp), inv_pL, c ? b1 : b0);
    }
    // the values of unif32_halton
    __device__ __forceinline__ Unif32 unif32(uint32_t R, uint32_t c) const {
        const bool lo = R < (c ? thr1 : thr0);
        const uint32_t Rs = lo ? R : pL - 1u - R;
        const float off = c ? (lo ? a1 : b1) : (lo ? a0 : b0);
        return Unif32{fmaf((float)Rs, inv_pL, off), lo};
    }
};
struct HaltonRow : HaltonRow32 {
    unsigned long long P, S0, S1;
    double invD;
    __device__ __forceinline__ explicit HaltonRow(const HaltonDim &h)
        : HaltonRow32(h), P(h.P), S0(h.S[0]), S1(h.S[1]), invD(h.invD) {}
    __device__ __forceinline__ unsigned long long num(uint32_t R, uint32_t c) const {
        return (unsigned long long)R * P + (c ? S1 : S0);
    }
    // the values of unif64_halton
    __device__ __forceinline__ Unif64 unif64(uint32_t R, uint32_t c) const {
        const unsigned long long n = num(R, c);
        const unsigned long long D1 = (unsigned long long)pL * P - 1ull;
        const bool lo = n <= D1 - n;
        return Unif64{((double)(lo ? n : D1 - n) + 0.5) * invD, lo};
    }
};

// One lane's run of kRun points (p >= 7): lowest digit d0 of its first point, the higher-digit
// sums R'(q0) and R'(q0 + 1) and the carries before and after the wrap of the lowest digit
// (R1 = R0 where no lane of the warp wraps).
struct HaltonRun {
    uint32_t d0, R0, R1, c0, c1;
    bool any_wrap;   // warp-uniform: some lane's run wraps its lowest digit
};
__device__ __forceinline__ HaltonRun halton_run(const HaltonDim &h, const uint16_t *__restrict__ sg, uint32_t i0,
                                                uint32_t pLm1) {
    HaltonRun r;
    uint32_t low = h.lo0 + i0;
    r.c0 = low >= h.pL ? 1u : 0u;
    low -= r.c0 ? h.pL : 0u;
    uint32_t q0 = __umulhi(low, h.magic);
    r.d0 = low - q0 * h.p;
    if ((int32_t)r.d0 < 0) {
        r.d0 += h.p;
        q0 -= 1;
    }
    // the run reaches p^L: the low part wraps into the carry (and q0 + 1 to 0)
    r.c1 = q0 + 1 == pLm1 ? 1u : r.c0;
    // R'(q0 + 1) only where some lane's run wraps its lowest digit: always for small p, in
    // about 256/p of the warps for p > 256
    r.any_wrap = __any_sync(0xffffffffu, r.d0 + (kRun - 1) >= h.p);
    if (r.any_wrap) {
        halton_high2(h, sg, q0, &r.R0, &r.R1);
    } else {
        r.R0 = halton_high(h, sg, q0);
        r.R1 = r.R0;
    }
    return r;
}

// The (q, side) pairs of a Halton run (p >= 7) from the split of HaltonRow::split: a point costs
// one permutation lookup (the padded table, see kSigPad), one integer compare, two selects and,
// per two points, a packed subtraction and a packed multiply-add.  low: bit k = point k is in the
// lower half.
__device__ __forceinline__ void halton_run_q(const HaltonRow32 &hr, const HaltonRun &r, const uint16_t *__restrict__ sg,
                                             uint32_t p, f32x2 (&q)[kRun / 2], bool (&low)[kRun]) {
    uint32_t T0;
    float A0, B0;
    hr.split(r.R0, r.c0, T0, A0, B0);
    const uint16_t *sb = sg + r.d0;   // sb[k] = sigma((d0 + k) mod p)
    float t[kRun], off[kRun];
    const f32x2 pm1 = dup2(hr.pm1f), mone = dup2(-1.0f), ip = dup2(hr.inv_p);
    if (!r.any_wrap) {
#pragma unroll
        for (int k = 0; k < kRun; ++k) {
            const uint32_t sk = sb[k];
            t[k] = (float)sk;
            low[k] = sk < T0;
            off[k] = low[k] ? A0 : B0;
        }
    } else {
        uint32_t T1;
        float A1, B1;
        hr.split(r.R1, r.c1, T1, A1, B1);
        const uint32_t kw = p - r.d0;   // points k >= kw are past the wrap: R'(q0 + 1), carry c1
#pragma unroll
        for (int k = 0; k < kRun; ++k) {
            const bool w = (uint32_t)k >= kw;
            const uint32_t sk = sb[k];
            t[k] = (float)sk;
            low[k] = sk < (w ? T1 : T0);
            off[k] = low[k] ? (w ? A1 : A0) : (w ? B1 : B0);
        }
    }
#pragma unroll
    for (int h = 0; h < kRun / 2; ++h) {
        const f32x2 f = pack2(t[2 * h], t[2 * h + 1]), g = fma2(f, mone, pm1);   // p - 1 - sigma, exact
        const f32x2 d = pack2(low[2 * h] ? lo2(f) : lo2(g), low[2 * h + 1] ? hi2(f) : hi2(g));
        q[h] = fma2(d, ip, pack2(off[2 * h], off[2 * h + 1]));
    }
}

}  // namespace rqmc
