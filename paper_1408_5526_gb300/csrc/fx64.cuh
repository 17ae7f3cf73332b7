// fx64.cuh -- 64-bit fixed-point exponential and logistic factor of the FP64 caplet paths.
//
// The FP64 pipe of this GPU starts two operations per SM and clock, so one FP64 forward update
// (exp, division, four more) takes it about 14 clocks per path.  The 32-bit integer pipes take a
// 64-bit high product in an eighth of a clock.  The log-forward X = log2(delta L) is therefore
// held as a signed integer in units of 2^-55 (32 times finer than a double near X = -6), and
//   t = 2^-|X|  by a table of 2^(-i/2048) and a degree-4 polynomial (Tang's method),
//   rho = 1 / (1 + t)  from the FP32 reciprocal by one second-order Newton step on integers,
// each exact to about 2^-56, give delta L / (1 + delta L) = rho (X >= 0) or 1 - rho.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "fp64_tables.h"

namespace rqmc {

constexpr int kFxBits = 55;   // fraction bits of X
constexpr int kFxWBits = 56;  // fraction bits of the drift and noise W

__host__ __device__ __forceinline__ uint64_t fx_mulhi(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
__host__ __device__ __forceinline__ int64_t fx_mulhi_s(int64_t a, int64_t b) {
#ifdef __CUDA_ARCH__
    return __mul64hi(a, b);
#else
    return (int64_t)(((__int128)a * b) >> 64);
#endif
}
__host__ __device__ __forceinline__ uint32_t fx_mulhi32(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}

// g 2^-E = 2^-|X| with g in (1/2, 1] as a 64-bit fraction.
__host__ __device__ __forceinline__ uint64_t fx_exp2(int64_t X, const uint64_t *__restrict__ T, uint32_t &E) {
    const uint64_t m = (uint64_t)(X < 0 ? -X : X);
    E = (uint32_t)(m >> kFxBits);
    const uint64_t f = m << (64 - kFxBits), v = f << RQMC_EXP2_BITS;
    const uint32_t vh = (uint32_t)(v >> 32);
    uint32_t c = RQMC_EXP2_C3 - fx_mulhi32(vh, RQMC_EXP2_C4);
    c = RQMC_EXP2_C2 - fx_mulhi32(vh, c);
    const uint64_t h = fx_mulhi(v, RQMC_EXP2_C1 - ((uint64_t)fx_mulhi32(vh, c) << 19));   // 2048 (1 - 2^(-v/2048))
#ifdef __CUDA_ARCH__
    const uint64_t t = __ldg(reinterpret_cast<const unsigned long long *>(T) + (f >> (64 - RQMC_EXP2_BITS)));
#else
    const uint64_t t = T[f >> (64 - RQMC_EXP2_BITS)];
#endif
    return t - (fx_mulhi(t, h) >> RQMC_EXP2_BITS);
}

// rho = 1 / (1 + g 2^-E) as a 63-bit fraction in [1/2, 1].
__host__ __device__ __forceinline__ uint64_t fx_rho(uint64_t g, uint32_t E) {
    const uint64_t D = 0x8000000000000000ull + ((g >> (E < 63u ? E : 63u)) >> 1);   // (1 + t) 2^63
    const uint32_t dh = (uint32_t)(D >> 32), dl = (uint32_t)D;
#ifdef __CUDA_ARCH__
    float rf;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rf) : "f"((float)dh));
    const uint32_t r0 = __float2uint_rz(rf * 9.223372036854775808e18f);   // saturates at 2^32 - 1
#else
    const double rf = (double)((1.0f / (float)dh) * 9.223372036854775808e18f);
    const uint32_t r0 = rf >= 4294967295.0 ? 0xFFFFFFFFu : (uint32_t)rf;
#endif
    // D r0 = 2^95 (1 - e), |e| < 2^-21; rho = r0 2^-32 (1 + e + e^2) + O(e^3)
    const int64_t e = (int64_t)(0x8000000000000000ull - ((uint64_t)dh * r0 + (((uint64_t)dl * r0) >> 32)));
    const int32_t eh = (int32_t)(e >> 20);
    const int64_t ee = e + (((int64_t)eh * eh) >> 23);
    return ((uint64_t)r0 << 31) + (((uint64_t)(uint32_t)ee * r0) >> 32) + (uint64_t)((int64_t)(int32_t)(ee >> 32) * (int64_t)(uint64_t)r0);
}

}  // namespace rqmc
