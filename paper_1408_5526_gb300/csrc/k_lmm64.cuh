// k_lmm64.cuh -- FP64 log-Euler caplets in 64-bit fixed point (fx64.cuh), for plans whose paths stay in
// its range.
//
// One thread = one path.  With s_n = sigma_n sqrt(h log2 e) (as in k_lmm32.cuh) a forward's update is
//     W += s_n a(X_n),  X_n += s_n (W - s_n / 2),   X = log2(delta L), a = 1 / (1 + 2^-X),
// X in units of 2^-55, W in 2^-56, s in 2^-63, all products 64-bit high products.  The forwards
// are a shared-memory column per thread, so the code is one loop over the alive forwards (four at a
// time) for every strip length.  Only the normal, the payoffs and their sums are FP64
// operations.
//
// |X| >= 128 (forwards beyond 2^128 / delta or below its inverse) leaves the range: the kernel sets
// the plan's guard, and the FP64 floating-point kernel launched behind it, which otherwise
// returns at once, prices all paths again.  The host keeps plans away whose volatilities could
// carry W past 2^7 (fx_fits).
//
// Bound by the integer pipes (about 150 instructions an update, normals and payoffs included).  40 forwards, three strikes,
// N = 16384, M = 8, Sobol': 8.14 ms with the floating-point kernel, 0.95 ms here, error against 64 bits 1.8e-14 -> 6.9e-16 (relative 2-norm of the caplets).
#pragma once
#include <cmath>

#include "fx64.cuh"
#include "k_lmm32.cuh"

namespace rqmc {

static __device__ const uint64_t kFxExp2[1 << RQMC_EXP2_BITS] = RQMC_EXP2_T;

struct LmmFx {
    int64_t S[kMaxFwd];    // s_n in 2^-63
    int64_t X0[kMaxFwd];   // log2(delta L_n(0)) in 2^-55
};

constexpr int kFxSteps = 4;   // steps per payoff block
constexpr int kFxPad = LmmMath<double>::PAD;

__host__ __device__ __forceinline__ size_t lmm64_smem_layout(const GenParams &g, int threads, int nf, int nK, size_t *o_s,
                                                             size_t *o_x, size_t *o_buf, size_t *o_acc) {
    const int nw = threads / 32;
    size_t off = align16(stage_bytes(g));
    *o_s = off;
    off = align16(off + sizeof(int64_t) * (2 * (size_t)nf + kMaxStrikes));   // S, X0, delta K
    *o_x = off;
    off += sizeof(int64_t) * (size_t)nf * threads;
    *o_buf = off;
    off = align16(off + sizeof(double) * (size_t)nw * kFxSteps * nK * kFxPad);
    *o_acc = off;
    off += sizeof(double) * (size_t)nw * nf * nK;
    return off;
}

// U adjacent updates: the exponentials are independent, W is the chain.
template <int U>
__device__ __forceinline__ void fx_update(int64_t *x, int stride, const int64_t *S, int64_t &W, int64_t bias, uint32_t &ovf) {
    int64_t X[U], s[U], a[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
        X[k] = x[k * stride];
        s[k] = S[k];
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
        uint32_t E;
        const uint64_t g = fx_exp2(X[k], kFxExp2, E);
        const uint64_t rho = fx_rho(g, E);
        a[k] = (int64_t)((X[k] < 0 ? 0x8000000000000000ull - rho : rho) >> 1);
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
        W += fx_mulhi_s(a[k], s[k]) >> 5;
        X[k] += fx_mulhi_s(W - (s[k] >> 8), s[k]) + bias;
        const uint32_t h = (uint32_t)((uint64_t)X[k] >> 32);
        ovf |= h ^ (h << 1);   // top bit: |X| >= 128
        x[k * stride] = X[k];
    }
}

template <int SEQ>
__global__ void __launch_bounds__(128, 3) lmm_caplet64_kernel(const GenParams g, const LmmFx fx, const LmmModel<double> md,
                                                           const RedParams r) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nw = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, BD = blockDim.x;
    const int nf = md.nf, nK = md.nK, nout = r.nout;
    size_t o_s, o_x, o_buf, o_acc;
    lmm64_smem_layout(g, BD, nf, nK, &o_s, &o_x, &o_buf, &o_acc);
    int64_t *S = reinterpret_cast<int64_t *>(smem_raw + o_s), *X0 = S + nf;
    double *Ks = reinterpret_cast<double *>(X0 + nf);
    int64_t *x = reinterpret_cast<int64_t *>(smem_raw + o_x) + threadIdx.x;   // forward n at x[n BD]
    double *wbuf = reinterpret_cast<double *>(smem_raw + o_buf) + (size_t)warp * kFxSteps * nK * kFxPad;
    double *acc = reinterpret_cast<double *>(smem_raw + o_acc), *wacc = acc + warp * nout;
    for (int k = threadIdx.x; k < nf; k += BD) {
        S[k] = fx.S[k];
        X0[k] = fx.X0[k];
    }
    if (threadIdx.x < kMaxStrikes) Ks[threadIdx.x] = md.dl * md.K[threadIdx.x];   // delta K
    for (int o = threadIdx.x; o < nw * nout; o += BD) acc[o] = 0.0;
    const double zc = md.z_scale * 72057594037927936.0;   // sqrt(log2 e) 2^56
    uint32_t ovf = 0;
    uint32_t u0, u1;
    unit_range(r, u0, u1);
    GenView gv;
    int staged_m = -1;
    for (uint32_t u = u0; u < u1; ++u) {
        const int m = (int)(u / r.tiles_per_m);
        const uint32_t tile = u % r.tiles_per_m;
        if (m != staged_m) {
            __syncthreads();
            stage_tables(g, m, smem_raw, gv);
            staged_m = m;
        }
        __syncthreads();
        for (int pp = 0; pp < r.ppt; ++pp) {
            const uint32_t i = tile * r.tile + (uint32_t)(pp * BD + threadIdx.x);
            const bool active = i < r.N;
            if (!__any_sync(0xffffffffu, active)) break;
            PathGen<SEQ> pg;
            pg.init(gv, active ? i : 0u);
            for (int n = 0; n < nf; ++n) x[n * BD] = X0[n];
            double disc = active ? md.disc0 : 0.0;
            for (int t = 0; t < nf; ++t) {
                int64_t W = __double2ll_rn(Draw<double>::normal(pg, t) * zc);
                const int64_t bias = t & 1;   // the products round down: half a unit a step on average
                int n = t;
                if ((nf - t) & 1) {
                    fx_update<1>(x + n * BD, BD, S + n, W, bias, ovf);
                    ++n;
                }
                if ((nf - n) & 2) {
                    fx_update<2>(x + n * BD, BD, S + n, W, bias, ovf);
                    n += 2;
                }
                for (; n < nf; n += 4) fx_update<4>(x + n * BD, BD, S + n, W, bias, ovf);
                // the forward fixed at the end of the step: delta L and 1 / (1 + delta L)
                const int64_t Xf = x[t * BD];
                double L, inv;
                if (Xf < 0) {
                    uint32_t E;
                    const uint64_t gg = fx_exp2(Xf, kFxExp2, E);
                    L = (double)gg * __longlong_as_double((long long)(1023 - 64 - (int)E) << 52);
                    inv = (double)fx_rho(gg, E) * 0x1p-63;
                } else {
                    L = exp2((double)Xf * 0x1p-55);
                    inv = 1.0 / (1.0 + L);
                }
                disc *= inv;
                double *row = wbuf + (size_t)(t & (kFxSteps - 1)) * nK * kFxPad + lane;
                for (int kk = 0; kk < nK; ++kk) {
                    const double pay = L - Ks[kk];   // the positive part on the integer pipe
                    row[kk * kFxPad] = (__double_as_longlong(pay) < 0 ? 0.0 : pay) * disc;
                }
                if ((t & (kFxSteps - 1)) == kFxSteps - 1 || t == nf - 1) {
                    const int t0 = t & ~(kFxSteps - 1), nrows = (t - t0 + 1) * nK;
                    __syncwarp();
                    for (int rw = lane; rw < nrows; rw += 32) wacc[t0 * nK + rw] += row_sum32<double>(wbuf + (size_t)rw * kFxPad);
                    __syncwarp();
                }
            }
        }
        __syncthreads();
        for (int o = threadIdx.x; o < nout; o += BD) {
            double s = 0.0;
            for (int w = 0; w < nw; ++w) {
                s += acc[w * nout + o];
                acc[w * nout + o] = 0.0;
            }
            r.partials[(size_t)u * nout + o] = s;
        }
        __syncthreads();
    }
    if ((int32_t)ovf < 0) atomicOr(r.guard, 1u);
}

// Whether a plan's paths can be carried in fixed point: s below 1, initial forwards inside the
// range, and |W| <= sqrt(log2 e) |Z| + sum |s| < 2^7 for every normal the generators produce (below 10).
inline bool fx_fits(const LmmModel<double> &md, LmmFx &fx) {
    double sum = 0.0;
    for (int n = 0; n < md.nf; ++n) {
        const double s = md.sig[n] * md.s_scale;
        const long double x = (long double)md.X0[n] * 1.442695040888963407359924681L;
        if (!(std::fabs(s) < 0.99) || !(x > -120.0L && x < 120.0L)) return false;
        sum += std::fabs(s);
        fx.S[n] = (int64_t)std::llrint(s * 9223372036854775808.0);
        fx.X0[n] = (int64_t)(x * 36028797018963968.0L + (x < 0 ? -0.5L : 0.5L));
    }
    return sum < 100.0;
}

// Whether a plan's launch shape and paths let the fixed-point kernel run (smem: its shared memory).
inline bool lmm64_applies(const Plan &pl, LmmFx &fx, size_t &smem) {
    size_t a, b, c, d;
    smem = lmm64_smem_layout(pl.gen, pl.threads, pl.lmm64.nf, pl.lmm64.nK, &a, &b, &c, &d);
    return pl.prec == RQMC_FP64 && pl.scheme != RQMC_EULER && pl.threads <= 128 && pl.red.guard && smem <= 227 * 1024 &&
           fx_fits(pl.lmm64, fx);
}

// Launches the fixed-point kernel where it applies (*launched); the caller launches the guarded
// floating-point kernel behind it.
template <int SEQ>
static cudaError_t launch_lmm64(const Plan &pl, cudaStream_t st, bool *launched) {
    *launched = false;
    LmmFx fx;
    size_t smem;
    if (!lmm64_applies(pl, fx, smem)) return cudaSuccess;
    auto kern = lmm_caplet64_kernel<SEQ>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int occ = 0, dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, pl.threads, smem);
    if (occ < 1) occ = 1;
    const unsigned grid = (unsigned)std::min<unsigned long long>(pl.red.units, (unsigned long long)occ * sms);
    kern<<<grid, pl.threads, smem, st>>>(pl.gen, fx, pl.lmm64, pl.red);
    *launched = true;
    return cudaGetLastError();
}

// Caplet kernels that generate their normals, by precision and scheme (k_lmm_{halton,sobol,philox}.cu).
template <int SEQ>
cudaError_t launch_caplets_seq(const Plan &pl, cudaStream_t st, unsigned *rows_grid) {
    const bool f32 = pl.prec == RQMC_FP32;
    if (f32 && pl.scheme != RQMC_EULER) return launch_lmm32<SEQ, false>(pl, st, rows_grid);
    bool fixed = false;   // FP64 log-Euler: the fixed-point kernel, then the floating-point one behind its guard
    if (!f32) {
        const cudaError_t e = launch_lmm64<SEQ>(pl, st, &fixed);
        if (e != cudaSuccess) return e;
    }
    switch (pl.nf_bucket) {
        case 16: return f32 ? launch_lmm_t<16, SEQ>(pl, pl.lmm32, st) : launch_lmm_t<16, SEQ>(pl, pl.lmm64, st, fixed);
        case 40: return f32 ? launch_lmm_t<40, SEQ>(pl, pl.lmm32, st) : launch_lmm_t<40, SEQ>(pl, pl.lmm64, st, fixed);
        case 80: return f32 ? launch_lmm_t<80, SEQ>(pl, pl.lmm32, st) : launch_lmm_t<80, SEQ>(pl, pl.lmm64, st, fixed);
        case 160: return f32 ? launch_lmm_t<160, SEQ>(pl, pl.lmm32, st) : launch_lmm_t<160, SEQ>(pl, pl.lmm64, st, fixed);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace rqmc
