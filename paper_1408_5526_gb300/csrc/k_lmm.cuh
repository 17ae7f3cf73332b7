// k_lmm.cuh -- fused LIBOR-market-model caplet kernel (Sec. 5), instantiated per sequence
// by k_lmm_halton.cu, k_lmm_sobol.cu and k_lmm_philox.cu.
//
// One thread = one path of one replication.  Per time step t (grid t_i = T_i, h = delta):
// coordinate t of the point (Halton/Rasrap digits, Sobol', or Philox) -> Phi^-1 -> one
// log-Euler step of every alive forward under the spot measure,
//     log L_n += sigma_n (h mu'_n + sqrt(h) Z) - sigma_n^2 h / 2,
//     mu'_n = sum_{j=eta}^{n} sigma_j delta L_j / (1 + delta L_j)   (a running prefix),
// then L_{t+1}(T_{t+1}) is fixed, the spot numeraire is advanced by (1 + delta L_{t+1}) and
// the caplet payoffs delta (L_{t+1} - K)^+ / prod_{j<=t+1}(1 + delta L_j(T_j)) are staged
// for the warp reduction.
//
// This file: FP64 (both schemes) and the FP32 Euler scheme; FP32 log-Euler paths are k_lmm32.cuh's.
//
// Layout: the forwards live in registers as X_n = log(delta L_n) (Euler: X_n = delta L_n).  Within
// a step the drift is carried as W_n = h mu'_n + sqrt(h) Z: a = 1 / (1 + e^-X), W += (h sigma_n) a,
// X += sigma_n W + cc_n.  Forward n sits in slot n-1 of an NF-slot array (NF = 16/40/80/160).
// Steps run in blocks of 8; after each block the array shifts down by 8 slots, so at step tp of a
// block the alive slots are tp..7 of group 0 (entered through an 8-way fall-through switch) plus
// whole groups of 8 that a uniform test skips once they are dead.  The code holds NF update
// bodies, not NF^2/2.  Per-forward constants (sigma_n, h sigma_n, cc_n) come from shared memory.
// Payoffs are written to a padded per-warp transpose buffer and summed once per block (lane r
// sums row r), then added to the warp's accumulator (Kahan in FP32).
#pragma once
#include "paths_common.cuh"

namespace rqmc {

template <typename T>
struct LmmMath;
// ld.shared of one forward's constants at the point of use (volatile: the compiler
// must not hoist the 2 x NF constants of a block into registers).
// Per-forward constants: x = sigma_n, y = h sigma_n (h in the state's log units), z = cc_n.
struct LmmC64 {
    double x, y, z, w;
};
template <>
struct LmmMath<float> {
    using C = float4;
    static constexpr int PAD = 36;   // row stride of the transpose buffer (conflict-free 16-byte reads)
    static __device__ __forceinline__ float expb(float x) { return ex2_approx(x); }
    static __device__ __forceinline__ float rcp(float x) { return rcp_approx(x); }
    static __device__ __forceinline__ float4 lds(const float4 *p) {
        float4 v;
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                     : "r"((unsigned)__cvta_generic_to_shared(p)));
        return v;
    }
};
template <>
struct LmmMath<double> {
    using C = LmmC64;
    static constexpr int PAD = 34;
    static __device__ __forceinline__ double expb(double x) { return exp(x); }
    static __device__ __forceinline__ double rcp(double x) { return 1.0 / x; }
    static __device__ __forceinline__ LmmC64 lds(const LmmC64 *p) {
        LmmC64 v;
        const unsigned a = (unsigned)__cvta_generic_to_shared(p);
        asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a));
        asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v.z) : "r"(a + 16));
        v.w = 0.0;
        return v;
    }
};

// The folded drift constant H = 1 / (h sigma_n); a zero (or vanishing) h sigma_n is replaced by
// 2^-40 of the same sign, whose drift term h sigma_n a_n <= 2^-40 is far below the FP32
// rounding of W, so that d' and the product of a pair of them stay finite.
__host__ __device__ __forceinline__ float lmm_fold_inv(float hs) {
    const float m = 9.094947e-13f;   // 2^-40
    return 1.0f / (fabsf(hs) < m ? copysignf(m, hs) : hs);
}

// One forward of one FP64 path: c = (sigma, h sigma, cc, 0), X the log-forward.
__device__ __forceinline__ void lmm_update(double &X, const LmmC64 c, double &W) {
    const double e = LmmMath<double>::expb(-X);
    const double a = LmmMath<double>::rcp(1.0 + e);   // delta L / (1 + delta L), old L
    W = fma(c.y, a, W);                               // drift through j = n
    X = fma(c.x, W, X) + c.z;
}

// One forward of one path under the Euler scheme (eq. L_n_discrete), X = delta L:
// a = X / (1 + X), W += h sigma a, X *= 1 + sigma W.
template <typename T>
__device__ __forceinline__ void lmm_update_euler(T &X, const typename LmmMath<T>::C c, T &W) {
    const T a = X * LmmMath<T>::rcp(T(1) + X);
    W = fmaT(c.y, a, W);
    X = fmaT(X * c.x, W, X);
}

template <typename T>
__device__ __forceinline__ T row_sum32(const T *row) {
    T s[4] = {T(0), T(0), T(0), T(0)};
#pragma unroll
    for (int c = 0; c < 32; c += 4) {
        s[0] += row[c];
        s[1] += row[c + 1];
        s[2] += row[c + 2];
        s[3] += row[c + 3];
    }
    return (s[0] + s[1]) + (s[2] + s[3]);
}

// Scalars of one LMM caplet strip as the path code uses them.
template <typename T>
struct LmmScal {
    int nf, nK;
    T disc0, hc, sqhc;
};

// Fill the constants [NF] of (sigma_n, h sigma_n, cc_n, 0) and the initial state X0 (all threads of
// the CTA; the caller synchronises).
template <int NF, typename T>
__device__ __forceinline__ void lmm_fill_constants(const LmmModel<T> &md, typename LmmMath<T>::C *cst, T *X0) {
    using CC = typename LmmMath<T>::C;
    for (int k = threadIdx.x; k < NF; k += blockDim.x) {
        cst[k] = CC{md.sig[k], md.hc * md.sig[k], md.cc[k], T(0)};
        X0[k] = md.X0[k];
    }
}

// Shared memory: [generator stage][constants][X0 x NF, K x 8][normals zsets x 8 x P x threads]
//                [transpose buffers][acc][cmp]
// zsets = 2 when the normals are loaded: the next block's are copied in while a block runs.
template <int NF, typename T, int P = 1>
__host__ __device__ __forceinline__ size_t lmm_smem_layout(const GenParams &g, int nw, int nK, int nout,
                                                           size_t *o_cst, size_t *o_x0, size_t *o_z, size_t *o_buf,
                                                           size_t *o_acc, int zsets = 1) {
    size_t off = stage_bytes(g);
    *o_cst = off;
    off = align16(off + sizeof(typename LmmMath<T>::C) * NF);
    *o_x0 = off;
    off = align16(off + sizeof(T) * (NF + kMaxStrikes));
    *o_z = off;
    off = align16(off + sizeof(T) * 8 * P * 32 * (size_t)nw * (size_t)zsets);
    *o_buf = off;
    off = align16(off + sizeof(T) * (size_t)nw * 8 * nK * LmmMath<T>::PAD);
    *o_acc = off;
    off += 2 * sizeof(T) * (size_t)nw * nout;
    return off;
}

// Strips of at least this many forward slots keep the step loop of a block rolled.
#ifndef RQMC_LMM_ROLL_MIN_NF
#define RQMC_LMM_ROLL_MIN_NF 80
#endif

// CTAs per SM to plan registers for: forwards take NF (FP32) or 2 NF (FP64) registers.
#ifndef RQMC_LMM_EXTRA_REGS
#define RQMC_LMM_EXTRA_REGS 44
#endif
template <int NF, typename T>
constexpr int lmm_ilp();
template <int NF, typename T>
constexpr int lmm_min_blocks() {
    constexpr int regs = (int)(NF * sizeof(T) / 4) * lmm_ilp<NF, T>() + RQMC_LMM_EXTRA_REGS;
    return regs <= 64 ? 4 : regs <= 85 ? 3 : regs <= 128 ? 2 : 1;
}

// P paths in lockstep: forwards in registers, per-step payoffs (summed over the P paths) into
// the warp's transpose buffer, block sums into the warp's accumulators (wacc/wcmp, indexed by
// output t nK + k).  The P paths share every constant load and all control flow, and give each
// warp P independent dependency chains.
// ZG (FP32): the normals are not generated here but read from zg, normals [step][zN] written
// beforehand by the point-stream kernel: path i takes zg[t zN + i], copied into the thread's
// shared columns a block ahead.
// Ks holds delta K, the payoff is (delta L - delta K)^+ D.
template <int NF, int SEQ, typename T, int P, bool EU, bool ZG>
__device__ __forceinline__ void lmm_path(PathGen<SEQ> (&pg)[P], const bool (&active)[P], const LmmScal<T> &sc,
                                         const typename LmmMath<T>::C *cst, const T *X0, const T *Ks, T *zb,
                                         T *wbuf, T *wacc, T *wcmp, const int lane, const T *zg, size_t zN) {
    static_assert(sizeof(T) == 8 || EU, "FP32 log-Euler paths are lmm32_path");
    using M = LmmMath<T>;
    using CC = typename M::C;
    constexpr int PAD = M::PAD;
    const int nf = sc.nf, nK = sc.nK;
    const T sqhc = sc.sqhc;
    const int zs = P * blockDim.x;   // stride of one step in the normals buffer
    T X[P][NF];
#pragma unroll
    for (int k = 0; k < NF; ++k) {
        const T x0 = X0[k];
#pragma unroll
        for (int p = 0; p < P; ++p) X[p][k] = x0;
    }
    T disc[P];
#pragma unroll
    for (int p = 0; p < P; ++p) disc[p] = sc.disc0;
    const int nblk = (nf + 7) >> 3;
    // loaded normals: block bb's go to set bb & 1 of the thread's columns by asynchronous copies
    auto zload = [&](const int bb) {
        if (bb < nblk) {
            const int nb = min(8, nf - 8 * bb);
            T *dst = zb + (bb & 1) * 8 * zs;
#pragma unroll
            for (int tp = 0; tp < 8; ++tp)
#pragma unroll
                for (int p = 0; p < P; ++p)
                    if (tp < nb)
                        cp_async4(dst + tp * zs + p * blockDim.x, zg + (size_t)(8 * bb + tp) * zN + pg[p].i);
        }
        cp_async_commit();   // an empty group past the last block keeps the wait count uniform
    };
    if constexpr (ZG) zload(0);
    for (int b = 0; b < nblk; ++b) {
        const int ngrp = (nf - 8 * b + 7) >> 3;   // groups of 8 shifted slots still alive
        const CC *cb0 = cst + 8 * b;              // constants of original slot 8b + k (row 0)
        const int nst = min(8, nf - 8 * b);
        // phase A: the block's normals (copied in during the previous block, or one short
        // generator loop)
        T *zbb = zb;
        if constexpr (ZG) {
            zload(b + 1);          // the set it overwrites was last read in block b - 1
            cp_async_wait<1>();    // block b's copies have landed
            zbb = zb + (b & 1) * 8 * zs;
        } else {
            for (int tp = 0; tp < nst; ++tp) {
                if constexpr (sizeof(T) == 4) {
                    float z[P];
                    normals32<SEQ, P>(pg, 8 * b + tp, z);
#pragma unroll
                    for (int p = 0; p < P; ++p) zb[tp * zs + p * blockDim.x] = z[p];
                } else {
#pragma unroll
                    for (int p = 0; p < P; ++p) zb[tp * zs + p * blockDim.x] = Draw<T>::normal(pg[p], 8 * b + tp);
                }
            }
        }
        // phase B: forward updates and payoffs (each thread reads back its own columns).  The
        // step loop of the wider strips stays rolled: eight copies of an 80- or 160-slot update
        // body would overflow the instruction cache.
        auto step = [&](const int tp) {
            T W[P];
#pragma unroll
            for (int p = 0; p < P; ++p) W[p] = sqhc * zbb[tp * zs + p * blockDim.x];
            // slot k of the P paths
            auto update_slot = [&](const int k, const CC c) {
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    if constexpr (EU) lmm_update_euler<T>(X[p][k], c, W[p]);
                    else lmm_update(X[p][k], c, W[p]);
                }
            };
            // group 0: alive slots tp..7, entered through a fall-through switch
            switch (tp) {
#define RQMC_G0(k)                            \
    case (k): {                               \
        const CC c = M::lds(cb0 + (k));       \
        update_slot(k, c);                    \
    }
                RQMC_G0(0) RQMC_G0(1) RQMC_G0(2) RQMC_G0(3) RQMC_G0(4) RQMC_G0(5) RQMC_G0(6) RQMC_G0(7)
#undef RQMC_G0
                default:
                    break;
            }
#pragma unroll
            for (int gi = 1; gi < NF / 8; ++gi) {
                if (gi < ngrp) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const CC c = M::lds(cb0 + 8 * gi + k);
                        update_slot(8 * gi + k, c);
                    }
                }
            }
            // L_{t+1}(T_{t+1}) = b^X / delta sits in shifted slot tp
            T Xf[P];
#pragma unroll
            for (int p = 0; p < P; ++p) Xf[p] = X[p][0];
            switch (tp) {
#define RQMC_PK(k)                                                       \
    case (k):                                                            \
        _Pragma("unroll") for (int p = 0; p < P; ++p) Xf[p] = X[p][(k)]; \
        break;
                RQMC_PK(1) RQMC_PK(2) RQMC_PK(3) RQMC_PK(4) RQMC_PK(5) RQMC_PK(6) RQMC_PK(7)
#undef RQMC_PK
                default:
                    break;
            }
            T Lf[P], dd[P];   // delta L, D
#pragma unroll
            for (int p = 0; p < P; ++p) {
                Lf[p] = EU ? Xf[p] : M::expb(Xf[p]);
                disc[p] *= M::rcp(T(1) + Lf[p]);
                dd[p] = active[p] ? disc[p] : T(0);
            }
            T *row = wbuf + (size_t)tp * nK * PAD + lane;
            for (int kk = 0; kk < nK; ++kk) {
                const T K = Ks[kk];
                T pay = T(0);
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    pay = fmaT(fmax(Lf[p] - K, T(0)), dd[p], pay);
                }
                row[kk * PAD] = pay;
            }
        };
        if constexpr (NF >= RQMC_LMM_ROLL_MIN_NF) {
#pragma unroll 1
            for (int tp = 0; tp < nst; ++tp) step(tp);
        } else {
            for (int tp = 0; tp < nst; ++tp) step(tp);
        }
        __syncwarp();
        const int nrows = nst * nK;
        for (int rw = lane; rw < nrows; rw += 32) {
            const T v = row_sum32<T>(wbuf + (size_t)rw * PAD);
            const int o = 8 * b * nK + rw;
            T s = wacc[o], c = wcmp[o];
            if constexpr (sizeof(T) == 4) kahan_add(s, c, v);
            else s += v;
            wacc[o] = s;
            wcmp[o] = c;
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k + 8 < NF; ++k) {
#pragma unroll
            for (int p = 0; p < P; ++p) X[p][k] = X[p][k + 8];
        }
    }
}

// Paths per thread in lockstep for a bucket: two where the registers allow it.
template <int NF, typename T>
constexpr int lmm_ilp() {
#ifdef RQMC_LMM_ILP
    return (NF * (int)sizeof(T) / 4) <= 40 ? RQMC_LMM_ILP : 1;
#else
    return (NF * (int)sizeof(T) / 4) <= 40 ? 2 : 1;
#endif
}

// ZG: normals read from zg ([M][nf][N], see lmm_path); g.stage is then 0 and no generator
// table is staged.
template <int NF, int SEQ, typename T, bool EU, bool ZG>
__global__ void __launch_bounds__(256, lmm_min_blocks<NF, T>()) lmm_caplet_kernel(const GenParams g, const LmmModel<T> md, const RedParams r,
                                                                            const T *__restrict__ zg) {
    using M = LmmMath<T>;
    using CC = typename M::C;
    constexpr int PAD = M::PAD;
    if (r.guard && *reinterpret_cast<volatile uint32_t *>(r.guard) == 0u) return;   // the fixed-point kernel's result stands
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nw = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nK = md.nK, nout = r.nout;
    constexpr int P = lmm_ilp<NF, T>();
    size_t o_cst, o_x0, o_z, o_buf, o_acc;
    lmm_smem_layout<NF, T, P>(g, nw, nK, nout, &o_cst, &o_x0, &o_z, &o_buf, &o_acc, ZG ? 2 : 1);
    T *zb = reinterpret_cast<T *>(smem_raw + o_z) + threadIdx.x;   // [zsets][8][P][blockDim], own columns
    CC *cst = reinterpret_cast<CC *>(smem_raw + o_cst);
    T *X0 = reinterpret_cast<T *>(smem_raw + o_x0);
    T *Ks = X0 + NF;
    T *wbuf = reinterpret_cast<T *>(smem_raw + o_buf) + (size_t)warp * 8 * nK * PAD;
    T *acc = reinterpret_cast<T *>(smem_raw + o_acc);
    T *cmp = acc + nw * nout;
    T *wacc = acc + warp * nout, *wcmp = cmp + warp * nout;
    lmm_fill_constants<NF, T>(md, cst, X0);
    if (threadIdx.x < kMaxStrikes) Ks[threadIdx.x] = md.dl * md.K[threadIdx.x];   // delta K
    zero_acc(acc, cmp, nw * nout);
    const LmmScal<T> sc{md.nf, md.nK, md.disc0, md.hc, md.sqhc};
    uint32_t u0, u1;
    unit_range(r, u0, u1);
    GenView gv;
    int staged_m = -1;
    for (uint32_t u = u0; u < u1; ++u) {
        const int m = (int)(u / r.tiles_per_m);
        const uint32_t tile = u % r.tiles_per_m;
        if (m != staged_m) {
            __syncthreads();
            if constexpr (ZG) view_tables(g, m, gv);
            else stage_tables(g, m, smem_raw, gv);
            staged_m = m;
        }
        __syncthreads();
        for (int pp = 0; pp < r.ppt; pp += P) {
            PathGen<SEQ> pg[P];
            bool active[P];
            bool any = false;
#pragma unroll
            for (int p = 0; p < P; ++p) {
                const uint32_t i = tile * r.tile + (uint32_t)((pp + p) * blockDim.x + threadIdx.x);
                active[p] = pp + p < r.ppt && i < r.N;
                any = any || active[p];
                pg[p].init(gv, active[p] ? i : 0u);
            }
            if (!__any_sync(0xffffffffu, any)) break;
            lmm_path<NF, SEQ, T, P, EU, ZG>(pg, active, sc, cst, X0, Ks, zb, wbuf, wacc, wcmp, lane,
                                            ZG ? zg + (size_t)m * md.nf * normals_ld(r.N) : nullptr, normals_ld(r.N));
        }
        flush_unit(r, u, acc, cmp);
    }
}

template <int NF, int SEQ, typename T, bool ZG = false>
static cudaError_t launch_lmm_t(const Plan &pl, const LmmModel<T> &md, cudaStream_t st, bool guarded = false) {
    auto kern = lmm_caplet_kernel<NF, SEQ, T, true, ZG>;
    if constexpr (sizeof(T) == 8)
        if (pl.scheme != RQMC_EULER) kern = lmm_caplet_kernel<NF, SEQ, T, false, ZG>;
    GenParams g = pl.gen;
    if (ZG) g.stage = 0;   // no generator table is read
    const int threads = pl.threads;
    size_t a, b, c, d, e2;
    const size_t smem = lmm_smem_layout<NF, T, lmm_ilp<NF, T>()>(g, threads / 32, md.nK, pl.red.nout, &a, &b, &c, &d,
                                                                 &e2, ZG ? 2 : 1);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    int occ = 0, dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, threads, smem);
    if (occ < 1) occ = 1;
    const unsigned grid = (unsigned)std::min<unsigned long long>(pl.red.units, (unsigned long long)occ * sms);
    RedParams red = pl.red;
    if (!guarded) red.guard = nullptr;
    kern<<<grid, threads, smem, st>>>(g, md, red, ZG ? reinterpret_cast<const T *>(pl.znorm) : nullptr);
    return cudaGetLastError();
}

}  // namespace rqmc
