// k_lmm32.cuh -- FP32 log-Euler paths of the LIBOR market model (the model, the payoffs and the
// block structure of k_lmm.cuh), on packed FP32 pairs.  Used by the caplet kernels of FP32
// plans and by the strip classes of the batch.
//
// Units: s_n = sigma_n sqrt(h log2 e), so that h sigma_j sigma_n log2 e = s_j s_n, and the normal
// enters as W = sqrt(log2 e) Z.  Forward n is carried as X_n = log2(delta L_n); with W the step's
// running drift and noise through forward n its update is
//     e = 2^-X_n,  d = H_n + H_n e  (H_n = 1/s_n),  W += 1/d  (= s_n delta L/(1 + delta L)),
//     X_n += s_n (W - s_n / 2),
// and two adjacent forwards share one reciprocal, 1/d0 = d1 / (d0 d1): per forward one ex2,
// half an rcp and 4.5 FP32 operations.  Subtracting s_n / 2 from W (small numbers) and not from
// X_n keeps one rounding of X_n a step.  The two constants of a forward do not depend on the
// step; a thread's paths read them from shared memory with one 16-byte load.
//
// FLAT: all volatilities are equal.  Then s and H are two registers, W is carried with s/2
// already taken off (once per step), and an update needs neither the load nor the subtraction.
//
// Packing.  P = 2 paths per thread (or 4): each 64-bit register holds one forward of two
// paths, all operations but ex2 and rcp are packed (9 packed operations for two forwards of
// two paths).  P = 1 (the longest strips, whose forwards fill the registers): a register
// holds two adjacent forwards of the path; the two steps of the drift chain are scalar.
//
// Layout.  Forward n of a strip of nf sits in slot NF - nf + n - 1, so the alive slots of a
// step are always the last ones and no step runs over unused slots; slot k is fixed at the end
// of step k.  Steps go in sub-blocks of GR: the step code of a sub-block is compiled for its
// first slot and is one straight line, GR slots of which the dead ones are masked (their drift
// terms vanish, see below) and then every later slot.  Straight-line code is what makes the kernel
// fast: the updates' long chains (ex2, rcp) overlap only inside a basic block, and a version that
// jumped into a chain of 8-slot blocks ran at half the rate with the same instructions.  GR trades masked slots against code
// size (NF^2 / (2 GR) updates).
//
// Payoffs.  A step leaves (delta L, D) of its forward (for the batch (L, delta D), the same product) in the warp's buffer; after 8 steps each
// lane takes a row (step, strike), or a part of one, sums (delta L - delta K)^+ D over the
// warp's paths and adds the sum to the warp's Kahan accumulator.
#pragma once
#include "f32x2.cuh"
#include "k_lmm.cuh"

namespace rqmc {

struct Lmm32Scal {
    int nf, nK;
    float disc0, zscale;   // zscale = sqrt(log2 e)
    float s, H;            // FLAT: the strip's constants
    float l_scale, d_scale;   // payoff (l_scale delta L - Ks)^+ d_scale D
};

// Constants in shared memory: P >= 2, entry k = (s, s, H, H) of slot k, then one for dead slots; P = 1,
// entry q = (s, s, H, H) of slots (2q, 2q + 1); then x0[NF] = log2(delta L(0)).  Slots below NF - nf
// are never alive.
//
// A dead slot's state is not read: forwards fall without bound (2^-90 from a tiny initial value or a
// volatility of some hundred percent), and 1 + 2^-X of one that is fixed must not overflow the
// product that an alive neighbour's reciprocal comes from.  Its update reads X = -40 (FLAT and P = 1, drift
// term s 2^-40), or the entry s = 0, H = 2^40 with a state that was cleared when it was fixed (P >= 2
// with constants from memory, where selecting the state instead of the address took 40 forwards,
// N = 65536, M = 64 from 1.527 to 1.556 ms; as it is 1.535).
constexpr float kLmmDeadX = -40.0f, kLmmDeadH = 1.099511627776e12f;   // 2^40
template <int NF, int P>
__host__ __device__ constexpr size_t lmm32_const_bytes() {
    return (P == 1 ? NF / 2 : NF + 1) * sizeof(float4) + NF * sizeof(float);
}
template <int NF, int P>
__device__ __forceinline__ float *lmm32_x0(float4 *cst) {
    return reinterpret_cast<float *>(cst + (P == 1 ? NF / 2 : NF + 1));
}
template <int NF, int P>
__device__ __forceinline__ void lmm32_fill_constants(const LmmModel<float> &md, float4 *cst) {
    float *x0 = lmm32_x0<NF, P>(cst);
    const int sh = NF - md.nf;
    const float c = md.s_scale;
    for (int k = threadIdx.x; k < NF; k += blockDim.x) {
        const int n = k - sh;
        const float s = n >= 0 ? md.sig[n] * c : 0.0f, H = n >= 0 ? lmm_fold_inv(s) : 1.0f;
        x0[k] = n >= 0 ? md.X0[n] : 0.0f;
        if constexpr (P == 1) {
            float *e = reinterpret_cast<float *>(cst + (k >> 1)) + (k & 1);
            e[0] = s;
            e[2] = H;
        } else {
            cst[k] = make_float4(s, s, H, H);
        }
    }
    if (P > 1 && threadIdx.x == 0) cst[NF] = make_float4(0.0f, 0.0f, kLmmDeadH, kLmmDeadH);
}
// One entry, loaded at the point of use (volatile: the compiler must not keep a strip's
// constants in registers).
struct Lmm32C {
    f32x2 s, H;
};
__device__ __forceinline__ Lmm32C lmm32_lds(unsigned p) {
    Lmm32C v;
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(v.s), "=l"(v.H) : "r"(p));
    return v;
}

template <int K>
struct IntC {
    static constexpr int value = K;
};
template <int N, int I = 0, class F>
__device__ __forceinline__ void lmm32_for(const F &f) {   // f(0) .. f(N - 1) with constant arguments
    if constexpr (I < N) {
        f(IntC<I>{});
        lmm32_for<N, I + 1>(f);
    }
}

// Floats of a step's row in a warp's payoff buffer (8 rows): per lane (delta L, D) of its path, or per
// two paths (delta L, delta L, D, D); padded by 16 bytes against bank conflicts between rows.
template <int P>
__host__ __device__ constexpr int lmm32_row() {
    return 64 * P + 4;
}

// P paths of one thread (adjacent points): see the header.  pg supplies the normals (ZG = false)
// or only the point index: with ZG the normals are read from zg, [step][zN], point i at column
// i - zi0, copied into the thread's shared columns a block of 8 slots ahead.  The caller's paths
// past the end are dropped by a zero numeraire (active).  Ks holds the strikes, times delta where
// l_scale is 1.
template <int NF, int GR, int SEQ, int P, bool ZG, bool FLAT>
__device__ __forceinline__ void lmm32_path(PathGen<SEQ> (&pg)[P], const bool (&active)[P], const Lmm32Scal &sc,
                                           float4 *cst, const float *Ks, float *zb, float *wbuf, float *wacc,
                                           float *wcmp, const int lane, const float *zg, size_t zN, uint32_t zi0) {
    constexpr int S = P == 1 ? 1 : P / 2;   // packed path pairs
    constexpr int NY = P == 1 ? NF / 2 : NF;
    constexpr int ROW = lmm32_row<P>();
    static_assert(P == 1 || P % 2 == 0, "one path or packed pairs");
    static_assert(NF % GR == 0 && (GR % 8 == 0 || 8 % GR == 0), "whole sub-blocks");
    const int nK = sc.nK, sh = NF - sc.nf;
    const unsigned ca = (unsigned)__cvta_generic_to_shared(cst);
    const f32x2 mhalf = dup2(-0.5f), fs = dup2(sc.s), fH = dup2(sc.H);
    f32x2 X[S][NY];
    {
        const float *x0 = lmm32_x0<NF, P>(cst);
#pragma unroll
        for (int k = 0; k < NY; ++k)
#pragma unroll
            for (int s = 0; s < S; ++s) X[s][k] = P == 1 ? reinterpret_cast<const f32x2 *>(x0)[k] : dup2(x0[k]);
    }
    float disc[P];
#pragma unroll
    for (int p = 0; p < P; ++p) disc[p] = active[p] ? sc.disc0 : 0.0f;
    const int zs = P * blockDim.x;   // one step of the normals buffer; the thread's P values are adjacent
    auto zload = [&](const int bb) {   // slots 8 bb .. 8 bb + 7 (from sh on) into set bb & 1
        if (bb < NF / 8) {
            float *dst = zb + (bb & 1) * 8 * zs;
            const float *src = zg + ((ptrdiff_t)(8 * bb - sh) * (ptrdiff_t)zN + (ptrdiff_t)(pg[0].i - zi0));
#pragma unroll
            for (int tp = 0; tp < 8; ++tp)
                if (8 * bb + tp >= sh) cp_async_n<4 * P>(dst + tp * zs, src + (size_t)tp * zN);
        }
        cp_async_commit();   // an empty group past the last block keeps the wait count uniform
    };
    const int b0 = sh >> 3;
    if constexpr (ZG) zload(b0);
#pragma unroll 1
    for (int b = b0; b < NF / 8; ++b) {
        const int lo = max(8 * b, sh);   // the block's first step
        float *zbb = zb;
        if constexpr (ZG) {
            zload(b + 1);          // the set it overwrites was last read in block b - 1
            cp_async_wait<1>();    // block b's copies have landed
            zbb = zb + (b & 1) * 8 * zs;
        } else {
            for (int k = lo; k < 8 * b + 8; ++k) {
                float z[P];
                normals32<SEQ, P>(pg, k - sh, z);
#pragma unroll
                for (int p = 0; p < P; ++p) zb[(k & 7) * zs + p] = z[p];
            }
        }
        // step `slot` of the sub-block that starts at slot S0
        auto step = [&](auto SUB, const int slot) {
            constexpr int S0 = decltype(SUB)::value;
            f32x2 W[S];
            float w = 0.0f;   // P = 1
            float Xf[P];
            const float *zp = zbb + (slot & 7) * zs;
            if constexpr (P == 1) {
                w = FLAT ? fmaf(sc.zscale, zp[0], -0.5f * sc.s) : sc.zscale * zp[0];
            } else {
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    const f32x2 z = *reinterpret_cast<const f32x2 *>(zp + 2 * s);
                    W[s] = FLAT ? fma2(z, dup2(sc.zscale), dup2(-0.5f * sc.s)) : mul2(z, dup2(sc.zscale));
                }
            }
            // the state that slot k's drift term comes from
            auto state = [&](const float x, const int k, const bool masked) { return (FLAT || P == 1) && masked && slot > k ? kLmmDeadX : x; };
            // slots 2q, 2q + 1; masked: some of them may be dead
            auto pair = [&](const int q, const bool masked) {
                if constexpr (P == 1) {
                    Lmm32C c{fs, fH};
                    if constexpr (!FLAT) c = lmm32_lds(ca + 16 * q);
                    f32x2 &x = X[0][q];
                    const f32x2 e = pack2(ex2_approx(-state(lo2(x), 2 * q, masked)), ex2_approx(-state(hi2(x), 2 * q + 1, masked)));
                    const f32x2 d = fma2(e, c.H, c.H);
                    const float r = rcp_approx(lo2(d) * hi2(d));
                    const float w0 = fmaf(r, hi2(d), w);
                    w = fmaf(r, lo2(d), w0);
                    const f32x2 v = pack2(w0, w);
                    x = fma2(c.s, FLAT ? v : fma2(c.s, mhalf, v), x);
                    if (masked) {
                        if (slot == 2 * q) Xf[0] = lo2(x);
                        if (slot == 2 * q + 1) Xf[0] = hi2(x);
                    }
                } else {
                    Lmm32C c0{fs, fH}, c1{fs, fH};
                    if constexpr (!FLAT) {
                        c0 = lmm32_lds(masked && slot > 2 * q ? ca + 16 * NF : ca + 32 * q);
                        c1 = lmm32_lds(masked && slot > 2 * q + 1 ? ca + 16 * NF : ca + 32 * q + 16);
                    }
#pragma unroll
                    for (int s = 0; s < S; ++s) {
                        f32x2 &xa = X[s][(2 * q) % NY], &xb = X[s][(2 * q + 1) % NY];
                        const f32x2 e0 = pack2(ex2_approx(-state(lo2(xa), 2 * q, masked)), ex2_approx(-state(hi2(xa), 2 * q, masked)));
                        const f32x2 e1 = pack2(ex2_approx(-state(lo2(xb), 2 * q + 1, masked)), ex2_approx(-state(hi2(xb), 2 * q + 1, masked)));
                        const f32x2 d0 = fma2(e0, c0.H, c0.H), d1 = fma2(e1, c1.H, c1.H), m = mul2(d0, d1);
                        const f32x2 r = pack2(rcp_approx(lo2(m)), rcp_approx(hi2(m)));
                        W[s] = fma2(r, d1, W[s]);
                        xa = fma2(c0.s, FLAT ? W[s] : fma2(c0.s, mhalf, W[s]), xa);
                        W[s] = fma2(r, d0, W[s]);
                        xb = fma2(c1.s, FLAT ? W[s] : fma2(c1.s, mhalf, W[s]), xb);
                        if (masked) {
                            if (slot == 2 * q) {
                                Xf[2 * s] = lo2(xa);
                                Xf[(2 * s + 1) % P] = hi2(xa);
                                if constexpr (!FLAT) xa = 0ull;
                            }
                            if (slot == 2 * q + 1) {
                                Xf[2 * s] = lo2(xb);
                                Xf[(2 * s + 1) % P] = hi2(xb);
                                if constexpr (!FLAT) xb = 0ull;
                            }
                        }
                    }
                }
            };
#pragma unroll
            for (int p = 0; p < P; ++p) Xf[p] = 0.0f;
            if constexpr (GR > 8) {   // whole dead groups of 8 slots are skipped
#pragma unroll
                for (int g = 0; g < GR / 8; ++g)
                    if (slot < S0 + 8 * g + 8) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) pair(S0 / 2 + 4 * g + q, true);
                    }
            } else {
#pragma unroll
                for (int q = 0; q < GR / 2; ++q) pair(S0 / 2 + q, true);
            }
#pragma unroll
            for (int q = (S0 + GR) / 2; q < NF / 2; ++q) pair(q, false);
            float v[2 * P];   // delta L of the fixed forward and D
#pragma unroll
            for (int p = 0; p < P; ++p) {
                v[p] = ex2_approx(Xf[p]);
                disc[p] *= rcp_approx(1.0f + v[p]);
                v[p] *= sc.l_scale;
                v[P + p] = disc[p] * sc.d_scale;
            }
            float *row = wbuf + (slot & 7) * ROW + 2 * P * lane;
            if constexpr (P == 1) {
                *reinterpret_cast<float2 *>(row) = make_float2(v[0], v[1]);
            } else {
#pragma unroll
                for (int h = 0; h < P / 2; ++h)
                    reinterpret_cast<float4 *>(row)[h] = make_float4(v[2 * h], v[2 * h + 1], v[P + 2 * h], v[P + 2 * h + 1]);
            }
        };
        auto block = [&](auto B) {   // block b of 8 slots: its steps, sub-block by sub-block
            constexpr int k0 = 8 * decltype(B)::value;
            if constexpr (k0 < NF) {
                if constexpr (GR >= 8) {
#pragma unroll 1
                    for (int k = lo; k < 8 * b + 8; ++k) step(IntC<k0 / GR * GR>{}, k);
                } else {
                    lmm32_for<8 / GR>([&](auto I) {
                        constexpr int s0 = k0 + GR * decltype(I)::value;
#pragma unroll 1
                        for (int k = max(lo, s0); k < s0 + GR; ++k) step(IntC<s0>{}, k);
                    });
                }
            }
        };
        if constexpr (GR <= 8) {
            switch (b) {
#define RQMC_B(n) \
    case n: block(IntC<n>{}); break;
                RQMC_B(0) RQMC_B(1) RQMC_B(2) RQMC_B(3) RQMC_B(4) RQMC_B(5) RQMC_B(6) RQMC_B(7) RQMC_B(8) RQMC_B(9)
                RQMC_B(10) RQMC_B(11) RQMC_B(12) RQMC_B(13) RQMC_B(14) RQMC_B(15) RQMC_B(16) RQMC_B(17) RQMC_B(18)
                RQMC_B(19)
                default: break;
            }
        } else {
            switch (b / (GR / 8)) {
#define RQMC_C(n) \
    case n: block(IntC<(n) * (GR / 8)>{}); break;
                RQMC_C(0) RQMC_C(1) RQMC_C(2) RQMC_C(3) RQMC_C(4) RQMC_C(5) RQMC_C(6) RQMC_C(7) RQMC_C(8) RQMC_C(9)
                default: break;
            }
        }
#undef RQMC_B
#undef RQMC_C
        __syncwarp();
        // rows (step, strike): `lpr` lanes share a row, each takes every lpr-th lane's paths
        const int k0 = lo & 7, nrows = (8 - k0) * nK;
        const int lpr = nrows <= 8 ? 4 : nrows <= 16 ? 2 : 1;
        for (int base = 0; base < nrows; base += 32 / lpr) {
            const int rw = base + lane / lpr, part = lane % lpr;
            const bool on = rw < nrows;
            const int k = on ? rw / nK : 0;
            const float nKv = on ? -Ks[rw - k * nK] : 0.0f;
            const f32x2 nk2 = dup2(nKv);
            const float *src = wbuf + (k0 + k) * ROW;
            // four accumulators of two halves, so that a chain is at most 8 additions
            f32x2 tk[4] = {dup2(0.0f), dup2(0.0f), dup2(0.0f), dup2(0.0f)};
            constexpr int NL = P == 1 ? 16 : 32;   // loads a row
#pragma unroll
            for (int l = part; l < NL; l += 4 * lpr) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if constexpr (P == 1) {   // two paths (delta L, D, delta L, D) per 16-byte load
                        const float4 a = reinterpret_cast<const float4 *>(src)[l + k * lpr];
                        const f32x2 x = add2(pack2(a.x, a.z), nk2);
                        tk[k] = fma2(pack2(fmaxf(lo2(x), 0.0f), fmaxf(hi2(x), 0.0f)), pack2(a.y, a.w), tk[k]);
                    } else {
#pragma unroll
                        for (int h = 0; h < P / 2; ++h) {
                            const ulonglong2 q = reinterpret_cast<const ulonglong2 *>(src + 2 * P * (l + k * lpr))[h];
                            const f32x2 x = add2(q.x, nk2);
                            tk[k] = fma2(pack2(fmaxf(lo2(x), 0.0f), fmaxf(hi2(x), 0.0f)), q.y, tk[k]);
                        }
                    }
                }
            }
            const f32x2 ta = add2(tk[0], tk[1]), tb = add2(tk[2], tk[3]);
            float t = (lo2(ta) + lo2(tb)) + (hi2(ta) + hi2(tb));
            if (lpr > 1) t += __shfl_xor_sync(0xffffffffu, t, 1);
            if (lpr > 2) t += __shfl_xor_sync(0xffffffffu, t, 2);
            if (on && part == 0) {
                const int o = (lo - sh) * nK + rw;
                float s = wacc[o], c = wcmp[o];
                kahan_add(s, c, t);
                wacc[o] = s;
                wcmp[o] = c;
            }
        }
        __syncwarp();
    }
}

// Paths per thread, CTAs per SM to plan registers for, and the sub-block by bucket.  Measured
// (ms per plan execute, N = 65536; 40 forwards, three strikes, M = 64 | 80, 160 forwards, M = 16, 8):
// two paths 1.40, one path at 3 CTAs 1.51, four paths at one CTA 1.75 | two paths 1.23, one 1.20.
// Sub-blocks of 2 / 4 / 8 slots at 40 forwards 1.42 / 1.40 / 1.50, 4 / 8 at 80 1.27 / 1.20 and 8 / 16
// at 160 2.30 / 2.21.  Before (unpacked, 8-slot entry switches): 1.48 | 1.55, 3.35.
template <int NF>
__host__ __device__ constexpr int lmm32_paths() {
    return NF <= 40 ? 2 : 1;
}
template <int NF>
__host__ __device__ constexpr int lmm32_sub() {
    return NF <= 40 ? 4 : NF <= 80 ? 8 : 16;
}
template <int NF>
constexpr int lmm32_min_blocks() {
    return NF <= 16 ? 3 : NF <= 80 ? 2 : 1;
}

// Shared memory: [generator stage][constants][delta K x 8][normals zsets x 8 x P x threads]
//                [payoff buffers][acc][cmp]
template <int NF, int P>
__host__ __device__ __forceinline__ size_t lmm32_smem_layout(const GenParams &g, int nw, int nout, size_t *o_cst,
                                                             size_t *o_k, size_t *o_z, size_t *o_buf, size_t *o_acc, int zsets) {
    size_t off = align16(stage_bytes(g));
    *o_cst = off;
    off = align16(off + lmm32_const_bytes<NF, P>());
    *o_k = off;
    off += sizeof(float) * kMaxStrikes;
    *o_z = off;
    off += sizeof(float) * 8 * P * 32 * (size_t)nw * (size_t)zsets;
    *o_buf = off;
    off = align16(off + sizeof(float) * (size_t)nw * 8 * lmm32_row<P>());
    *o_acc = off;
    off += 2 * sizeof(float) * (size_t)nw * nout;
    return off;
}

// The caplet kernel of FP32 log-Euler plans.  A CTA's warps keep their accumulators over the
// CTA's consecutive units of one replication and write one row at the last of them (run_ends).
template <int NF, int SEQ, bool ZG, bool FLAT>
__global__ void __launch_bounds__(256, lmm32_min_blocks<NF>())
    lmm_caplet32_kernel(const GenParams g, const LmmModel<float> md, const RedParams r, const float *__restrict__ zg) {
    constexpr int P = lmm32_paths<NF>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nw = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nout = r.nout;
    size_t o_cst, o_k, o_z, o_buf, o_acc;
    lmm32_smem_layout<NF, P>(g, nw, nout, &o_cst, &o_k, &o_z, &o_buf, &o_acc, ZG ? 2 : 1);
    float4 *cst = reinterpret_cast<float4 *>(smem_raw + o_cst);
    float *Ks = reinterpret_cast<float *>(smem_raw + o_k);
    float *zb = reinterpret_cast<float *>(smem_raw + o_z) + P * threadIdx.x;
    float *wbuf = reinterpret_cast<float *>(smem_raw + o_buf) + (size_t)warp * 8 * lmm32_row<P>();
    float *acc = reinterpret_cast<float *>(smem_raw + o_acc);
    float *cmp = acc + nw * nout;
    lmm32_fill_constants<NF, P>(md, cst);
    if (threadIdx.x < kMaxStrikes) Ks[threadIdx.x] = md.dl * md.K[threadIdx.x];
    const Lmm32Scal sc{md.nf, md.nK, md.disc0, md.z_scale, md.sig[0] * md.s_scale, lmm_fold_inv(md.sig[0] * md.s_scale), 1.0f, 1.0f};
    zero_acc(acc, cmp, nw * nout);
    const size_t zN = normals_ld(r.N);
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
                const uint32_t at = (uint32_t)pp * blockDim.x + P * threadIdx.x + p, i = tile * r.tile + at;
                active[p] = at < r.tile && i < r.N;
                any = any || active[p];
                pg[p].init(gv, active[p] ? i : 0u);
            }
            if (!__any_sync(0xffffffffu, any)) continue;
            lmm32_path<NF, lmm32_sub<NF>(), SEQ, P, ZG, FLAT>(pg, active, sc, cst, Ks, zb, wbuf, acc + warp * nout, cmp + warp * nout, lane,
                                       ZG ? zg + (size_t)m * sc.nf * zN : nullptr, zN, 0u);
        }
        if (run_ends(r, u, u1)) flush_unit(r, u, acc, cmp);
    }
}

template <int NF, int SEQ, bool ZG, bool FLAT>
static cudaError_t launch_lmm32_v(const Plan &pl, cudaStream_t st, unsigned *rows_grid) {
    constexpr int P = lmm32_paths<NF>();
    auto kern = lmm_caplet32_kernel<NF, SEQ, ZG, FLAT>;
    const LmmModel<float> &md = pl.lmm32;
    GenParams g = pl.gen;
    if (ZG) g.stage = 0;   // no generator table is read
    const int threads = pl.threads;
    size_t a, b, c, d, e2;
    const size_t smem = lmm32_smem_layout<NF, P>(g, threads / 32, pl.red.nout, &a, &b, &c, &d, &e2, ZG ? 2 : 1);
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
    kern<<<grid, threads, smem, st>>>(g, md, pl.red, ZG ? reinterpret_cast<const float *>(pl.znorm) : nullptr);
    *rows_grid = grid;
    return cudaGetLastError();
}

template <int NF, int SEQ, bool ZG>
static cudaError_t launch_lmm32_t(const Plan &pl, cudaStream_t st, unsigned *rows_grid) {
    bool flat = true;
    for (int n = 1; n < pl.lmm32.nf; ++n) flat = flat && pl.lmm32.sig[n] == pl.lmm32.sig[0];
    return flat ? launch_lmm32_v<NF, SEQ, ZG, true>(pl, st, rows_grid)
                : launch_lmm32_v<NF, SEQ, ZG, false>(pl, st, rows_grid);
}

template <int SEQ, bool ZG>
static cudaError_t launch_lmm32(const Plan &pl, cudaStream_t st, unsigned *rows_grid) {
    switch (pl.nf_bucket) {
        case 16: return launch_lmm32_t<16, SEQ, ZG>(pl, st, rows_grid);
        case 40: return launch_lmm32_t<40, SEQ, ZG>(pl, st, rows_grid);
        case 80: return launch_lmm32_t<80, SEQ, ZG>(pl, st, rows_grid);
        case 160: return launch_lmm32_t<160, SEQ, ZG>(pl, st, rows_grid);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace rqmc
