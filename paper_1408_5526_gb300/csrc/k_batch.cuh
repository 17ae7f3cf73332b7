// k_batch.cuh -- persistent kernels over a batch of heterogeneous instruments (LMM caplet
// strips of 8..160 forwards and MBS of up to 4096 months), one kernel per work class
// (160-forward strips, MBS, smaller strips; see BatchLaunch), instantiated per sequence by
// k_batch_{halton,sobol,philox}.cu.
//
// Work items are (instrument, replication m, tile of consecutive points), listed longest
// first (LPT) per class.  Each CTA takes its class's next item with one atomicAdd on a
// ticket counter -- no CTA ever waits on another, so the loop cannot deadlock -- stages that
// instrument's tables for m into shared memory, runs the tile's paths with the same path code as the
// single-instrument kernels (FP32 paths, Kahan sums) and writes the item's own partial
// row.  Results therefore do not depend on which CTA took which item.
#pragma once
#include "k_lmm32.cuh"
#include "k_mbs_run.cuh"

namespace rqmc {

// Work class of an instrument (see BatchLaunch).
__host__ __device__ inline int batch_class(const BatchInst &bi) { return bi.kind != 0 ? 1 : bi.bucket == 160 ? 0 : 2; }

// A strip's item draws its normals before its paths (batch_item_normals) and reads them like the
// normals-loaded caplet kernel.
// The normals of the item's points i0 .. i0 + np - 1 (np <= ld) in dimensions 0 .. nd - 1, by
// all threads of the CTA: z[j ld + (i - i0)].  A task is one lane-run of 8 consecutive points
// in a block of 4 dimensions (the Philox counter block); the 8 points are drawn in lockstep,
// each value bit-identical to the path's own draw.  Points past N repeat point N - 1 (never
// read: a path past N reads slot 0).
template <int SEQ>
__device__ __forceinline__ void batch_item_normals(const GenView &gv, uint32_t i0, uint32_t np, uint32_t N, int nd,
                                                   float *__restrict__ z, uint32_t ld) {
    const uint32_t nrun = (np + 7) >> 3, nblk = (uint32_t)(nd + 3) >> 2;
    for (uint32_t t = threadIdx.x; t < nrun * nblk; t += blockDim.x) {
        const uint32_t jb = t / nrun, r = t % nrun;
        PathGen<SEQ> pg[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) pg[k].init(gv, min(i0 + 8 * r + (uint32_t)k, N - 1));
        for (int jj = 0; jj < 4; ++jj) {
            const int j = 4 * (int)jb + jj;
            if (j >= nd) break;
            float v[8];
            normals32<SEQ, 8>(pg, j, v);
            float4 *dst = reinterpret_cast<float4 *>(z + (size_t)j * ld + 8 * r);
            dst[0] = make_float4(v[0], v[1], v[2], v[3]);
            dst[1] = make_float4(v[4], v[5], v[6], v[7]);
        }
    }
}

// zs: this CTA's normals buffer, at least NF x r.tile floats.  Batch strips have one volatility.
template <int NF, int SEQ>
__device__ __forceinline__ void batch_lmm(const BatchInst &bi, const BatchItem &it, const GenView &gv,
                                          const RedParams &r, unsigned char *smem_raw, float *zs) {
    constexpr int P = lmm32_paths<NF>();
    const int nw = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const LmmModel<float> *md = bi.lmm;
    const int nout = r.nout;
    size_t o_cst, o_k, o_z, o_buf, o_acc;
    lmm32_smem_layout<NF, P>(bi.g, nw, nout, &o_cst, &o_k, &o_z, &o_buf, &o_acc, 2);
    float *zb = reinterpret_cast<float *>(smem_raw + o_z) + P * threadIdx.x;
    float4 *cst = reinterpret_cast<float4 *>(smem_raw + o_cst);
    float *Ks = reinterpret_cast<float *>(smem_raw + o_k);
    float *wbuf = reinterpret_cast<float *>(smem_raw + o_buf) + (size_t)warp * 8 * lmm32_row<P>();
    float *acc = reinterpret_cast<float *>(smem_raw + o_acc);
    float *cmp = acc + nw * nout;
    lmm32_fill_constants<NF, P>(*md, cst);
    if (threadIdx.x < kMaxStrikes) Ks[threadIdx.x] = md->K[threadIdx.x];
    zero_acc(acc, cmp, nw * nout);
    const float s = md->sig[0] * md->s_scale;
    const Lmm32Scal sc{md->nf, md->nK, md->disc0, md->z_scale, s, lmm_fold_inv(s), md->inv_dl, md->dl};
    const uint32_t i0 = it.tile * r.tile;   // the item's first point
    __syncthreads();   // the staged tables are complete before any thread draws from them
    batch_item_normals<SEQ>(gv, i0, min(r.tile, r.N - i0), r.N, md->nf, zs, r.tile);
    __syncthreads();
    for (int pp = 0; pp < r.ppt; pp += P) {
        PathGen<SEQ> pg[P];
        bool act[P];
        bool any = false;
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const uint32_t at = (uint32_t)pp * blockDim.x + P * threadIdx.x + p, i = i0 + at;
            act[p] = at < r.tile && i < r.N;
            any = any || act[p];
            pg[p].init(gv, act[p] ? i : i0);
        }
        if (!__any_sync(0xffffffffu, any)) continue;
        lmm32_path<NF, lmm32_sub<NF>(), SEQ, P, true, true>(pg, act, sc, cst, Ks, zb, wbuf, acc + warp * nout,
                                                            cmp + warp * nout, lane, zs, r.tile, i0);
    }
    flush_unit(r, it.m * bi.tiles_per_m + it.tile, acc, cmp);
}

// The paths of the MBS run kernel, passes of 8 points per thread over the item's tile.
template <int SEQ>
__device__ __forceinline__ void batch_mbs(const BatchInst &bi, const BatchItem &it, const RedParams &r,
                                          unsigned char *smem_raw) {
    const int nw = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const GenParams g = bi.g;
    const MbsModel<float> md = *bi.mbs;
    double *acc = reinterpret_cast<double *>(smem_raw + mbs_run_stage_bytes<SEQ>(g.s, blockDim.x));
    float *ck = reinterpret_cast<float *>(acc + nw);
    MbsRunGen<SEQ> gen(g, smem_raw);
    gen.stage((int)it.m);
    for (int k = threadIdx.x; k <= md.months; k += blockDim.x) ck[k] = md.ck[k];
    const uint32_t base = it.tile * r.tile, end = min(base + r.tile, r.N);
    double sum = 0.0;
    for (uint32_t first = base; first < end; first += 8 * blockDim.x) {
        __syncthreads();   // the tables are complete, the words of the last pass have been read
        gen.pass(first);
        __syncthreads();
        if (first + 256u * warp >= end) continue;   // warp-uniform
        const uint32_t i0 = first + 8 * threadIdx.x;
        gen.i0 = min(i0, (r.N - 1u) & ~7u);
        f32x2 pv[4];
        mbs_run_paths<SEQ>(gen, md, ck, pv);
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (i0 + k < end) s += (double)((k & 1) ? hi2(pv[k / 2]) : lo2(pv[k / 2]));
        sum += warp_sum(s);
    }
    if (lane == 0) acc[warp] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < nw; ++w) t += acc[w];
        r.partials[it.m * bi.tiles_per_m + it.tile] = t;
    }
    __syncthreads();
}

// One persistent kernel per work class KIND (see BatchLaunch).
// CTA timing record: SM id, global-timer start and end of the CTA's item loop.
__device__ __forceinline__ unsigned long long batch_clock() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ uint32_t batch_smid() {
    uint32_t id;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(id));
    return id;
}

template <int SEQ, int KIND>
__global__ void __launch_bounds__(256, KIND == 0 ? 1 : KIND == 1 ? mbs_run_blocks<SEQ>() : 2) batch_kernel(const BatchInst *__restrict__ insts,
                                                                    const BatchItem *__restrict__ items,
                                                                    uint32_t n_items, uint32_t *counter,
                                                                    double *partials, int ppt,
                                                                    unsigned long long *stats, uint32_t stats_cap,
                                                                    float *znorm, size_t zstride) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_ticket;
    const unsigned long long t_start = batch_clock();
    for (;;) {
        if (threadIdx.x == 0) s_ticket = atomicAdd(counter, 1u);
        __syncthreads();
        const uint32_t t = s_ticket;
        __syncthreads();   // every thread has read the ticket before thread 0 takes the next one
        if (t >= n_items) break;
        const BatchItem it = items[t];
        const BatchInst &bi = insts[it.inst];
        GenView gv;
        if constexpr (KIND != 1) stage_tables(bi.g, (int)it.m, smem_raw, gv);
        RedParams r;
        r.nout = bi.nout;
        r.ppt = ppt;
        r.tile = blockDim.x * (uint32_t)ppt;
        r.tiles_per_m = bi.tiles_per_m;
        r.units = bi.tiles_per_m * (uint32_t)bi.g.M;
        r.N = bi.N;
        r.partials = partials + bi.part_off;
        r.status = nullptr;
        r.guard = nullptr;
        float *zs = znorm ? znorm + (size_t)blockIdx.x * zstride : nullptr;   // the CTA's normals buffer
        if constexpr (KIND == 0) {
            batch_lmm<160, SEQ>(bi, it, gv, r, smem_raw, zs);
        } else if constexpr (KIND == 2) {
            switch (bi.bucket) {
                case 16: batch_lmm<16, SEQ>(bi, it, gv, r, smem_raw, zs); break;
                case 40: batch_lmm<40, SEQ>(bi, it, gv, r, smem_raw, zs); break;
                default: batch_lmm<80, SEQ>(bi, it, gv, r, smem_raw, zs); break;
            }
        } else {
            batch_mbs<SEQ>(bi, it, r, smem_raw);
        }
    }
    if (threadIdx.x == 0 && stats && blockIdx.x < stats_cap) {
        unsigned long long *rec = stats + 3ull * ((unsigned long long)KIND * stats_cap + blockIdx.x);
        rec[0] = batch_smid();
        rec[1] = t_start;
        rec[2] = batch_clock();
    }
}

template <int SEQ, int KIND>
cudaError_t launch_batch_class(const BatchLaunch &bl, cudaStream_t st) {
    auto kern = batch_kernel<SEQ, KIND>;
    const size_t smem = bl.smem[KIND];
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    int occ = 0, dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, bl.threads, smem);
    if (occ < 1) occ = 1;
    unsigned grid = (unsigned)std::min<unsigned long long>(bl.n_items[KIND], (unsigned long long)occ * sms);
    if (bl.znorm[KIND]) grid = std::min<unsigned>(grid, bl.zctas[KIND]);   // one normals buffer per CTA
    kern<<<grid, bl.threads, smem, st>>>(bl.insts, bl.items[KIND], bl.n_items[KIND], bl.counter + KIND, bl.partials,
                                         bl.class_ppt[KIND], bl.stats, bl.stats_cap, bl.znorm[KIND], bl.zstride[KIND]);
    return cudaGetLastError();
}

template <int SEQ>
cudaError_t launch_batch_seq(const BatchLaunch &bl, int kind, cudaStream_t st) {
    return kind == 0   ? launch_batch_class<SEQ, 0>(bl, st)
           : kind == 1 ? launch_batch_class<SEQ, 1>(bl, st)
                       : launch_batch_class<SEQ, 2>(bl, st);
}

}  // namespace rqmc
