// k_lmm.cu -- dispatch of the LMM caplet kernels by sequence.
#include "k_lmm64.cuh"

namespace rqmc {

extern template cudaError_t launch_caplets_seq<kRasrap>(const Plan &, cudaStream_t, unsigned *);
extern template cudaError_t launch_caplets_seq<kSobolDS>(const Plan &, cudaStream_t, unsigned *);
extern template cudaError_t launch_caplets_seq<kPhilox>(const Plan &, cudaStream_t, unsigned *);

cudaError_t launch_caplets_loaded(const Plan &pl, cudaStream_t st, unsigned *rows_grid);

cudaError_t launch_caplets(const Plan &pl, cudaStream_t st, unsigned *rows_grid) {
    *rows_grid = 0;
    if (pl.znorm && pl.prec == RQMC_FP32) return launch_caplets_loaded(pl, st, rows_grid);
#define RQMC_L(S) launch_caplets_seq<S>(pl, st, rows_grid)
    return RQMC_SEQ_DISPATCH(pl.seq, RQMC_L);
#undef RQMC_L
}

bool caplets_fixed_point(const Plan &pl) {
    LmmFx fx;
    size_t smem;
    return lmm64_applies(pl, fx, smem);
}

}  // namespace rqmc
