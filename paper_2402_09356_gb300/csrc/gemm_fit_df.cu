// Paired-FP32 linear GEMMs (a translation unit of their own: they compile in parallel).
#include "gemm_fit.cuh"

namespace tlr {

void gemm_fit_df(cudaStream_t s, bool ta, bool tb, int tiles, const GemmProb *dp, const int *dt, int np, int tnmax,
                 double alpha, double beta) {
    launch_fit<true>(s, ta, tb, tiles, dp, dt, np, tnmax, alpha, beta);
}

}  // namespace tlr
