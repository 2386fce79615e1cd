// Dense FP64 tile operations (declarations; see dense.cu).
#pragma once

#include "common.cuh"

namespace tlr {

// A = L L' in place (lower; strict upper zeroed) and X = L^-1 (m x m, lower,
// ld ldx), both in FP64; m <= 1024.  One launch on one thread-block cluster up
// to 288 rows, in blocks with substitutions and batched products between them
// above.  A non-positive pivot sets NOT_SPD (info = row_base + local row); X
// then holds nothing of use.
void potrf_inv(tlr_ctx *ctx, cudaStream_t s, double *A, int lda, int m, double *X, int ldx, long long row_base);

// The same for several tiles, sharing every launch (one cluster each); every job
// reports a non-positive pivot in its own status word st.  scratch is set by
// the call.
struct PotrfJob {
    double *A;
    int lda, m;
    double *X;
    int ldx;
    double *scratch;
    DevStatus *st;
    long long row_base;
};
struct PotrfBatch {
    PotrfJob job[kMaxGroup];
};
void potrf_inv_batched(tlr_ctx *ctx, cudaStream_t s, std::vector<PotrfJob> jobs);

// acc[0] += sum_r log A[r, r] (skipped once the status word holds an error);
// maxinv (optional): running maximum of 1 / A[r, r]^2.
void diag_logsum(cudaStream_t s, const double *A, int lda, int m, double *acc, const DevStatus *st,
                 double *maxinv = nullptr);

// acc[0] += |v|^2
void sumsq(cudaStream_t s, const double *v, int m, double *acc);

}  // namespace tlr
