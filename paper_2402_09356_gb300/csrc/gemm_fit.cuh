// Kernel of the linear GEMMs (instantiated by gemm_fit_f64.cu and gemm_fit_df.cu).
#pragma once

#include "gemm.cuh"

namespace tlr {

// The linear products (every GEMM but the panel generation), FP64 or paired
// FP32, in output tiles cut to the problem: 32 or 64 rows x 8 to 64 columns, in
// steps of 8 (a thread holds TM rows 32 apart and TN columns 8 apart; lanes run
// down the rows, the warps across the columns).  The low-rank products have
// 32 to 200 columns in multiples of 8 and ranks of a few tens; tiles of 64 x 64
// spent up to 60% of these pipe-bound kernels on padding.  Shapes mix in one
// launch (a switch per tile), where one launch per shape queued behind the
// other's last wave.  The next 16 steps of K are loaded into registers while
// the current ones are multiplied, two shared-memory stages.  Every output
// accumulates its terms in the order of k, as k_gemm_f64 / k_gemm_df do.
template <bool kDf>
struct FitArith;
template <>
struct FitArith<false> {
    using T = double;
    struct Acc {
        double d = 0.0;
    };
    static __device__ __forceinline__ const T *a(const GemmProb &p) { return p.A; }
    static __device__ __forceinline__ const T *b(const GemmProb &p) { return p.B; }
    static __device__ __forceinline__ T zero() { return 0.0; }
    static __device__ __forceinline__ void fma_(Acc &c, T x, T y) { c.d = fma(x, y, c.d); }
    static __device__ __forceinline__ double val(const Acc &c) { return c.d; }
};
template <>
struct FitArith<true> {
    using T = float2;
    struct Acc {
        float h = 0.f, l = 0.f;
    };
    static __device__ __forceinline__ const T *a(const GemmProb &p) { return p.A2; }
    static __device__ __forceinline__ const T *b(const GemmProb &p) { return p.B2; }
    static __device__ __forceinline__ T zero() { return make_float2(0.f, 0.f); }
    static __device__ __forceinline__ void fma_(Acc &c, T x, T y) { df_fma(x.x, x.y, y.x, y.y, c.h, c.l); }
    static __device__ __forceinline__ double val(const Acc &c) { return (double)c.h + (double)c.l; }
};

constexpr int kFitK = 16, kFitLd = 65;  // 65: conflict-free stores of transposed operands

template <bool kDf, bool TA, bool TB, int TM, int TN>
__device__ __forceinline__ void fit_tile(const GemmProb &p, int m0, int n0, int n1, double alpha, double beta,
                                         typename FitArith<kDf>::T (*As)[kFitK][kFitLd],
                                         typename FitArith<kDf>::T (*Bs)[kFitK][kFitLd]) {
    using Ar = FitArith<kDf>;
    using T = typename Ar::T;
    constexpr int R = 32 * TM, C = 8 * TN;
    constexpr int kLa = R * kFitK / kGemmThreads, kLb = (C * kFitK + kGemmThreads - 1) / kGemmThreads;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const T *A = Ar::a(p), *B = Ar::b(p);
    typename Ar::Acc acc[TM][TN];
    T ra[kLa], rb[kLb];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int u = 0; u < kLa; ++u) {
            const int e = tid + u * kGemmThreads, r = TA ? e / kFitK : e % R, kk = TA ? e % kFitK : e / R;
            const int gr = m0 + r, gk = k0 + kk;
            ra[u] = gr < p.m && gk < p.k ? (TA ? A[(int64_t)gr * p.lda + gk] : A[(int64_t)gk * p.lda + gr]) : Ar::zero();
        }
#pragma unroll
        for (int u = 0; u < kLb; ++u) {
            const int e = tid + u * kGemmThreads, c = TB ? e % C : e / kFitK, kk = TB ? e / C : e % kFitK;
            const int gc = n0 + c, gk = k0 + kk;
            rb[u] = e < C * kFitK && gc < n1 && gk < p.k
                        ? (TB ? B[(int64_t)gk * p.ldb + gc] : B[(int64_t)gc * p.ldb + gk]) : Ar::zero();
        }
    };
    auto store = [&](int s) {
#pragma unroll
        for (int u = 0; u < kLa; ++u) {
            const int e = tid + u * kGemmThreads, r = TA ? e / kFitK : e % R, kk = TA ? e % kFitK : e / R;
            As[s][kk][r] = ra[u];
        }
#pragma unroll
        for (int u = 0; u < kLb; ++u) {
            const int e = tid + u * kGemmThreads, c = TB ? e % C : e / kFitK, kk = TB ? e / C : e % kFitK;
            if (e < C * kFitK) Bs[s][kk][c] = rb[u];
        }
    };
    if (p.k > 0) {
        fetch(0);
        store(0);
    }
    __syncthreads();
    int s = 0;
    for (int k0 = 0; k0 < p.k; k0 += kFitK, s ^= 1) {
        const bool more = k0 + kFitK < p.k;
        if (more) fetch(k0 + kFitK);
        // an inner dimension that is a rank (about 20) ends inside a step: its
        // padding, exact zeros, is left out in twos.  n = 40,000 tensor: P operands
        // 41 -> 33 ms, corrections 32 -> 30; batch of eight: 110 -> 95, 41.5 -> 39
        const int kn = min(kFitK, p.k - k0);
        for (int k2 = 0; k2 < kn; k2 += 2) {
#pragma unroll
            for (int kk = k2; kk < k2 + 2; ++kk) {
                T a[TM], b[TN];
#pragma unroll
                for (int i = 0; i < TM; ++i) a[i] = As[s][kk][lane + 32 * i];
#pragma unroll
                for (int j = 0; j < TN; ++j) b[j] = Bs[s][kk][warp + 8 * j];
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < TN; ++j) Ar::fma_(acc[i][j], a[i], b[j]);
            }
        }
        if (more) store(s ^ 1);
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < TN; ++j) {
        const int c = n0 + warp + 8 * j;
        if (c >= n1) continue;
#pragma unroll
        for (int i = 0; i < TM; ++i) {
            const int r = m0 + lane + 32 * i;
            if (r >= p.m) continue;
            double *cp = p.C + (int64_t)c * p.ldc + r;
            const double ab = alpha * Ar::val(acc[i][j]);
            if (p.sym) {
                if (r > c) continue;
                p.C[(int64_t)r * p.ldc + c] = ab;  // and *cp, from the upper triangle (beta = 0)
            }
            *cp = beta == 0.0 ? ab : ab + beta * (*cp);
        }
    }
}

template <bool kDf, bool TA, bool TB>
__global__ void __launch_bounds__(kGemmThreads, 2)
k_gemm_fit(const GemmProb *__restrict__ probs, const int *__restrict__ tile_off, int nprob, int tnmax, double alpha,
           double beta) {
    using T = typename FitArith<kDf>::T;
    __shared__ T As[2][kFitK][kFitLd], Bs[2][kFitK][kFitLd];
    const int t = blockIdx.x;
    int lo = 0, hi = nprob - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (tile_off[mid] <= t) lo = mid; else hi = mid - 1;
    }
    GemmProb p = probs[lo];
    const int local = t - tile_off[lo], rt = (p.m + 63) / 64, ct = fit_col_tiles(p.n, tnmax), tc = local / rt;
    // Triangular A: a row tile ends at its own diagonal (the terms left out are
    // exact zeros), the longest tiles first.  V <- L^-1 V of an n = 16,000 FP64
    // evaluation 10.8 -> 7.2 ms, of a batch of eight datasets 71 -> 48 ms
    const int m0 = (!TA && p.lower ? rt - 1 - local % rt : local % rt) * 64;
    if (!TA && p.lower) p.k = min(p.k, m0 + 64);
    // column groups of 8, dealt evenly to the ct column tiles
    const int ncg = (p.n + 7) / 8, base = ncg / ct, rem = ncg % ct;
    const int n0 = 8 * (tc * base + min(tc, rem)), tn = base + (tc < rem), n1 = min(p.n, n0 + 8 * tn);
    if (p.sym && m0 >= n1) return;  // C = A'A: the upper triangle's tiles
#define TLR_FIT(TMV, TNV) \
    case TNV: fit_tile<kDf, TA, TB, TMV, TNV>(p, m0, n0, n1, alpha, beta, As, Bs); break;
    // the widths without a body of their own take the next one (their columns
    // past n1 are zero)
    if (p.m - m0 > 32) {
        switch (tn == 7 ? 8 : tn) {
            TLR_FIT(2, 1)
            TLR_FIT(2, 2)
            TLR_FIT(2, 3)
            TLR_FIT(2, 4)
            TLR_FIT(2, 5)
            TLR_FIT(2, 6)
            TLR_FIT(2, 8)
        }
    } else {
        switch (tn > 4 ? 8 : (tn == 3 ? 4 : tn)) {
            TLR_FIT(1, 1)
            TLR_FIT(1, 2)
            TLR_FIT(1, 4)
            TLR_FIT(1, 8)
        }
    }
#undef TLR_FIT
}

template <bool kDf>
static void launch_fit(cudaStream_t s, bool ta, bool tb, int tiles, const GemmProb *dp, const int *dt, int np, int tnmax,
                       double alpha, double beta) {
    auto go = [&](void (*k)(const GemmProb *, const int *, int, int, double, double)) {
        launch(k, (unsigned)tiles, kGemmThreads, 0, s, dp, dt, np, tnmax, alpha, beta);
    };
    if (ta) go(k_gemm_fit<kDf, true, false>);
    else if (tb) go(k_gemm_fit<kDf, false, true>);
    else go(k_gemm_fit<kDf, false, false>);
    TLR_CHECK_LAUNCH();
}

}  // namespace tlr
