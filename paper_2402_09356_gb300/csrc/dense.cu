// Dense FP64 tile kernels of the TLR Cholesky (Sec. 2; the diagonal tiles stay
// dense): blocked right-looking Cholesky of one diagonal tile with its
// inverse, and the log-determinant / quadratic-form reductions of Eq. 1.2.
//
// Blocks of 32 rows/columns are factored or solved by one CTA in shared
// memory; everything else is a batched GEMM update so that it spreads over
// the whole GPU (one SM's FP64 pipe alone would take milliseconds per tile).
#include <algorithm>
#include <mutex>

#include <cooperative_groups.h>

#include "common.cuh"
#include "dense.cuh"
#include "gemm.cuh"
#include "tlr_internal.cuh"

namespace tlr {

namespace cg = cooperative_groups;

constexpr int kBlk = 32;


// ---------------------------------------------------------------------------
// Cholesky and inverse of one diagonal tile in a single launch.
//
// One cluster of kCl CTAs (tiles wider than kPotrfOuter come block by block,
// see potrf_inv_batched); the tile (m <= 1024, column major) stays in global
// memory, which for one tile is L2-resident, and every load goes to L2
// (__ldcg: another CTA may have written the line in an earlier phase).  A
// cluster barrier (release/acquire at cluster scope) separates dependent
// phases.  The factorisation and the inverse X = L^-1 advance together, in
// 32-wide block steps, two barriers a step.  Block step k:
//   1. (all CTAs) the panel rows below the block, A[r, k] <- A[r, k] L_kk^-T,
//      and the inverse's block row, X[k, :] <- L_kk^-1 X[k, :] (columns
//      < end of block k; X starts as I), with L_kk^-1 from step k - 1;
//   -- barrier --
//   2. CTA 0 updates the next diagonal block, A_{k+1,k+1} -= L_{k+1,k}
//      L_{k+1,k}', and factors and inverts it in shared memory
//      (potrf_diag_block): the diagonal block of step k + 1 is ready when step k ends.  The other
//      CTAs take, round robin, the rest of the trailing lower triangle,
//      A_IJ -= L_Ik L_Jk' (I >= J > k), and the inverse's update
//      X_IJ -= L_Ik X_kJ (I > k, J <= k), 32 x 32 output tiles, loading
//      their next tile's operands into registers while they update the
//      current one;
//   -- barrier --
// FP64 throughout.  A non-positive pivot sets NOT_SPD (info = row_base + row)
// and every CTA leaves at the next barrier.
constexpr int kPotrfThreads = 256;
constexpr int kTileLoads = kBlk * kBlk / kPotrfThreads;  // operand elements per thread and tile

// C (32 x 32, rows r0.., cols c0.. of a column-major matrix) -= A B' or A B:
// a, b are 32 x 32 operand blocks already in shared memory as [row][k].
__device__ __forceinline__ void tile_update32(double *C, int ldc, const double (*a)[kBlk + 1],
                                              const double (*b)[kBlk + 1], int rows, int cols, bool lower_only) {
    const int tid = threadIdx.x, tr = (tid & 15) * 2, tc = (tid >> 4) * 2;
    // the C entries are read before the product, so that their latency
    // overlaps with it (only this CTA updates this tile in this step)
    double cv[2][2];
#pragma unroll
    for (int x = 0; x < 2; ++x)
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            const int r = tr + x, c = tc + y;
            cv[x][y] = (r < rows && c < cols && (!lower_only || c <= r)) ? __ldcg(C + (int64_t)c * ldc + r) : 0.0;
        }
    double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll 8
    for (int k = 0; k < kBlk; ++k) {
        const double a0 = a[tr][k], a1 = a[tr + 1][k], b0 = b[tc][k], b1 = b[tc + 1][k];
        acc[0][0] = fma(a0, b0, acc[0][0]);
        acc[0][1] = fma(a0, b1, acc[0][1]);
        acc[1][0] = fma(a1, b0, acc[1][0]);
        acc[1][1] = fma(a1, b1, acc[1][1]);
    }
#pragma unroll
    for (int x = 0; x < 2; ++x)
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            const int r = tr + x, c = tc + y;
            if (r < rows && c < cols && (!lower_only || c <= r)) C[(int64_t)c * ldc + r] = cv[x][y] - acc[x][y];
        }
}

// 1 / sqrt(d) for d > 0 (normal): the PTX approximation y (error e = 1 - d y^2
// ~ 2^-19), then one third-order step y + y e (1/2 + 3/8 e), to about an ulp.
// The pivot chain of a diagonal block runs through it once per column, and
// every FP64 instruction takes 64 cycles: five of them against eight for two
// Newton steps.
__device__ __forceinline__ double rsqrt_step(double d) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
    const double e = fma(-(d * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// Cholesky of the w x w diagonal block at (p, p) of A by the calling CTA,
// with the block's inverse: L_kk into A (lower; upper part of the block 0),
// L_kk^-1 into Li (32 x 32, row major).  The block's lower triangle is in M on
// entry.  Returns the first failing column (non-positive pivot) or -1, the
// same on every thread.
// Factor and inverse advance together: after column c, M[r][j] holds L^-1's
// entry (of the elimination so far) for j <= c and the updated A for j > c, so
// that one rank-1 update a column serves both (ov: row c of the inverse up to
// column c, column c of L behind it).  Warp 0 keeps the diagonal in
// registers (lane r: entry (r, r)) and runs the chain that bounds the block --
// scale, diagonal update, reciprocal square root, about 600 cycles a column --
// while the other warps update the rows behind it: 19,000 cycles a block, where
// a column-wise factorisation and then a row-wise inverse took 59,000.
__device__ int potrf_diag_block(double *A, int lda, int p, int w, double *Li, double (*M)[kBlk + 1], double *ov,
                                double *sy, int *s_bad) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double diag = 0.0, y = 0.0;
    if (warp == 0) {
        diag = lane < w ? M[lane][lane] : 1.0;
        const double d0 = __shfl_sync(0xFFFFFFFFu, diag, 0);
        if (lane == 0) *s_bad = d0 > 0.0 ? -1 : 0;
        y = rsqrt_step(d0);
        if (lane == 0) *sy = y;
    }
    __syncthreads();
    const int r = tid >> 3, q = tid & 7;  // the update: row r, columns q, q + 8, ...
    for (int c = 0; c < w; ++c) {
        if (*s_bad >= 0) break;  // written before the last barrier: uniform
        // column c of L and row c of the inverse
        if (warp == 0) {
            double l = 0.0;
            if (lane > c && lane < w) l = M[lane][c] * y;
            if (lane > c) ov[lane] = l;
            diag = fma(-l, l, diag);
            if (lane < w) A[(int64_t)(p + c) * lda + p + lane] = lane > c ? l : (lane == c ? diag * y : 0.0);
        } else if (warp == 1) {
            const double yc = *sy, x = lane < c ? M[c][lane] * yc : (lane == c ? yc : 0.0);
            if (lane <= c) ov[lane] = x;
            Li[c * kBlk + lane] = x;
        }
        __syncthreads();
        if (warp == 0 && c + 1 < w) {
            const double d = __shfl_sync(0xFFFFFFFFu, diag, c + 1);
            y = rsqrt_step(d);
            if (lane == 0) {
                *sy = y;
                if (!(d > 0.0)) *s_bad = c + 1;
            }
        }
        if (r > c && r < w) {
            const double l = ov[r];
#pragma unroll
            for (int k = 0; k < kBlk / 8; ++k) {
                const int j = q + 8 * k;
                if (j < r) M[r][j] = fma(-l, ov[j], j == c ? 0.0 : M[r][j]);
            }
        }
        __syncthreads();
    }
    const int bad = *s_bad;
    if (bad >= 0) return bad;
    for (int e = w * kBlk + tid; e < kBlk * kBlk; e += kPotrfThreads) Li[e] = 0.0;  // rows past the block
    return -1;
}

// `scratch`: 32 x 1024 doubles for the diagonal block inverses, then one
// word through which CTA 0 tells the cluster to stop (the context's status
// word may be set by kernels on other streams at any time, so the CTAs do not
// each read it to decide).
// One cluster per job (blockIdx.x / kCl): the diagonal tiles of several
// factorisations in one launch (the jobs travel in the kernel parameters).
template <int kCl>
__global__ void __launch_bounds__(kPotrfThreads) k_potrf_inv(const PotrfBatch jobs) {
    const PotrfJob J = jobs.job[blockIdx.x / kCl];
    double *const A = J.A, *const X = J.X, *const scratch = J.scratch;
    const int lda = J.lda, m = J.m, ldx = J.ldx;
    DevStatus *const st = J.st;
    const long long row_base = J.row_base;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), tid = threadIdx.x;
    const int gtid = rank * kPotrfThreads + tid, gthreads = kCl * kPotrfThreads;
    __shared__ double sa[kBlk][kBlk + 1], sb[kBlk][kBlk + 1], sl[kBlk][kBlk + 1];
    __shared__ double ov[kBlk], sy;
    __shared__ int s_bad;
    const int nbk = (m + kBlk - 1) / kBlk;
    double *dinv = scratch;
    long long *stop = reinterpret_cast<long long *>(scratch + (int64_t)kBlk * kBlk * kBlk);
    // X = I; CTA 0 factors the first diagonal block
    for (int64_t e = gtid; e < (int64_t)m * m; e += gthreads) {
        const int r = (int)(e % m), c = (int)(e / m);
        X[(int64_t)c * ldx + r] = (r == c) ? 1.0 : 0.0;
    }
    if (rank == 0) {
        // one read of the status word decides for the whole CTA (another
        // stream's kernel may set it at any time)
        if (tid == 0) s_bad = __ldcg(&st->code) ? 1 : 0;
        __syncthreads();
        long long halt = s_bad ? 1LL : 0LL;
        __syncthreads();
        if (!halt) {
            for (int e = tid; e < kBlk * kBlk; e += kPotrfThreads) {
                const int r = e % kBlk, c = e / kBlk;
                sa[r][c] = (r < m && c <= r) ? __ldcg(A + (int64_t)c * lda + r) : 0.0;
            }
            __syncthreads();
            const int bad = potrf_diag_block(A, lda, 0, min(kBlk, m), dinv, sa, ov, &sy, &s_bad);
            if (bad >= 0) {
                if (tid == 0) set_status(st, TLR_ERR_NOT_SPD, row_base + bad);
                halt = 1;
            }
        }
        if (tid == 0) __stcg(stop, halt);
    }
    cl.sync();
    if (__ldcg(stop)) return;
    for (int kb = 0; kb < nbk; ++kb) {
        const int p = kb * kBlk, w = min(kBlk, m - p);
        const double *Li = dinv + (int64_t)kb * kBlk * kBlk;  // L_kk^-1, row major
        // 1. panel rows below the block: x <- a L_kk^-T, x_c = sum_{k<=c} a_k Linv[c][k];
        //    inverse block row: X[k-block, c] <- L_kk^-1 X[k-block, c], c < p + w
        for (int e = tid; e < kBlk * kBlk; e += kPotrfThreads) {
            sl[e / kBlk][e % kBlk] = __ldcg(Li + e);
        }
        __syncthreads();
        // rows and columns dealt to the CTAs in turn, eight threads each (thread
        // q forms entries q, q + 8, ...: every scheduler takes a share, and a
        // chain is 80 multiply-adds, not 528); operands through shared memory,
        // 32 rows or columns at a time
        const int q8 = tid & 7, u8 = tid >> 3;
        const int rows_per = (m - p - w + kCl - 1) / kCl, r_hi = min(m, p + w + (rank + 1) * rows_per);
        for (int b0 = p + w + rank * rows_per; b0 < r_hi; b0 += kBlk) {
            __syncthreads();
            for (int e = tid; e < kBlk * kBlk; e += kPotrfThreads) {
                const int r = b0 + e % kBlk, k = e / kBlk;
                sa[e % kBlk][k] = (r < r_hi && k < w) ? __ldcg(A + (int64_t)(p + k) * lda + r) : 0.0;
            }
            __syncthreads();
            const int r = b0 + u8;
            if (r < r_hi) {
#pragma unroll
                for (int t = 0; t < kBlk / 8; ++t) {
                    const int c = q8 + 8 * t;
                    double x0 = 0.0, x1 = 0.0;
#pragma unroll 4
                    for (int k = 0; k < 8 * t + 8; k += 2) {  // L_kk^-1 is 0 right of its diagonal
                        x0 = fma(sa[u8][k], sl[c][k], x0);
                        x1 = fma(sa[u8][k + 1], sl[c][k + 1], x1);
                    }
                    if (c < w) A[(int64_t)(p + c) * lda + r] = x0 + x1;
                }
            }
        }
        for (int b0 = rank; b0 < p + w; b0 += kCl * kBlk) {
            __syncthreads();
            for (int e = tid; e < kBlk * kBlk; e += kPotrfThreads) {
                const int c = b0 + kCl * (e / kBlk), k = e % kBlk;
                const bool in = c < p + w && k < w;
                sa[e / kBlk][k] = in ? __ldcg(X + (int64_t)c * ldx + p + k) : 0.0;
            }
            __syncthreads();
            const int c = b0 + kCl * u8;
            if (c < p + w) {
#pragma unroll
                for (int t = 0; t < kBlk / 8; ++t) {
                    const int r = q8 + 8 * t;
                    double x0 = 0.0, x1 = 0.0;
#pragma unroll 4
                    for (int k = 0; k < 8 * t + 8; k += 2) {
                        x0 = fma(sl[r][k], sa[u8][k], x0);
                        x1 = fma(sl[r][k + 1], sa[u8][k + 1], x1);
                    }
                    if (r < w) X[(int64_t)c * ldx + p + r] = x0 + x1;
                }
            }
        }
        cl.sync();
        if (kb + 1 >= nbk) break;
        // 2. trailing and inverse updates by this block column; CTA 0 also
        //    prepares the next diagonal block
        const int nt = nbk - kb - 1;            // block rows below
        const int ntr = nt * (nt + 1) / 2;      // trailing tiles (I >= J > kb); tile 0 is (kb+1, kb+1)
        const int ntot = ntr + nt * (kb + 1);   // + inverse tiles (I > kb, J <= kb)
        // tile t -> operands: trailing (I, J): C = A_IJ, a = L_I,kb, b = L_J,kb (as [row][k]);
        //                     inverse (I, J): C = X_IJ, a = L_I,kb, b = X_kb,J (as [col][k])
        auto tile_of = [&](int t, bool &inv, int &I, int &Jb) {
            if (t < ntr) {
                int bi = 0, rem = t;
                while (rem > bi) { rem -= bi + 1; ++bi; }
                inv = false;
                I = kb + 1 + bi;
                Jb = kb + 1 + rem;
            } else {
                const int u = t - ntr;
                inv = true;
                I = kb + 1 + u % nt;
                Jb = u / nt;
            }
        };
        double ra[kTileLoads], rb[kTileLoads];
        auto fetch = [&](int t) {
            bool inv;
            int I, Jb;
            tile_of(t, inv, I, Jb);
            const int ri = I * kBlk, cj = Jb * kBlk, rows = min(kBlk, m - ri), cols = min(kBlk, m - cj);
#pragma unroll
            for (int u = 0; u < kTileLoads; ++u) {
                const int e = tid + u * kPotrfThreads, r = e % kBlk, k = e / kBlk;
                ra[u] = (r < rows && k < w) ? __ldcg(A + (int64_t)(p + k) * lda + ri + r) : 0.0;
                if (inv) rb[u] = (r < cols && k < w) ? __ldcg(X + (int64_t)(cj + r) * ldx + p + k) : 0.0;
                else rb[u] = (r < cols && k < w) ? __ldcg(A + (int64_t)(p + k) * lda + cj + r) : 0.0;
            }
        };
        auto apply = [&](int t) {
            bool inv;
            int I, Jb;
            tile_of(t, inv, I, Jb);
            const int ri = I * kBlk, cj = Jb * kBlk, rows = min(kBlk, m - ri), cols = min(kBlk, m - cj);
            __syncthreads();
#pragma unroll
            for (int u = 0; u < kTileLoads; ++u) {
                const int e = tid + u * kPotrfThreads;
                sa[e % kBlk][e / kBlk] = ra[u];
                sb[e % kBlk][e / kBlk] = rb[u];
            }
            __syncthreads();
            return inv ? (X + (int64_t)cj * ldx + ri) : (A + (int64_t)cj * lda + ri);
        };
        if (rank == 0) {
            // tile (kb+1, kb+1): its lower triangle, entry e in packed order,
            // then the next diagonal block
            const int pn = (kb + 1) * kBlk, wn = min(kBlk, m - pn);
            fetch(0);
            apply(0);
            for (int e = tid; e < kBlk * (kBlk + 1) / 2; e += kPotrfThreads) {
                int r = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
                r += (r + 1) * (r + 2) / 2 <= e;
                r -= r * (r + 1) / 2 > e;
                const int c = e - r * (r + 1) / 2;
                double v = 0.0;
                if (r < wn) {
                    v = __ldcg(A + (int64_t)(pn + c) * lda + pn + r);
                    double x0 = 0.0, x1 = 0.0;
#pragma unroll 8
                    for (int k = 0; k < kBlk; k += 2) {
                        x0 = fma(sa[r][k], sa[c][k], x0);
                        x1 = fma(sa[r][k + 1], sa[c][k + 1], x1);
                    }
                    v -= x0 + x1;
                }
                sl[r][c] = v;
            }
            __syncthreads();
            const int bad = potrf_diag_block(A, lda, pn, wn, dinv + (int64_t)(kb + 1) * kBlk * kBlk, sl, ov, &sy, &s_bad);
            if (bad >= 0 && tid == 0) {
                set_status(st, TLR_ERR_NOT_SPD, row_base + pn + bad);
                __stcg(stop, 1LL);
            }
        } else {
            const int step = kCl - 1;
            if (1 + rank - 1 < ntot) fetch(1 + rank - 1);
            for (int t = 1 + rank - 1; t < ntot; t += step) {
                bool inv;
                int I, Jb;
                tile_of(t, inv, I, Jb);
                const int ri = I * kBlk, cj = Jb * kBlk, rows = min(kBlk, m - ri), cols = min(kBlk, m - cj);
                double *C = apply(t);
                if (t + step < ntot) fetch(t + step);
                tile_update32(C, inv ? ldx : lda, sa, sb, rows, cols, !inv && I == Jb);
            }
        }
        cl.sync();
        if (__ldcg(stop)) return;  // written by CTA 0 only, before the barrier
    }
    // zero the strict upper triangle of the factor
    for (int64_t e = gtid; e < (int64_t)m * m; e += gthreads) {
        const int r = (int)(e % m), c = (int)(e / m);
        if (r < c) A[(int64_t)c * lda + r] = 0.0;
    }
}

// One cluster launch for the blocks of `act` (m <= 1024 each): Cholesky and inverse.
static void potrf_cluster(tlr_ctx *ctx, cudaStream_t s, const std::vector<PotrfJob> &act) {
    PotrfBatch b{};
    // scratch per job: the diagonal-block inverses and the cluster's stop word
    const size_t per = (size_t)kBlk * kBlk * kBlk + 8;
    for (size_t q = 0; q < act.size(); ++q) {
        b.job[q] = act[q];
        b.job[q].scratch = ctx->d_potrf_scratch + per * q;
    }
    static std::once_flag once;
    static int csize = 8;  // 16 CTAs where the device runs such clusters, else 8
    std::call_once(once, [] {
        if (cudaFuncSetAttribute(k_potrf_inv<16>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(16);
            cfg.blockDim = dim3(kPotrfThreads);
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = 16;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            int nclusters = 0;
            if (cudaOccupancyMaxActiveClusters(&nclusters, k_potrf_inv<16>, &cfg) == cudaSuccess && nclusters > 0)
                csize = 16;
        }
        cudaGetLastError();  // clear any error of the queries
    });
    const int nc = (int)act.size();
    if (csize == 16) launch_clustered(k_potrf_inv<16>, 16, nc, kPotrfThreads, 0, s, b);
    else launch_clustered(k_potrf_inv<8>, 8, nc, kPotrfThreads, 0, s, b);
}

// Around the diagonal blocks (width w) of a tile that is factored in blocks:
// zero A above them, X and S outside them.
struct PotrfEdge {
    double *A, *X, *S;
    int lda, ldx, lds, m, w;
};
struct PotrfEdges {
    PotrfEdge e[kMaxGroup];
};
__global__ void k_potrf_edges(const PotrfEdges jobs) {
    const PotrfEdge J = jobs.e[blockIdx.y];
    for (int c = blockIdx.x; c < J.m; c += gridDim.x) {
        const int b0 = c / J.w * J.w, b1 = min(J.m, b0 + J.w);
        for (int r = threadIdx.x; r < J.m; r += blockDim.x) {
            if (r < b0) J.A[(int64_t)c * J.lda + r] = 0.0;
            if (r < b0 || r >= b1) {
                J.X[(int64_t)c * J.ldx + r] = 0.0;
                J.S[(int64_t)c * J.lds + r] = 0.0;
            }
        }
    }
}

// Substitution with a factored diagonal block L_bb (w <= kPotrfOuter columns) in
// steps of 32, the inverses of its 32 x 32 diagonal blocks taken from X_bb's:
// `rows` rows a of A below the block become those of L (x L_bb' = a, in place),
// `cols` columns of S the inverse's (L_bb y = s, into Y).
struct PotrfSub {
    const double *L, *X;
    double *A;
    const double *S;
    double *Y;
    int ldl, ldx, lds, w, rows, cols;
};
struct PotrfSubs {
    PotrfSub j[kMaxGroup];
};
// One warp a right-hand side, its entry r of a step in lane r, four a CTA (a row
// of L that a warp reads serves the others from L1; four adjacent rows of A are a
// 32-byte sector).  No barrier: a warp's steps depend on its own vector only.
// w^2 / 64 + w / 2 multiply-adds a warp of 64 cycles each, one warp a scheduler at
// m = 800: the FP64 pipe is 41% busy, the rest is latency (L comes from L2 16
// columns ahead); 115 us for 512 vectors of 288 alone and cold.  The
// sums are of 32 terms, each taken from the entry.  A product with X_bb takes as
// long, but |L L' - A| and |L X - I| of smooth fields are then two to six times
// those of the algorithm that inverts 32 x 32 blocks only, which these are.
constexpr int kSubThreads = 128, kSubVecs = kSubThreads / 32, kSubAhead = 16;
constexpr int kPotrfOuter = 288, kPotrfChunk = 96;
__global__ void __launch_bounds__(kSubThreads) k_potrf_sub(const PotrfSubs jobs) {
    __shared__ double ys[kSubVecs][kPotrfOuter], ts[kSubVecs][kBlk];
    const PotrfSub J = jobs.j[blockIdx.y];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, w = J.w;
    const int row_ctas = (J.rows + kSubVecs - 1) / kSubVecs, bx = blockIdx.x;
    const bool row = bx < row_ctas;
    const int v0 = (row ? bx : bx - row_ctas) * kSubVecs, nv = min(kSubVecs, (row ? J.rows : J.cols) - v0);
    if (nv <= 0) return;
    if (row) {
        for (int e = tid; e < kSubVecs * w; e += kSubThreads) {
            const int v = e % kSubVecs, k = e / kSubVecs;
            if (v < nv) ys[v][k] = J.A[(int64_t)k * J.ldl + v0 + v];
        }
    } else {
        for (int v = 0; v < nv; ++v)
            for (int k = tid; k < w; k += kSubThreads) ys[v][k] = J.S[(int64_t)(v0 + v) * J.lds + k];
    }
    __syncthreads();
    if (warp < nv) {
        double *y = ys[warp], *t = ts[warp];
        for (int p = 0; p < w; p += kBlk) {
            const bool in = p + lane < w;
            const double *Lr = J.L + p + lane, *Xr = J.X + (int64_t)p * J.ldx + p + lane;
            double x[kBlk], l[2][kSubAhead];
            auto load = [&](int k0, double (&v)[kSubAhead]) {
#pragma unroll
                for (int k = 0; k < kSubAhead; ++k) v[k] = in && k0 < p ? Lr[(int64_t)(k0 + k) * J.ldl] : 0.0;
            };
            load(0, l[0]);
#pragma unroll
            for (int k = 0; k < kBlk; ++k) x[k] = in && k <= lane ? Xr[(int64_t)k * J.ldx] : 0.0;
            double a = in ? y[p + lane] : 0.0;
            for (int k0 = 0; k0 < p; k0 += 2 * kSubAhead) {  // 32 columns: two loads ahead of their use
                double s0 = 0.0, s1 = 0.0;
                load(k0 + kSubAhead, l[1]);
#pragma unroll
                for (int k = 0; k < kSubAhead; k += 2) {
                    s0 = fma(l[0][k], y[k0 + k], s0);
                    s1 = fma(l[0][k + 1], y[k0 + k + 1], s1);
                }
                load(k0 + 2 * kSubAhead, l[0]);
#pragma unroll
                for (int k = 0; k < kSubAhead; k += 2) {
                    s0 = fma(l[1][k], y[k0 + kSubAhead + k], s0);
                    s1 = fma(l[1][k + 1], y[k0 + kSubAhead + k + 1], s1);
                }
                a -= s0 + s1;
            }
            t[lane] = a;
            __syncwarp();
            double s0 = 0.0, s1 = 0.0;
#pragma unroll
            for (int k = 0; k < kBlk; k += 2) {
                s0 = fma(x[k], t[k], s0);
                s1 = fma(x[k + 1], t[k + 1], s1);
            }
            if (in) y[p + lane] = s0 + s1;
            __syncwarp();
        }
    }
    __syncthreads();
    if (row) {
        for (int e = tid; e < kSubVecs * w; e += kSubThreads) {
            const int v = e % kSubVecs, k = e / kSubVecs;
            if (v < nv) J.A[(int64_t)k * J.ldl + v0 + v] = ys[v][k];
        }
    } else {
        for (int v = 0; v < nv; ++v)
            for (int k = tid; k < w; k += kSubThreads) J.Y[(int64_t)(v0 + v) * J.ldx + k] = ys[v][k];
    }
}

// Tiles wider than kPotrfOuter are factored in blocks of w <= kPotrfOuter
// columns: the cluster kernel factors and inverts a diagonal block, the rows of L
// below it and its rows of the inverse follow by substitution (k_potrf_sub), and
// the products between blocks run as batched FP64 GEMMs over the whole GPU.
// For block b, with X_bb = L_bb^-1:
//   L_ib L_bb' = A_ib  (i > b);   A_ij -= L_ib L_jb'  (i >= j > b);
//   L_bb X_bj = S_bj  (j < b);    S_ij -= L_ib X_bj  (i > b >= j),
// S_ij the negated sum of L_ik X_kj so far.  One cluster alone runs the tile's
// m^3 / 3 multiply-adds twice over on 16 of the 152 SMs, and its trailing
// updates, not its pivot chain, take most of the time.  One tile alone, one
// cluster -> blocks: m = 300 0.99 -> 0.55 ms, 400 1.31 -> 0.72, 512 1.81 -> 0.92,
// 576 2.26 -> 1.05, 800 4.63 -> 1.56, 1,024 8.59 -> 2.30; up to 288 there is one
// block.  (At m = 800 widths of 224 and 160 took a tenth longer: more launches,
// each as long as one 32 x 32 output tile's FP64 chain.)  The GEMMs are split
// by column chunks so that the triangular factors' zeros are skipped, and sum 32
// terms at a time (of 288 terms in one sum each rounding is of the whole entry:
// |L L' - A| of a rough field was twice the 32-wide algorithm's).
void potrf_inv_batched(tlr_ctx *ctx, cudaStream_t s, std::vector<PotrfJob> jobs) {
    std::vector<PotrfJob> act;
    for (const PotrfJob &J : jobs) {
        if (J.m <= 0) continue;
        if (J.m > kBlk * kBlk) throw make_error(TLR_ERR_ARG, "tile too large for the cluster POTRF (%d)", J.m);
        act.push_back(J);
    }
    if (act.empty()) return;
    if ((int)act.size() > kMaxGroup) throw make_error(TLR_ERR_ARG, "more than %d diagonal tiles in one launch", kMaxGroup);
    const size_t per = (size_t)kBlk * kBlk * kBlk + 8;
    if ((int)act.size() > ctx->potrf_scratch_jobs) {
        if (ctx->d_potrf_scratch) TLR_CUDA_TRY(cudaFree(ctx->d_potrf_scratch));  // syncs the device
        ctx->d_potrf_scratch = nullptr;
        ctx->potrf_scratch_jobs = 0;
        const int want = std::max((int)act.size(), 2 * ctx->potrf_scratch_jobs);
        TLR_CUDA_TRY(cudaMalloc(&ctx->d_potrf_scratch, per * want * sizeof(double)));
        ctx->potrf_scratch_jobs = want;
    }
    // per job: block width and count, and the scratch panel S with leading dimension m
    struct Blocked {
        int w = 0, n = 1;
        double *S = nullptr;
    };
    std::vector<Blocked> bl(act.size());
    size_t words = 0;
    int blocks = 1;
    for (size_t q = 0; q < act.size(); ++q) {
        const int m = act[q].m;
        bl[q].w = m;
        if (m <= kPotrfOuter) continue;
        bl[q].n = (int)ceil_div(m, kPotrfOuter);
        bl[q].w = (int)(ceil_div(ceil_div(m, bl[q].n), kBlk) * kBlk);
        bl[q].n = (int)ceil_div(m, bl[q].w);
        blocks = std::max(blocks, bl[q].n);
        words += (size_t)m * m;
    }
    if (blocks == 1) {
        potrf_cluster(ctx, s, act);
        return;
    }
    DevBuf buf(words * sizeof(double), s);
    PotrfEdges edges{};
    int nedge = 0, mmax = 0;
    words = 0;
    for (size_t q = 0; q < act.size(); ++q) {
        if (bl[q].n == 1) continue;
        const PotrfJob &J = act[q];
        bl[q].S = buf.as<double>() + words;
        words += (size_t)J.m * J.m;
        edges.e[nedge++] = PotrfEdge{J.A, J.X, bl[q].S, J.lda, J.ldx, J.m, J.m, bl[q].w};
        mmax = std::max(mmax, J.m);
    }
    launch(k_potrf_edges, dim3((unsigned)std::min(mmax, 256), (unsigned)nedge), 256, 0, s, edges);
    TLR_CHECK_LAUNCH();
    auto prob = [](const double *A, int lda, const double *B, int ldb, double *C, int ldc, int m, int n, int k) {
        GemmProb g{};
        g.A = A; g.lda = lda; g.B = B; g.ldb = ldb; g.C = C; g.ldc = ldc;
        g.m = m; g.n = n; g.k = k;
        return g;
    };
    for (int b = 0; b < blocks; ++b) {
        std::vector<PotrfJob> diag;
        std::vector<GemmProb> ga, gs;
        PotrfSubs subs{};
        int nsub = 0, ctas = 0;
        for (size_t q = 0; q < act.size(); ++q) {
            const PotrfJob &J = act[q];
            const Blocked &B = bl[q];
            if (b >= B.n) continue;
            const int p = b * B.w, w = std::min(B.w, J.m - p), e = p + w, rest = J.m - e;
            PotrfJob D = J;
            D.A = J.A + (int64_t)p * J.lda + p;
            D.X = J.X + (int64_t)p * J.ldx + p;
            D.m = w;
            D.row_base = J.row_base + p;
            diag.push_back(D);
            if (B.n == 1) continue;
            double *Lib = J.A + (int64_t)p * J.lda + e;
            subs.j[nsub++] = PotrfSub{D.A, D.X, Lib, B.S + p, J.X + p, J.lda, J.ldx, J.m, w, rest, p};
            ctas = std::max(ctas, (int)(ceil_div(rest, kSubVecs) + ceil_div(p, kSubVecs)));
            if (rest <= 0) continue;
            // S_ib, columns c0 .. c1: X_bb is zero above row c0
            for (int c0 = 0; c0 < w; c0 += kPotrfChunk) {
                const int c1 = std::min(w, c0 + kPotrfChunk);
                gs.push_back(prob(Lib + (int64_t)c0 * J.lda, J.lda, D.X + (int64_t)c0 * J.ldx + c0, J.ldx,
                                  B.S + (int64_t)(p + c0) * J.m + e, J.m, rest, c1 - c0, w - c0));
            }
            if (p > 0) gs.push_back(prob(Lib, J.lda, J.X + p, J.ldx, B.S + e, J.m, rest, p, w));
            // lower part of the trailing matrix; no chunk crosses a block
            // boundary, so that nothing above the diagonal blocks is written
            for (int c0 = e, c1; c0 < J.m; c0 = c1) {
                c1 = std::min({J.m, c0 + kPotrfChunk, (c0 / B.w + 1) * B.w});
                const double *Lc = J.A + (int64_t)p * J.lda + c0;
                ga.push_back(prob(Lc, J.lda, Lc, J.lda, J.A + (int64_t)c0 * J.lda + c0, J.lda, J.m - c0, c1 - c0, w));
            }
        }
        potrf_cluster(ctx, s, diag);
        launch(k_potrf_sub, dim3((unsigned)ctas, (unsigned)nsub), kSubThreads, 0, s, subs);
        TLR_CHECK_LAUNCH();
        gemm_batched_small(ctx, s, false, true, ga, -1.0, 1.0, true);  // trailing update
        gemm_batched_small(ctx, s, false, false, gs, -1.0, 1.0, true);  // S
    }
}

void potrf_inv(tlr_ctx *ctx, cudaStream_t s, double *A, int lda, int m, double *X, int ldx, long long row_base) {
    potrf_inv_batched(ctx, s, {PotrfJob{A, lda, m, X, ldx, nullptr, ctx->d_status, row_base}});
}

// acc[0] += sum_r log A[r, r]  (one block, fixed reduction order); if maxinv
// is not null, *maxinv = max(*maxinv, max_r 1 / A[r, r]^2) (the largest
// inverse squared pivot, i.e. the smallest conditional variance seen so far;
// positive doubles order like their bit patterns, so an integer atomicMax
// keeps the result independent of launch order).
__global__ void k_diag_logsum(const double *__restrict__ A, int lda, int m, double *acc,
                              const DevStatus *st, double *maxinv) {
    __shared__ double part[256], pmax[256];
    double s = 0.0, mx = 0.0;
    for (int r = threadIdx.x; r < m; r += blockDim.x) {
        const double d = A[(int64_t)r * lda + r];
        s += log(d);
        mx = fmax(mx, 1.0 / (d * d));
    }
    part[threadIdx.x] = s;
    pmax[threadIdx.x] = mx;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (threadIdx.x < h) {
            part[threadIdx.x] += part[threadIdx.x + h];
            pmax[threadIdx.x] = fmax(pmax[threadIdx.x], pmax[threadIdx.x + h]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0 && !st->code) {
        acc[0] += part[0];
        if (maxinv && pmax[0] > 0.0 && pmax[0] <= 1.7e308)
            atomicMax(reinterpret_cast<unsigned long long *>(maxinv), (unsigned long long)__double_as_longlong(pmax[0]));
    }
}

// acc[0] += sum v_r^2 (one block, fixed reduction order)
__global__ void k_sumsq(const double *__restrict__ v, int m, double *acc) {
    __shared__ double part[256];
    double s = 0.0;
    for (int r = threadIdx.x; r < m; r += blockDim.x) s += v[r] * v[r];
    part[threadIdx.x] = s;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (threadIdx.x < h) part[threadIdx.x] += part[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) acc[0] += part[0];
}

void diag_logsum(cudaStream_t s, const double *A, int lda, int m, double *acc, const DevStatus *st, double *maxinv) {
    launch(k_diag_logsum, 1, 256, 0, s, A, lda, m, acc, st, maxinv);
    TLR_CHECK_LAUNCH();
}

void sumsq(cudaStream_t s, const double *v, int m, double *acc) {
    launch(k_sumsq, 1, 256, 0, s, v, m, acc);
    TLR_CHECK_LAUNCH();
}

}  // namespace tlr
