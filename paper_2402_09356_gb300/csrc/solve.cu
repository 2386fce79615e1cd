// a5 on a kept factor: y = L^-1 z with the log-determinant and |y|^2 (Eq. 1.2),
// and z = L w.
//
// The factor is read once; its bytes are the floor (0.2 GB at n = 20,000: 30 us),
// and the FP64 pipe, one multiply-add per entry, is close behind (40 us).  What
// costs is the chain of the solve: tile column by tile column, and inside a
// diagonal tile block by block.  Per tile column three launches:
//   k_trsv      y_k <- L_kk^-1 y_k, one cluster, blocks of 32 rows whose
//               inverses were formed for all tiles by one launch at the start
//               (k_inv_blocks: a block's substitution is then one 32 x 32
//               product, three where its condition asks for a residual step,
//               not 32 dependent steps);
//   k_pair_dots c_ik = V_ik' y_k for all i > k, one warp a column of V;
//   k_pair_sub  y_i -= U_ik c_ik for all i > k.
// The product L w has no chain: one launch of k_pair_dots over all tiles, one
// of k_row_sums.  All descriptors go up once per call.  n = 20,000, tile 800: solve
// 42.4 -> 2.03 ms (k_trsv 55 us a tile, the two others 10 each), L w 1.46 -> 0.11.
#include <algorithm>

#include <cooperative_groups.h>

#include "common.cuh"
#include "dense.cuh"
#include "per_device.cuh"
#include "tlr_internal.cuh"

namespace tlr {

namespace cg = cooperative_groups;

namespace {

constexpr int kB = 32;             // rows of a diagonal block
constexpr int kThreads = 256, kWarps = kThreads / 32;
constexpr int kRows = 32;          // output rows a CTA
constexpr int kGroups = kThreads / kRows;

// One off-diagonal tile: U (m_i x r), V (m_k x r), both ld nb, and the place
// of its c = V' x among all of them.
struct Pair {
    const double *U, *V;
    int64_t off;
    int i, k, r, pad;
};

__device__ __forceinline__ int rows_of(int64_t n, int nb, int t) {
    const int64_t r = n - (int64_t)t * nb;
    return (int)(r < nb ? r : nb);
}

// Inverses X of the 32 x 32 diagonal blocks L (row major, zero right of the
// diagonal and past the tile) of every diagonal tile: one CTA a block.
// Column by column, M <- the elimination applied to the identity: row c is
// scaled by 1 / L_cc, the rows below it subtract their multiple.
// `fix`: whether a product with X needs its residual step in k_trsv, from the
// block's condition k = max_r (|X| |L| e)_r.  A product's error is up to k times
// substitution's; measured against extended precision over 640 blocks (nu 0.4
// to 2.5, beta 0.03 to 0.12) it is 0.6 to 0.7 times as large for k of 8 to 16,
// 0.8 to 0.9 for 16 to 32, 1.1 to 1.3 for 32 to 64, 1.9 to 2.2 for 64 to 128, 5 to 7 for 256
// to 1,024.  nu = 0.5: k is 16 in the middle, nu = 2.5: 520.
constexpr double kPlainCond = 24.0;
__global__ void __launch_bounds__(kThreads) k_inv_blocks(const double *__restrict__ D, int64_t n, int nb, int per_tile,
                                                          double *__restrict__ inv, int *__restrict__ fix) {
    __shared__ double L[kB][kB + 1], M[kB][kB + 1], rd[kB];
    __shared__ int s_fix;
    const int t = blockIdx.x / per_tile, b = blockIdx.x % per_tile, tid = threadIdx.x;
    const int m = rows_of(n, nb, t), p = b * kB, w = min(kB, m - p);
    double *out = inv + (int64_t)blockIdx.x * kB * kB;
    if (w <= 0) return;
    const double *A = D + (int64_t)t * nb * nb + (int64_t)p * nb + p;
    for (int e = tid; e < kB * kB; e += kThreads) {
        const int r = e % kB, c = e / kB;
        L[r][c] = r < w && c <= r ? A[(int64_t)c * nb + r] : 0.0;
        M[r][c] = r == c ? 1.0 : 0.0;
    }
    __syncthreads();
    if (tid < w) rd[tid] = 1.0 / L[tid][tid];
    if (tid == 0) s_fix = 0;
    __syncthreads();
    const int r = tid >> 3, q = tid & 7;
    for (int c = 0; c < w; ++c) {
        if (tid <= c) M[c][tid] *= rd[c];
        __syncthreads();
        if (r > c && r < w) {
            const double l = L[r][c];
#pragma unroll
            for (int k = 0; k < kB / 8; ++k)
                if (q + 8 * k <= c) M[r][q + 8 * k] = fma(-l, M[c][q + 8 * k], M[r][q + 8 * k]);
        }
        __syncthreads();
    }
    for (int e = tid; e < kB * kB; e += kThreads) {
        const int i = e / kB, c = e % kB;
        out[e] = i < w && c <= i ? M[i][c] : 0.0;
    }
    // the condition, eight lanes a row
    auto row_sum = [](double v) {
#pragma unroll
        for (int o = 4; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
        return v;
    };
    double v = 0.0;
    for (int c = q; c <= r; c += 8) v += fabs(L[r][c]);
    v = row_sum(v);
    if (q == 0) rd[r] = v;
    __syncthreads();
    v = 0.0;
    for (int c = q; c <= r; c += 8) v = fma(fabs(M[r][c]), rd[c], v);
    v = row_sum(v);
    if (r < w && !(v <= kPlainCond)) s_fix = 1;
    __syncthreads();
    if (tid == 0) fix[blockIdx.x] = s_fix;
}

// x <- L^-1 x for one diagonal tile (m <= 1024, ld ldl) by one cluster: CTA
// `rank` owns the blocks rank, rank + kCl, ... of the right-hand side, each
// kept by kThreads / kOwn threads (four or two a row).  Step b: the owner
// multiplies its block by the block's inverse, corrects the product by its
// residual, y += L_bb^-1 (x - L_bb y), where fix[b] asks for it, and stores the
// 32 values into every CTA; after one cluster barrier every CTA subtracts L's
// block column b times them from its blocks.  (Without the correction the
// right-hand sides of a smooth field, whose y is far smaller than |L^-1| |x|, had
// 2 to 50 times the error of substitution; with it, none of that.  It takes 36
// us of a tile of 800 if every block asks.)  The entries of block columns b + 1
// and b + 2 are on their way to registers meanwhile (the tile comes from HBM).
// Bound by the chain of a step: barrier, update of the next block, its product
// or three.
template <int kCl>
__global__ void __launch_bounds__(kThreads) k_trsv(const double *__restrict__ L, int ldl, int m,
                                                    const double *__restrict__ inv, const int *__restrict__ fix,
                                                    double *__restrict__ x) {
    constexpr int kOwn = kB / kCl;                 // blocks a CTA: at most 32 blocks in a tile
    constexpr int kQ = kThreads / kOwn / kB;       // threads a row
    constexpr int kN = kB / kQ;                    // columns a thread
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), tid = threadIdx.x;
    const int o = tid / (kThreads / kOwn), r = tid % (kThreads / kOwn) / kQ, q = tid % kQ;
    const int I = rank + o * kCl, row = I * kB + r;  // the thread's block and row
    __shared__ double rhs[kOwn][kB], own[2][kOwn][kB], xs[2][kB];
    const int nblk = (m + kB - 1) / kB;
    const bool correct = I < nblk && fix[I];  // the same for the block's threads
    if (q == 0) rhs[o][r] = row < m ? x[row] : 0.0;
    double a[2][kN], d[kN], g[kN];
    auto load = [&](int b, double (&v)[kN]) {  // L's block column b in the thread's row
        const bool in = b < I && row < m;
#pragma unroll
        for (int k = 0; k < kN; ++k) v[k] = in ? L[(int64_t)(b * kB + q + kQ * k) * ldl + row] : 0.0;
    };
    auto reduce = [](double v) {
#pragma unroll
        for (int s = kQ / 2; s; s >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, s);
        return v;
    };
#pragma unroll
    for (int k = 0; k < kN; ++k) {  // row r of the block's inverse and of the block
        const int c = q + kQ * k;
        d[k] = I < nblk ? inv[(int64_t)I * kB * kB + r * kB + c] : 0.0;
        g[k] = correct && row < m && c <= r ? L[(int64_t)(I * kB + c) * ldl + row] : 0.0;
    }
    // the thread's row of a block times entries 0 .. last of a vector in shared
    // memory (the others count as zero whatever they hold: an infinite or NaN
    // entry of the right-hand side leaves the rows above it as they are)
    auto times = [&](const double (&v)[kN], const double *w, int last) {
        double s0 = 0.0, s1 = 0.0;
#pragma unroll
        for (int k = 0; k < kN; k += 2) {
            const int c = q + kQ * k;
            const double w0 = w[c], w1 = w[c + kQ];  // loaded whatever c is: a load behind a test is a branch
            s0 = fma(v[k], c <= last ? w0 : 0.0, s0);
            s1 = fma(v[k + 1], c + kQ <= last ? w1 : 0.0, s1);
        }
        return reduce(s0 + s1);
    };
    auto block_sync = [&] { asm volatile("bar.sync %0, %1;" ::"r"(o + 1), "n"(kThreads / kOwn) : "memory"); };
    load(0, a[0]);
    load(1, a[1]);
    cl.sync();  // every CTA has started (its shared memory is written below)
    auto step = [&](int b, double (&v)[kN]) {
        if (b == I) {  // uniform over the warps of the block's threads
            double s = times(d, rhs[o], r);
            if (correct) {
                if (q == 0) own[0][o][r] = s;
                block_sync();
                const double t = times(g, own[0][o], r);
                if (q == 0) own[1][o][r] = rhs[o][r] - t;
                block_sync();
                const double e = times(d, own[1][o], r);
                if ((__double2hiint(e) & 0x7FF00000) != 0x7FF00000) s += e;
            }
#pragma unroll
            for (int k = q; k < kCl; k += kQ) cl.map_shared_rank(&xs[b & 1][0], k)[r] = s;
            if (q == 0 && row < m) x[row] = s;
        }
        cl.sync();
        if (b < I) {
            const double s = times(v, xs[b & 1], kB);
            if (q == 0) rhs[o][r] -= s;
        }
        load(b + 2, v);
        __syncthreads();
    };
    for (int b = 0; b < nblk; b += 2) {
        step(b, a[0]);
        if (b + 1 < nblk) step(b + 1, a[1]);
    }
}

// c = V' x of the pairs p0 + blockIdx.y: eight columns a CTA, one a warp.
__global__ void __launch_bounds__(kThreads) k_pair_dots(const Pair *__restrict__ pairs, int p0, int64_t n, int nb,
                                                         const double *__restrict__ x, double *__restrict__ c) {
    const Pair P = pairs[p0 + blockIdx.y];
    const int lane = threadIdx.x & 31, col = blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (col >= P.r) return;
    const double *v = P.V + (int64_t)col * nb, *y = x + (int64_t)P.k * nb;
    const int m = rows_of(n, nb, P.k);
    double s0 = 0.0, s1 = 0.0;
    int i = lane;
#pragma unroll 4
    for (; i + 32 < m; i += 64) {
        s0 = fma(v[i], y[i], s0);
        s1 = fma(v[i + 32], y[i + 32], s1);
    }
    if (i < m) s0 = fma(v[i], y[i], s0);
    s0 += s1;
#pragma unroll
    for (int o = 16; o; o >>= 1) s0 += __shfl_xor_sync(0xFFFFFFFFu, s0, o);
    if (lane == 0) c[P.off + col] = s0;
}

// Row `row` of A (m x k, ld lda) times v, columns g, g + kGroups, ...
__device__ __forceinline__ double row_part(const double *__restrict__ A, int lda, int k, int g,
                                           const double *__restrict__ v) {
    double s0 = 0.0, s1 = 0.0;
    int j = g;
#pragma unroll 4
    for (; j + kGroups < k; j += 2 * kGroups) {
        s0 = fma(A[(int64_t)j * lda], v[j], s0);
        s1 = fma(A[(int64_t)(j + kGroups) * lda], v[j + kGroups], s1);
    }
    if (j < k) s0 = fma(A[(int64_t)j * lda], v[j], s0);
    return s0 + s1;
}

__device__ __forceinline__ double sum_parts(const double (*part)[kRows], int u) {
    return ((part[0][u] + part[1][u]) + (part[2][u] + part[3][u])) + ((part[4][u] + part[5][u]) + (part[6][u] + part[7][u]));
}

// y_i -= U_ik c_ik for the pairs p0 + blockIdx.y: 32 rows a CTA, the columns
// split over eight threads a row.
__global__ void __launch_bounds__(kThreads) k_pair_sub(const Pair *__restrict__ pairs, int p0, int64_t n, int nb,
                                                        const double *__restrict__ c, double *__restrict__ y) {
    __shared__ double part[kGroups][kRows];
    const Pair P = pairs[p0 + blockIdx.y];
    const int g = threadIdx.x / kRows, u = threadIdx.x % kRows, row = blockIdx.x * kRows + u;
    const int m = rows_of(n, nb, P.i);
    part[g][u] = row < m ? row_part(P.U + row, nb, P.r, g, c + P.off) : 0.0;
    __syncthreads();
    if (g == 0 && row < m) y[(int64_t)P.i * nb + row] -= sum_parts(part, u);
}

// z_i = D_i w_i + sum_k U_ik c_ik: blockIdx.y = i, 32 rows a CTA; the pairs of
// row i are first[i] .. first[i + 1].  D's columns past the row are zero and
// left out.
__global__ void __launch_bounds__(kThreads) k_row_sums(const Pair *__restrict__ pairs, const int *__restrict__ first,
                                                        int64_t n, int nb, const double *__restrict__ D,
                                                        const double *__restrict__ w, const double *__restrict__ c,
                                                        double *__restrict__ z) {
    __shared__ double part[kGroups][kRows];
    const int i = blockIdx.y, g = threadIdx.x / kRows, u = threadIdx.x % kRows, row = blockIdx.x * kRows + u;
    const int m = rows_of(n, nb, i);
    double s = 0.0;
    if (row < m) {
        s = row_part(D + (int64_t)i * nb * nb + row, nb, row + 1, g, w + (int64_t)i * nb);
        for (int p = first[i]; p < first[i + 1]; ++p) {
            const Pair P = pairs[p];
            s += row_part(P.U + row, nb, P.r, g, c + P.off);
        }
    }
    part[g][u] = s;
    __syncthreads();
    if (g == 0 && row < m) z[(int64_t)i * nb + row] = sum_parts(part, u);
}

// Per tile: sum log D_rr and |y|^2 (fixed reduction order), then their sums
// over the tiles in order, added to acc.
__global__ void __launch_bounds__(kThreads) k_tile_sums(const double *__restrict__ D, int64_t n, int nb,
                                                         const double *__restrict__ y, double *__restrict__ part) {
    __shared__ double sl[kThreads], sq[kThreads];
    const int t = blockIdx.x, tid = threadIdx.x, m = rows_of(n, nb, t);
    double l = 0.0, s = 0.0;
    for (int r = tid; r < m; r += kThreads) {
        l += log(D[(int64_t)t * nb * nb + (int64_t)r * nb + r]);
        const double v = y[(int64_t)t * nb + r];
        s += v * v;
    }
    sl[tid] = l;
    sq[tid] = s;
    __syncthreads();
    for (int h = kThreads / 2; h > 0; h >>= 1) {
        if (tid < h) {
            sl[tid] += sl[tid + h];
            sq[tid] += sq[tid + h];
        }
        __syncthreads();
    }
    if (tid == 0) {
        part[2 * t] = sl[0];
        part[2 * t + 1] = sq[0];
    }
}
__global__ void k_sum_tiles(const double *__restrict__ part, int nt, double *__restrict__ acc) {
    double s = acc[threadIdx.x];
    for (int t = 0; t < nt; ++t) s += part[2 * t + threadIdx.x];
    acc[threadIdx.x] = s;
}

// The tiles of nonzero rank, by column (by_row: by row), with the places of
// their c = V' x and the first pair of every column (row).
struct PairList {
    std::vector<Pair> pairs;
    std::vector<int> first, rmax;
    int64_t total = 0;
};
PairList list_pairs(const tlr_mat *M, bool by_row) {
    const int nt = M->nt;
    PairList L;
    for (int a = 0; a < nt; ++a) {
        L.first.push_back((int)L.pairs.size());
        int most = 0;
        for (int b = by_row ? 0 : a + 1; b < (by_row ? a : nt); ++b) {
            const int i = by_row ? a : b, k = by_row ? b : a, r = M->h_ranks[(size_t)i * nt + k];
            if (r <= 0) continue;
            const int64_t at = slot_col(M, i, k) * M->nb;
            L.pairs.push_back(Pair{M->U + at, M->V + at, L.total, i, k, r, 0});
            L.total += r;
            most = std::max(most, r);
        }
        L.rmax.push_back(most);
    }
    L.first.push_back((int)L.pairs.size());
    return L;
}

// Host data on the device for the kernels of stream s: through the pinned ring
// where it is small, else its own buffer.
const void *upload(tlr_ctx *ctx, cudaStream_t s, const void *data, size_t bytes, DevBuf &own) {
    if (bytes <= ((size_t)1 << 20)) return stage_push(ctx, data, bytes, s);
    own.alloc(bytes, s);
    TLR_CUDA_TRY(cudaMemcpyAsync(own.as<char>(), data, bytes, cudaMemcpyHostToDevice, s));
    TLR_CUDA_TRY(cudaStreamSynchronize(s));
    return own.as<char>();
}

// Whether clusters of 16 CTAs of k_trsv run on the current device.
bool trsv16_ok() {
    static PerDevice<bool> per_device;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    return per_device.get(dev, [] {
        bool ok = false;
        if (cudaFuncSetAttribute(k_trsv<16>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(16);
            cfg.blockDim = dim3(kThreads);
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = 16;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            int nc = 0;
            ok = cudaOccupancyMaxActiveClusters(&nc, k_trsv<16>, &cfg) == cudaSuccess && nc > 0;
        }
        cudaGetLastError();  // clear any error of the queries
        return ok;
    });
}

// Pairs a launch's grid may hold in its second dimension.
constexpr int kMaxGridY = 65535;

}  // namespace

// y = L^-1 z tile by tile; acc[0] += sum log L_ii, acc[1] += |y|^2.
void forward_solve(tlr_ctx *ctx, cudaStream_t st, const tlr_mat *M, const double *z, double *y, double *acc) {
    const int nt = M->nt, nb = M->nb, per_tile = (int)ceil_div(nb, kB);
    const int64_t n = M->n;
    if (y != z) TLR_CUDA_TRY(cudaMemcpyAsync(y, z, n * sizeof(double), cudaMemcpyDeviceToDevice, st));
    const PairList L = list_pairs(M, false);
    DevBuf own;
    const Pair *pairs = L.pairs.empty()
                            ? nullptr
                            : (const Pair *)upload(ctx, st, L.pairs.data(), L.pairs.size() * sizeof(Pair), own);
    DevBuf inv((size_t)nt * per_tile * kB * kB * sizeof(double), st);
    DevBuf cb((size_t)std::max<int64_t>(L.total, 1) * sizeof(double), st), part((size_t)2 * nt * sizeof(double), st);
    double *c = cb.as<double>();
    DevBuf fixb((size_t)nt * per_tile * sizeof(int), st);
    launch(k_inv_blocks, (unsigned)(nt * per_tile), kThreads, 0, st, M->D, n, nb, per_tile, inv.as<double>(),
           fixb.as<int>());
    TLR_CHECK_LAUNCH();
    const bool big = trsv16_ok();
    for (int k = 0; k < nt; ++k) {
        const double *D = M->D + (int64_t)k * nb * nb, *Di = inv.as<double>() + (int64_t)k * per_tile * kB * kB;
        const int *fix = fixb.as<int>() + (int64_t)k * per_tile;
        if (big) launch_clustered(k_trsv<16>, 16, 1, kThreads, 0, st, D, nb, tile_rows(n, nb, k), Di, fix,
                                  y + (int64_t)k * nb);
        else launch_clustered(k_trsv<8>, 8, 1, kThreads, 0, st, D, nb, tile_rows(n, nb, k), Di, fix,
                                  y + (int64_t)k * nb);
        const int p1 = L.first[(size_t)k + 1];
        for (int p = L.first[(size_t)k]; p < p1; p += kMaxGridY) {
            const unsigned cnt = (unsigned)std::min(kMaxGridY, p1 - p);
            launch(k_pair_dots, dim3((unsigned)ceil_div(L.rmax[(size_t)k], kWarps), cnt), kThreads, 0, st, pairs, p, n,
                   nb, y, c);
            launch(k_pair_sub, dim3((unsigned)ceil_div(nb, kRows), cnt), kThreads, 0, st, pairs, p, n, nb, c, y);
        }
        TLR_CHECK_LAUNCH();
    }
    launch(k_tile_sums, (unsigned)nt, kThreads, 0, st, M->D, n, nb, y, part.as<double>());
    launch(k_sum_tiles, 1, 2, 0, st, part.as<double>(), nt, acc);
    TLR_CHECK_LAUNCH();
}

// z = L w
void lmul(tlr_ctx *ctx, cudaStream_t st, const tlr_mat *M, const double *w, double *z) {
    const int nt = M->nt, nb = M->nb;
    const int64_t n = M->n;
    const PairList L = list_pairs(M, true);
    DevBuf own, ownf;
    const Pair *pairs = L.pairs.empty()
                            ? nullptr
                            : (const Pair *)upload(ctx, st, L.pairs.data(), L.pairs.size() * sizeof(Pair), own);
    const int *first = (const int *)upload(ctx, st, L.first.data(), L.first.size() * sizeof(int), ownf);
    DevBuf cb((size_t)std::max<int64_t>(L.total, 1) * sizeof(double), st);
    double *c = cb.as<double>();
    const int rmax = *std::max_element(L.rmax.begin(), L.rmax.end());
    for (int p = 0; p < (int)L.pairs.size(); p += kMaxGridY)
        launch(k_pair_dots, dim3((unsigned)ceil_div(rmax, kWarps), (unsigned)std::min(kMaxGridY, (int)L.pairs.size() - p)),
               kThreads, 0, st, pairs, p, n, nb, w, c);
    launch(k_row_sums, dim3((unsigned)ceil_div(nb, kRows), (unsigned)nt), kThreads, 0, st, pairs, first, n, nb, M->D, w,
           c, z);
    TLR_CHECK_LAUNCH();
}

}  // namespace tlr
