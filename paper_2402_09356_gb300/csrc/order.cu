// a1: spatial ordering of the locations (Sec. 3).  Up to the sizes of the last
// section of this file the whole ordering runs on one thread-block cluster;
// what follows is the layout above them, a launch per pass.
//
// Morton / Hilbert / random: one thread per point computes a 32-bit key
// (Sec. 3.1 "Encoding"), then a stable LSD radix sort orders (key, index)
// pairs (Sec. 3.1 "Sorting"; stability breaks ties by original index).
//
// KD-tree (Sec. 3.2): built level by level.  The segment structure of every
// level depends on n only (a node of m points has children of ceil(m/2) and
// floor(m/2) points), so each level is: per-segment coordinate ranges
// (atomics on order-preserving integer images of the doubles), choice of the
// wider dimension, and one stable radix sort of (segment, rank of the point
// along the chosen dimension).  The ranks come from two initial global sorts
// by (x, index) and (y, index), so sorting by rank inside a segment is sorting
// by (coordinate, index).
//
// Max-min (Sec. 3.3.1): one launch per selected point; every block updates
// the minimum squared distances of its points to the newest selection and
// publishes its (max, lowest index) partial; the next launch reduces the
// partials (double-buffered) to find the next point.  All distance arithmetic
// uses explicitly rounded intrinsics so that no multiply-add is contracted.
#include <algorithm>
#include <mutex>

#include <cooperative_groups.h>

#include "common.cuh"
#include "per_device.cuh"
#include "tlr_internal.cuh"

namespace tlr {

namespace cg = cooperative_groups;

static constexpr int kSortThreads = 256;
static constexpr int kSortItems = 16;  // keys per thread per block
static constexpr int kSortTile = kSortThreads * kSortItems;

// ---------------------------------------------------------------- key helpers
__device__ __forceinline__ uint32_t quantize16(double v) {
    double c = fmin(fmax(v, 0.0), 1.0);
    return (uint32_t)rint(__dmul_rn(c, 65535.0));  // round half to even
}

__device__ __forceinline__ uint32_t spread_bits(uint32_t v) {
    v &= 0xFFFFu;
    v = (v | (v << 8)) & 0x00FF00FFu;
    v = (v | (v << 4)) & 0x0F0F0F0Fu;
    v = (v | (v << 2)) & 0x33333333u;
    v = (v | (v << 1)) & 0x55555555u;
    return v;
}

// Hilbert index of a cell of the 2^16 x 2^16 grid, orientation of Figure 3:
// quadrants visited lower-left, upper-left, upper-right, lower-right.  The
// frame of the current sub-square is tracked as (swap, complement) flags:
// entering the lower-left quadrant transposes the frame, entering the
// lower-right quadrant transposes and complements it.
__device__ __forceinline__ uint32_t hilbert16(uint32_t qx, uint32_t qy) {
    uint32_t d = 0;
    bool sw = false, cp = false;
#pragma unroll
    for (int b = 15; b >= 0; --b) {
        uint32_t bx = (qx >> b) & 1u, by = (qy >> b) & 1u;
        if (cp) { bx ^= 1u; by ^= 1u; }
        if (sw) { uint32_t t = bx; bx = by; by = t; }
        uint32_t q = (bx << 1) | (bx ^ by);
        d = (d << 2) | q;
        if (q == 0u) sw = !sw;
        else if (q == 3u) { sw = !sw; cp = !cp; }
    }
    return d;
}

__device__ __forceinline__ uint64_t splitmix64(uint64_t s) {
    uint64_t z = s + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Order-preserving unsigned image of a double (total order of finite values).
__device__ __forceinline__ uint64_t dkey(double v) {
    uint64_t b = (uint64_t)__double_as_longlong(v);
    return (b & 0x8000000000000000ull) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double dkey_inv(uint64_t k) {
    uint64_t b = (k & 0x8000000000000000ull) ? (k & 0x7FFFFFFFFFFFFFFFull) : ~k;
    return __longlong_as_double((long long)b);
}

__global__ void k_sfc_keys(const double *__restrict__ xy, int64_t n, int method, uint64_t seed,
                           uint32_t *__restrict__ keys, uint32_t *__restrict__ vals) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t k;
    if (method == TLR_ORDER_RANDOM) {
        k = (uint32_t)(splitmix64(seed ^ (uint64_t)i) >> 32);
    } else {
        uint32_t qx = quantize16(xy[i]), qy = quantize16(xy[n + i]);
        k = (method == TLR_ORDER_MORTON) ? (spread_bits(qx) | (spread_bits(qy) << 1))
                                         : hilbert16(qx, qy);
    }
    keys[i] = k;
    vals[i] = (uint32_t)i;
}

// ------------------------------------------------------------- radix sort
template <typename K>
__global__ void k_radix_hist(const K *__restrict__ keys, int64_t n, int shift,
                             uint32_t *__restrict__ hist, int nblk) {
    __shared__ uint32_t sh[256];
    sh[threadIdx.x] = 0;
    __syncthreads();
    int64_t base = (int64_t)blockIdx.x * kSortTile;
    for (int c = 0; c < kSortItems; ++c) {
        int64_t i = base + (int64_t)c * kSortThreads + threadIdx.x;
        if (i < n) atomicAdd(&sh[(uint32_t)(keys[i] >> shift) & 0xFFu], 1u);
    }
    __syncthreads();
    hist[(int64_t)threadIdx.x * nblk + blockIdx.x] = sh[threadIdx.x];
}

// Exclusive scan of `len` uint32 in one block of 1024 threads.
__global__ void k_scan_exclusive(uint32_t *__restrict__ a, int64_t len) {
    __shared__ uint32_t part[1024];
    int t = threadIdx.x;
    int64_t chunk = (len + 1023) / 1024;
    int64_t lo = t * chunk, hi = lo + chunk < len ? lo + chunk : len;
    uint32_t s = 0;
    for (int64_t i = lo; i < hi; ++i) s += a[i];
    part[t] = s;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {  // Hillis-Steele inclusive scan
        uint32_t v = t >= off ? part[t - off] : 0u;
        __syncthreads();
        part[t] += v;
        __syncthreads();
    }
    uint32_t run = t ? part[t - 1] : 0u;
    for (int64_t i = lo; i < hi; ++i) {
        uint32_t v = a[i];
        a[i] = run;
        run += v;
    }
}

template <typename K>
__global__ void k_radix_scatter(const K *__restrict__ keys, const uint32_t *__restrict__ vals,
                                int64_t n, int shift, const uint32_t *__restrict__ hist, int nblk,
                                K *__restrict__ keys_out, uint32_t *__restrict__ vals_out) {
    __shared__ uint32_t s_base[256];
    __shared__ uint32_t s_cnt[kSortThreads / 32][256];
    __shared__ uint32_t s_tot[256];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    s_base[tid] = hist[(int64_t)tid * nblk + blockIdx.x];
    int64_t base = (int64_t)blockIdx.x * kSortTile;
    for (int c = 0; c < kSortItems; ++c) {
#pragma unroll
        for (int w = 0; w < kSortThreads / 32; ++w) s_cnt[w][tid] = 0;
        __syncthreads();
        int64_t i = base + (int64_t)c * kSortThreads + tid;
        bool valid = i < n;
        K k = valid ? keys[i] : K(0);
        uint32_t d = valid ? ((uint32_t)(k >> shift) & 0xFFu) : 0xFFFFFFFFu;
        uint32_t peers = __match_any_sync(0xFFFFFFFFu, d);
        uint32_t lower = __popc(peers & ((1u << lane) - 1u));
        if (valid && lower == 0) s_cnt[warp][d] = __popc(peers);
        __syncthreads();
        uint32_t run = 0;
#pragma unroll
        for (int w = 0; w < kSortThreads / 32; ++w) {
            uint32_t t = s_cnt[w][tid];
            s_cnt[w][tid] = run;
            run += t;
        }
        s_tot[tid] = run;
        __syncthreads();
        if (valid) {
            uint32_t pos = s_base[d] + s_cnt[warp][d] + lower;
            keys_out[pos] = k;
            vals_out[pos] = vals[i];
        }
        __syncthreads();
        s_base[tid] += s_tot[tid];
    }
}

// Stable sort of (key, val) pairs by the low `bits` bits of the key.  The
// result ends in (*keys, *vals) (the buffers are swapped as passes proceed).
template <typename K>
static void radix_sort(K **keys, uint32_t **vals, K **keys_tmp, uint32_t **vals_tmp, int64_t n,
                       int bits, uint32_t *hist, cudaStream_t s) {
    if (n <= 1) return;
    int nblk = (int)ceil_div(n, kSortTile);
    for (int shift = 0; shift < bits; shift += 8) {
        launch(k_radix_hist<K>, nblk, kSortThreads, 0, s, *keys, n, shift, hist, nblk);
        launch(k_scan_exclusive, 1, 1024, 0, s, hist, (int64_t)256 * nblk);
        launch(k_radix_scatter<K>, nblk, kSortThreads, 0, s, *keys, *vals, n, shift, hist, nblk,
                                                          *keys_tmp, *vals_tmp);
        TLR_CHECK_LAUNCH();
        std::swap(*keys, *keys_tmp);
        std::swap(*vals, *vals_tmp);
    }
}

static size_t hist_words(int64_t n) { return (size_t)256 * (size_t)ceil_div(n > 0 ? n : 1, kSortTile); }

// ------------------------------------------------------------- outputs
__global__ void k_perm_out(const uint32_t *__restrict__ vals, int64_t n, int64_t *__restrict__ perm) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) perm[i] = (int64_t)vals[i];
}

__global__ void k_iota32(int64_t n, uint32_t *__restrict__ v) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) v[i] = (uint32_t)i;
}

__global__ void k_iota(int64_t n, int64_t *__restrict__ perm) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) perm[i] = i;
}

__global__ void k_permute_xy(const double *__restrict__ xy, const int64_t *__restrict__ perm,
                             int64_t n, int quantize, double *__restrict__ out) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    int64_t p = perm[k];
    double x = xy[p], y = xy[n + p];
    if (quantize) {
        x = __ddiv_rn((double)quantize16(x), 65535.0);
        y = __ddiv_rn((double)quantize16(y), 65535.0);
    }
    out[k] = x;
    out[n + k] = y;
}

__global__ void k_gather(const int64_t *__restrict__ perm, const double *__restrict__ src,
                         int64_t n, double *__restrict__ dst) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    int64_t p = perm[k];
    dst[k] = (p >= 0 && p < n) ? src[p] : __longlong_as_double(0x7FF8000000000000ll);
}

// ------------------------------------------------------------- KD-tree
__global__ void k_coord_keys(const double *__restrict__ c, int64_t n, uint64_t *__restrict__ keys,
                             uint32_t *__restrict__ vals) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    keys[i] = dkey(c[i]);
    vals[i] = (uint32_t)i;
}

// rank[vals[p]] = p: the position of each point in the (coordinate, index) order
__global__ void k_invert(const uint32_t *__restrict__ vals, int64_t n, uint32_t *__restrict__ rank) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n) rank[vals[p]] = (uint32_t)p;
}

__device__ __forceinline__ int seg_of(const int64_t *__restrict__ starts, int nseg, int64_t p) {
    int lo = 0, hi = nseg - 1;  // last start <= p
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (starts[mid] <= p) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__global__ void k_kd_init_ranges(int nseg, unsigned long long *__restrict__ rng) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nseg) return;
    rng[4 * s + 0] = ~0ull;  // min x
    rng[4 * s + 1] = 0ull;   // max x
    rng[4 * s + 2] = ~0ull;  // min y
    rng[4 * s + 3] = 0ull;   // max y
}

__global__ void k_kd_ranges(const double *__restrict__ xy, int64_t n, const uint32_t *__restrict__ order,
                            const int64_t *__restrict__ starts, int nseg,
                            unsigned long long *__restrict__ rng) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    int s = seg_of(starts, nseg, p);
    uint32_t i = order[p];
    unsigned long long kx = dkey(xy[i]), ky = dkey(xy[n + i]);
    atomicMin(&rng[4 * s + 0], kx);
    atomicMax(&rng[4 * s + 1], kx);
    atomicMin(&rng[4 * s + 2], ky);
    atomicMax(&rng[4 * s + 3], ky);
}

__global__ void k_kd_keys(int64_t n, const uint32_t *__restrict__ order, const int64_t *__restrict__ starts,
                          int nseg, const unsigned long long *__restrict__ rng,
                          const uint32_t *__restrict__ rank_x, const uint32_t *__restrict__ rank_y,
                          int rbits, uint64_t *__restrict__ keys) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    int s = seg_of(starts, nseg, p);
    double rx = __dsub_rn(dkey_inv(rng[4 * s + 1]), dkey_inv(rng[4 * s + 0]));
    double ry = __dsub_rn(dkey_inv(rng[4 * s + 3]), dkey_inv(rng[4 * s + 2]));
    uint32_t i = order[p];
    uint32_t r = (rx >= ry) ? rank_x[i] : rank_y[i];  // equal ranges: x
    keys[p] = ((uint64_t)s << rbits) | (uint64_t)r;
}

// ------------------------------------------------------------- max-min
__device__ __forceinline__ double sqdist(double ax, double ay, double bx, double by) {
    double dx = __dsub_rn(ax, bx), dy = __dsub_rn(ay, by);
    return __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
}

struct MaxLoc {
    double v;
    long long i;
};

__device__ __forceinline__ bool better_max(double v, long long i, double bv, long long bi) {
    return v > bv || (v == bv && i < bi);
}
__device__ __forceinline__ bool better_min(double v, long long i, double bv, long long bi) {
    return v < bv || (v == bv && i < bi);
}

// Block reduction of (value, index) pairs; `is_max` picks max (else min),
// ties to the lower index.  Result valid in thread 0.
__device__ MaxLoc block_argext(double v, long long i, bool is_max) {
    __shared__ double sv[32];
    __shared__ long long si[32];
    for (int off = 16; off; off >>= 1) {
        double ov = __shfl_down_sync(0xFFFFFFFFu, v, off);
        long long oi = __shfl_down_sync(0xFFFFFFFFu, i, off);
        if (is_max ? better_max(ov, oi, v, i) : better_min(ov, oi, v, i)) { v = ov; i = oi; }
    }
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0) { sv[w] = v; si[w] = i; }
    __syncthreads();
    if (w == 0) {
        v = lane < nw ? sv[lane] : (is_max ? -INFINITY : INFINITY);
        i = lane < nw ? si[lane] : 0x7FFFFFFFFFFFFFFFll;
        for (int off = 16; off; off >>= 1) {
            double ov = __shfl_down_sync(0xFFFFFFFFu, v, off);
            long long oi = __shfl_down_sync(0xFFFFFFFFu, i, off);
            if (is_max ? better_max(ov, oi, v, i) : better_min(ov, oi, v, i)) { v = ov; i = oi; }
        }
    }
    return MaxLoc{v, i};
}

// Bounding box of all points (one block; grid-stride).
__global__ void k_bbox(const double *__restrict__ xy, int64_t n, double *__restrict__ bbox) {
    double mnx = INFINITY, mxx = -INFINITY, mny = INFINITY, mxy = -INFINITY;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
        double x = xy[i], y = xy[n + i];
        mnx = fmin(mnx, x); mxx = fmax(mxx, x);
        mny = fmin(mny, y); mxy = fmax(mxy, y);
    }
    MaxLoc a = block_argext(-mnx, 0, true);
    double r0 = -a.v;
    __syncthreads();
    MaxLoc b = block_argext(mxx, 0, true);
    __syncthreads();
    MaxLoc c = block_argext(-mny, 0, true);
    __syncthreads();
    MaxLoc d = block_argext(mxy, 0, true);
    if (threadIdx.x == 0) {
        bbox[0] = __dmul_rn(__dadd_rn(r0, b.v), 0.5);
        bbox[1] = __dmul_rn(__dadd_rn(-c.v, d.v), 0.5);
    }
}

// First point: nearest to the bounding-box centre (partials per block).
__global__ void k_maxmin_first(const double *__restrict__ xy, int64_t n, const double *__restrict__ ctr,
                               double *__restrict__ pv, long long *__restrict__ pi) {
    double cx = ctr[0], cy = ctr[1];
    double bv = INFINITY;
    long long bi = 0x7FFFFFFFFFFFFFFFll;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        double d = sqdist(xy[i], xy[n + i], cx, cy);
        if (better_min(d, i, bv, bi)) { bv = d; bi = i; }
    }
    MaxLoc r = block_argext(bv, bi, false);
    if (threadIdx.x == 0) { pv[blockIdx.x] = r.v; pi[blockIdx.x] = r.i; }
}

// One selection step.  Reduces the previous partials (min for the first
// step, max afterwards) to the point p taken at step k, records it, then
// updates the block's minimum distances and writes new partials.
__global__ void k_maxmin_step(const double *__restrict__ xy, int64_t n, int64_t k, int first,
                              const double *__restrict__ in_v, const long long *__restrict__ in_i,
                              double *__restrict__ out_v, long long *__restrict__ out_i,
                              double *__restrict__ mind, int64_t *__restrict__ perm) {
    __shared__ long long s_p;
    int nb = gridDim.x;
    double v = first ? INFINITY : -INFINITY;
    long long ii = 0x7FFFFFFFFFFFFFFFll;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        double ov = in_v[b];
        long long oi = in_i[b];
        if (first ? better_min(ov, oi, v, ii) : better_max(ov, oi, v, ii)) { v = ov; ii = oi; }
    }
    MaxLoc r = block_argext(v, ii, !first);
    if (threadIdx.x == 0) s_p = r.i;
    __syncthreads();
    long long p = s_p;
    if (p < 0 || p >= n) p = 0;  // only reachable with non-finite coordinates
    if (blockIdx.x == 0 && threadIdx.x == 0) perm[k] = p;
    double px = xy[p], py = xy[n + p];
    double bv = -INFINITY;
    long long bi = 0x7FFFFFFFFFFFFFFFll;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        double m = mind[i];
        if (i == p) m = -1.0;                      // taken
        else if (m >= 0.0) m = fmin(m, sqdist(xy[i], xy[n + i], px, py));
        mind[i] = m;
        if (better_max(m, i, bv, bi)) { bv = m; bi = i; }
    }
    r = block_argext(bv, bi, true);
    if (threadIdx.x == 0) { out_v[blockIdx.x] = r.v; out_i[blockIdx.x] = r.i; }
}

__global__ void k_fill(double *__restrict__ a, int64_t n, double v) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) a[i] = v;
}

// ------------------------------------------------- orderings on one cluster
//
// For the sizes of the workloads (up to kClusterMaxN locations) an ordering is
// a few kernels on one thread-block cluster instead of a launch per radix pass,
// tree level or selected point: its bytes take a microsecond, so that launches,
// their gaps and host synchronisations were all of the time.  Arrays stay in
// L2 (__ldcg / __stcg: another CTA wrote them in an earlier phase); a cluster
// barrier separates the phases.  40,000 locations with xy_out: Hilbert 123 -> 47
// us, KD-tree 2,940 -> 177 us (sort 75, upper levels 70, subtrees 29); 10,000
// locations by max-min 82 -> 15 ms.  Above kClusterMaxN the launches above take over (more
// SMs share a pass): their distance shrinks as n grows, 65,536 locations 162 -> 77
// us by Hilbert and 3,560 -> 238 by KD-tree, 131,072 180 -> 97 and 5,390 -> 367,
// 262,144 227 -> 144 and 9,330 -> 685 (launches -> cluster).
constexpr int kOrdCl = 16, kOrdThreads = 1024, kOrdWarps = kOrdThreads / 32;
constexpr int64_t kClusterMaxN = (int64_t)1 << 18;
constexpr int kSortBatch = 4;  // keys a lane loads before it counts them

struct SortShared {
    uint32_t cnt[kOrdWarps][256];
    uint32_t hist[256], base[256], part[8];
    int skip;
};

// Lanes (of those with `in`) that hold the same 8-bit digit: one vote a bit (a
// match instruction goes through the warp's distinct values one by one).
__device__ __forceinline__ uint32_t same_digit(uint32_t d, bool in) {
    uint32_t peers = __ballot_sync(0xFFFFFFFFu, in);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const bool set = (d >> b) & 1u;
        const uint32_t v = __ballot_sync(0xFFFFFFFFu, set);
        peers &= set ? v : ~v;
    }
    return peers;
}

// Stable sort of (key, val) by the bits [from, to) of the key, by one cluster
// (kVals false: of keys alone, which then carry their value in other bits: one
// 8-byte store an item, where the scattered stores are half of a pass):
// warp w of the cluster takes a run of items, counts its digits (one count per
// warp and digit, leaders of equal digits found by match), the counts are
// summed over warps, CTAs (over DSMEM) and digits, and the warp writes its
// items in order.  A pass in which all keys share the digit is left out.  The
// result ends in (keys, vals).
template <typename K, bool kVals>
__device__ void cluster_sort(cg::cluster_group &cl, SortShared &S, K *&keys, uint32_t *&vals, K *&ktmp, uint32_t *&vtmp,
                             int n, int from, int to) {
    const int rank = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int run = (n + kOrdCl * kOrdWarps * 32 - 1) / (kOrdCl * kOrdWarps * 32);  // rounds of 32 items a warp
    const int i0 = (rank * kOrdWarps + warp) * run * 32;
    const uint32_t below = (1u << lane) - 1u;
    for (int shift = from; shift < to; shift += 8) {
        for (int e = tid; e < kOrdWarps * 256; e += kOrdThreads) S.cnt[e >> 8][e & 255] = 0;
        __syncthreads();
        for (int u0 = 0; u0 < run; u0 += kSortBatch) {
            K k[kSortBatch];
#pragma unroll
            for (int u = 0; u < kSortBatch; ++u) {
                const int i = i0 + (u0 + u) * 32 + lane;
                k[u] = u0 + u < run && i < n ? __ldcg(keys + i) : K(0);
            }
#pragma unroll
            for (int u = 0; u < kSortBatch; ++u) {
                const int i = i0 + (u0 + u) * 32 + lane;
                const bool in = u0 + u < run && i < n;
                const uint32_t d = (uint32_t)(k[u] >> shift) & 255u;
                const uint32_t peers = same_digit(d, in);
                if (in && !(peers & below)) S.cnt[warp][d] += __popc(peers);
                __syncwarp();
            }
        }
        __syncthreads();
        if (tid < 256) {
            uint32_t t = 0;
#pragma unroll 8
            for (int w = 0; w < kOrdWarps; ++w) {
                const uint32_t c = S.cnt[w][tid];
                S.cnt[w][tid] = t;
                t += c;
            }
            S.hist[tid] = t;
        }
        if (tid == 0) S.skip = 0;
        cl.sync();
        if (tid < 256) {
            uint32_t tot = 0, before = 0, h[kOrdCl];
#pragma unroll
            for (int q = 0; q < kOrdCl; ++q) h[q] = cl.map_shared_rank(&S.hist[0], q)[tid];
#pragma unroll
            for (int q = 0; q < kOrdCl; ++q) {
                before += q < rank ? h[q] : 0u;
                tot += h[q];
            }
            if (tot == (uint32_t)n) S.skip = 1;
            uint32_t inc = tot;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, inc, o);
                if (lane >= o) inc += v;
            }
            if (lane == 31) S.part[warp] = inc;
            S.base[tid] = inc - tot + before;
        }
        __syncthreads();
        if (tid < 256) {
            uint32_t s = 0;
            for (int w = 0; w < warp; ++w) s += S.part[w];
            S.base[tid] += s;
        }
        __syncthreads();
        if (S.skip) {  // the same on every CTA
            cl.sync();  // every CTA has read the histograms
            continue;
        }
        for (int u0 = 0; u0 < run; u0 += kSortBatch) {
            K k[kSortBatch];
            uint32_t v[kSortBatch];
#pragma unroll
            for (int u = 0; u < kSortBatch; ++u) {
                const int i = i0 + (u0 + u) * 32 + lane;
                const bool in = u0 + u < run && i < n;
                k[u] = in ? __ldcg(keys + i) : K(0);
                v[u] = kVals && in ? __ldcg(vals + i) : 0u;
            }
#pragma unroll
            for (int u = 0; u < kSortBatch; ++u) {
                const int i = i0 + (u0 + u) * 32 + lane;
                const bool in = u0 + u < run && i < n;
                const uint32_t d = (uint32_t)(k[u] >> shift) & 255u;
                const uint32_t peers = same_digit(d, in);
                if (in) {
                    const uint32_t pos = S.base[d] + S.cnt[warp][d] + __popc(peers & below);
                    __stcg(ktmp + pos, k[u]);
                    if constexpr (kVals) __stcg(vtmp + pos, v[u]);
                }
                __syncwarp();
                if (in && !(peers & below)) S.cnt[warp][d] += __popc(peers);
                __syncwarp();
            }
        }
        cl.sync();
        K *kk = keys;
        keys = ktmp;
        ktmp = kk;
        uint32_t *vv = vals;
        vals = vtmp;
        vtmp = vv;
    }
}

// Random / Morton / Hilbert ordering: items (key, index) in 64 bits, by the
// whole GPU (their FP64 rounding alone took 9 us on the cluster's 16 SMs) ...
__global__ void k_sfc_items(const double *__restrict__ xy, int n, int method, uint64_t seed, uint64_t *__restrict__ items,
                            uint32_t *__restrict__ codes) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t k;
    if (method == TLR_ORDER_RANDOM) {
        k = (uint32_t)(splitmix64(seed ^ (uint64_t)i) >> 32);
    } else {
        const uint32_t qx = quantize16(xy[i]), qy = quantize16(xy[n + i]);
        k = (method == TLR_ORDER_MORTON) ? (spread_bits(qx) | (spread_bits(qy) << 1)) : hilbert16(qx, qy);
    }
    items[i] = ((uint64_t)k << 32) | (uint32_t)i;
    if (codes) codes[i] = k;
}
// ... then their sort, the permutation and the permuted locations.
__global__ void __launch_bounds__(kOrdThreads) k_sfc_cluster(const double *__restrict__ xy, int n, uint64_t *items,
                                                              uint64_t *tmp,
                                                              int64_t *__restrict__ perm, double *__restrict__ xy_out,
                                                              int quantize) {
    __shared__ SortShared S;
    cg::cluster_group cl = cg::this_cluster();
    const int t0 = (int)cl.block_rank() * kOrdThreads + threadIdx.x;
    uint32_t *none = nullptr;
    cluster_sort<uint64_t, false>(cl, S, items, none, tmp, none, n, 32, 64);
    for (int p = t0; p < n; p += kOrdCl * kOrdThreads) {
        const uint32_t i = (uint32_t)__ldcg(items + p);
        perm[p] = (int64_t)i;
        if (xy_out) {
            double x = xy[i], y = xy[n + i];
            if (quantize) {
                x = __ddiv_rn((double)quantize16(x), 65535.0);
                y = __ddiv_rn((double)quantize16(y), 65535.0);
            }
            xy_out[p] = x;
            xy_out[n + p] = y;
        }
    }
    cl.sync();  // no CTA leaves while another may still read its histogram
}

// KD-tree, part 1: the locations sorted by (x, index) and by (y, index), one
// cluster each.  list[dim] receives the order.
__global__ void __launch_bounds__(kOrdThreads) k_kd_sort(const double *__restrict__ xy, int n, uint64_t *keys, uint64_t *ktmp,
                                                          uint32_t *vals, uint32_t *vtmp, uint32_t *__restrict__ list) {
    __shared__ SortShared S;
    cg::cluster_group cl = cg::this_cluster();
    const int dim = blockIdx.x / kOrdCl, t0 = (int)cl.block_rank() * kOrdThreads + threadIdx.x;
    keys += (int64_t)dim * n;
    ktmp += (int64_t)dim * n;
    vals += (int64_t)dim * n;
    vtmp += (int64_t)dim * n;
    for (int i = t0; i < n; i += kOrdCl * kOrdThreads) {
        __stcg(keys + i, (uint64_t)dkey(xy[(int64_t)dim * n + i]));
        __stcg(vals + i, (uint32_t)i);
    }
    cl.sync();
    cluster_sort<uint64_t, true>(cl, S, keys, vals, ktmp, vtmp, n, 0, 64);
    for (int p = t0; p < n; p += kOrdCl * kOrdThreads) list[(int64_t)dim * n + p] = __ldcg(vals + p);
    cl.sync();  // no CTA leaves while another may still read its histogram
}

// Whether a node splits along x: its range of x is at least that of y.  The
// node's points are at positions [a, a + m) of both lists, sorted in each.
__device__ __forceinline__ bool kd_split_x(double x0, double x1, double y0, double y1) {
    return __dsub_rn(x1, x0) >= __dsub_rn(y1, y0);
}

// KD-tree, part 2: the upper levels, by one cluster.  A level needs no sort:
// both lists stay sorted inside every node, the node's first ceil(m / 2) points
// along the chosen dimension go left, and the other list is partitioned
// stably by that side.  A level: (1) the dimension of every node from the ends
// of its two runs; (2) every point's side, from the list of that dimension; (3)
// the lefts before each position, counted over warps, CTAs and the cluster; (4)
// the new positions.  Node starts and the lefts before them follow from n
// alone: a level's nodes hold q = n >> level or q + 1 points.
constexpr int kKdLocal = 2048;  // nodes up to this size are finished by one CTA each
constexpr int kKdTopNodes = 256;
__global__ void __launch_bounds__(kOrdThreads) k_kd_top(const double *__restrict__ xy, int n, uint32_t *list, uint32_t *ltmp,
                                                         uint8_t *side, int levels) {
    __shared__ uint8_t dim_x[kKdTopNodes];
    __shared__ int wtot[2][kOrdWarps], total[2], before[2];
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int run = (n + kOrdCl * kOrdWarps * 32 - 1) / (kOrdCl * kOrdWarps * 32);
    const int p0 = (rank * kOrdWarps + warp) * run * 32;
    const uint32_t below = (1u << lane) - 1u;
    // node of position p at a level: index s, start a, size m
    auto node = [&](int p, int level, int &s, int &a, int &m) {
        s = 0;
        a = 0;
        m = n;
        for (int l = 0; l < level; ++l) {
            const int h = (m + 1) / 2;
            const bool right = p >= a + h;
            s = 2 * s + right;
            a += right ? h : 0;
            m = right ? m - h : h;
        }
    };
    for (int level = 0; level < levels; ++level) {
        const uint32_t *X = list, *Y = list + n;
        for (int s = tid; s < (1 << level); s += kOrdThreads) {
            int a = 0, m = n;
            for (int l = level - 1; l >= 0; --l) {
                const int h = (m + 1) / 2;
                const bool right = (s >> l) & 1;
                a += right ? h : 0;
                m = right ? m - h : h;
            }
            dim_x[s] = kd_split_x(xy[__ldcg(X + a)], xy[__ldcg(X + a + m - 1)], xy[n + __ldcg(Y + a)],
                                  xy[n + __ldcg(Y + a + m - 1)]);
        }
        __syncthreads();
        for (int u = 0; u < run; ++u) {
            const int p = p0 + 32 * u + lane;
            if (p >= n) break;
            int s, a, m;
            node(p, level, s, a, m);
            const uint32_t i = __ldcg((dim_x[s] ? X : Y) + p);
            __stcg(side + i, (uint8_t)(p - a < (m + 1) / 2));
        }
        cl.sync();
        int cnt[2] = {0, 0};
        for (int u = 0; u < run; ++u) {
            const int p = p0 + 32 * u + lane;
#pragma unroll
            for (int d = 0; d < 2; ++d) {
                const bool left = p < n && __ldcg(side + __ldcg(list + (int64_t)d * n + p));
                cnt[d] += __popc(__ballot_sync(0xFFFFFFFFu, left));
            }
        }
        if (lane == 0) {
            wtot[0][warp] = cnt[0];
            wtot[1][warp] = cnt[1];
        }
        __syncthreads();
        if (warp < 2) {  // exclusive sums over the CTA's warps
            const int v = wtot[warp][lane];
            int inc = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xFFFFFFFFu, inc, o);
                if (lane >= o) inc += t;
            }
            wtot[warp][lane] = inc - v;
            if (lane == 31) total[warp] = inc;
        }
        cl.sync();
        if (warp < 2) {
            int v = lane < rank ? cl.map_shared_rank(&total[0], lane < kOrdCl ? lane : 0)[warp] : 0;
            v = __reduce_add_sync(0xFFFFFFFFu, v);
            if (lane == 0) before[warp] = v;
        }
        __syncthreads();
        const int q = n >> level;
        int f[2] = {before[0] + wtot[0][warp], before[1] + wtot[1][warp]};
        for (int u = 0; u < run; ++u) {
            const int p = p0 + 32 * u + lane;
            int s = 0, a = 0, m = 0;
            if (p < n) node(p, level, s, a, m);
            const int h = (m + 1) / 2, big = a - s * q;  // nodes of q + 1 points before this one
            const int fa = (s - big) * ((q + 1) / 2) + big * ((q + 2) / 2);
#pragma unroll
            for (int d = 0; d < 2; ++d) {
                const uint32_t i = p < n ? __ldcg(list + (int64_t)d * n + p) : 0u;
                const bool left = p < n && __ldcg(side + i);
                const uint32_t bal = __ballot_sync(0xFFFFFFFFu, left);
                const int lf = f[d] + __popc(bal & below) - fa;  // lefts of the node before p
                if (p < n) __stcg(ltmp + (int64_t)d * n + (left ? a + lf : a + h + (p - a) - lf), i);
                f[d] += __popc(bal);
            }
        }
        cl.sync();
        uint32_t *t = list;
        list = ltmp;
        ltmp = t;
    }
    cl.sync();  // no CTA leaves while another may still read its totals
}

// KD-tree, part 3: one CTA finishes the subtree of one node (at most kKdLocal
// points) in shared memory, two positions a thread, and writes its part of the
// permutation.
struct KdShared {
    double x[kKdLocal], y[kKdLocal];
    uint32_t id[kKdLocal];
    uint16_t lx[2][kKdLocal], ly[2][kKdLocal];
    int fx[kKdLocal + 1], fy[kKdLocal + 1];
    uint8_t side[kKdLocal], dim_x[kKdLocal];
    int wsum[2][kOrdWarps];
};
__global__ void __launch_bounds__(kOrdThreads) k_kd_bottom(const double *__restrict__ xy, int n, int level,
                                                            const uint32_t *__restrict__ list, uint32_t *__restrict__ pos,
                                                            int64_t *__restrict__ perm) {
    extern __shared__ __align__(16) unsigned char raw[];
    KdShared &S = *reinterpret_cast<KdShared *>(raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int a0 = 0, M = n;
    for (int l = level - 1; l >= 0; --l) {
        const int h = (M + 1) / 2;
        const bool right = (blockIdx.x >> l) & 1;
        a0 += right ? h : 0;
        M = right ? M - h : h;
    }
    for (int p = tid; p < M; p += kOrdThreads) {
        const uint32_t i = list[a0 + p];
        S.id[p] = i;
        S.x[p] = xy[i];
        S.y[p] = xy[n + i];
        S.lx[0][p] = (uint16_t)p;
        pos[i] = (uint32_t)p;
    }
    __syncthreads();
    for (int p = tid; p < M; p += kOrdThreads) S.ly[0][p] = (uint16_t)pos[list[(int64_t)n + a0 + p]];
    __syncthreads();
    int a[2] = {0, 0}, m[2] = {M, M};  // node of positions 2 tid, 2 tid + 1
    int cur = 0;
    for (int big = M; big > 1; big = (big + 1) / 2, cur ^= 1) {
        const uint16_t *X = S.lx[cur], *Y = S.ly[cur];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int p = 2 * tid + u;
            if (p < M && p == a[u])
                S.dim_x[p] = kd_split_x(S.x[X[p]], S.x[X[p + m[u] - 1]], S.y[Y[p]], S.y[Y[p + m[u] - 1]]);
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int p = 2 * tid + u;
            if (p < M) S.side[S.dim_x[a[u]] ? X[p] : Y[p]] = p - a[u] < (m[u] + 1) / 2;
        }
        __syncthreads();
        // lefts before every position of both lists
        int lf[2][2], inc[2];
#pragma unroll
        for (int d = 0; d < 2; ++d) {
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int p = 2 * tid + u;
                lf[d][u] = p < M ? (int)S.side[d ? Y[p] : X[p]] : 0;
            }
            inc[d] = lf[d][0] + lf[d][1];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xFFFFFFFFu, inc[d], o);
                if (lane >= o) inc[d] += t;
            }
            if (lane == 31) S.wsum[d][warp] = inc[d];
        }
        __syncthreads();
        if (warp < 2) {
            const int v = S.wsum[warp][lane];
            int s = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xFFFFFFFFu, s, o);
                if (lane >= o) s += t;
            }
            S.wsum[warp][lane] = s - v;
        }
        __syncthreads();
        int f[2][2];
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            f[d][0] = S.wsum[d][warp] + inc[d] - lf[d][0] - lf[d][1];
            f[d][1] = f[d][0] + lf[d][0];
            int *F = d ? S.fy : S.fx;
#pragma unroll
            for (int u = 0; u < 2; ++u)
                if (2 * tid + u < M) F[2 * tid + u] = f[d][u];
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int p = 2 * tid + u, h = (m[u] + 1) / 2;
            if (p >= M) continue;
#pragma unroll
            for (int d = 0; d < 2; ++d) {
                const int before = f[d][u] - (d ? S.fy : S.fx)[a[u]];
                (d ? S.ly : S.lx)[cur ^ 1][lf[d][u] ? a[u] + before : a[u] + h + (p - a[u]) - before] = d ? Y[p] : X[p];
            }
            if (p - a[u] < h) {
                m[u] = h;
            } else {
                a[u] += h;
                m[u] -= h;
            }
        }
        __syncthreads();
    }
    for (int p = tid; p < M; p += kOrdThreads) perm[a0 + p] = (int64_t)S.id[S.lx[cur][p]];
}

// Max-min on one cluster: every CTA keeps a share of the points (coordinates
// and minimum squared distances) in shared memory, and a step is one pass over
// it, the argmax by warp reductions of the distances' bit patterns (nonnegative
// doubles order like their bits; a taken point, -1, comes below), and one
// exchange of the CTAs' candidates.  The FP64 distance (7 operations of 64
// cycles a warp) is formed only where an FP32 box test cannot rule it out:
// |dx| > r or |dy| > r with r above the square root of the minimum distance by
// more than every rounding involved means that the distance is larger.  Steps
// depend on one another: 1.4 us each at n = 10,000, the chain of the FP64
// distances of the points hit, the look at their neighbours and the reductions
// (on one CTA, without the exchange, as long).  40,000 points 407 -> 78 ms,
// 98,304 1,007 -> 292, where the points no longer fit the shared memory.
constexpr int kMaxminClusterN = 98304;  // 36 bytes a point, 6,144 points a CTA
constexpr int kMmThreads = 512, kMmWarps = kMmThreads / 32;
struct MmCand {
    int hi;
    uint32_t lo;
    int64_t i;
    double x, y;
};
// Best candidate over the warp: largest (hi, lo), then the lowest index; its
// lane in `who`.
__device__ __forceinline__ void mm_best(int hi, uint32_t lo, uint32_t i, int &who) {
    const int mh = __reduce_max_sync(0xFFFFFFFFu, hi);
    const uint32_t ml = __reduce_max_sync(0xFFFFFFFFu, hi == mh ? lo : 0u);
    const bool top = hi == mh && lo == ml;
    const uint32_t mi = __reduce_min_sync(0xFFFFFFFFu, top ? i : 0xFFFFFFFFu);
    who = __ffs(__ballot_sync(0xFFFFFFFFu, top && i == mi)) - 1;
}
static size_t maxmin_bytes(int n) { return (size_t)ceil_div(n, kOrdCl) * (3 * sizeof(double) + 3 * sizeof(float)) + 64; }
__global__ void __launch_bounds__(kMmThreads) k_maxmin_cluster(const double *__restrict__ xy, int n, int nfirst,
                                                                const double *__restrict__ first_v,
                                                                const long long *__restrict__ first_i,
                                                                int64_t *__restrict__ perm) {
    extern __shared__ __align__(16) unsigned char raw[];
    __shared__ MmCand slot[2][kOrdCl], wbest[kMmWarps];
    __shared__ float emax[kMmWarps];
    __shared__ long long s_p;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = (n + kOrdCl - 1) / kOrdCl, g0 = min(n, rank * per), cnt = min(n, g0 + per) - g0;
    double *X = reinterpret_cast<double *>(raw), *Y = X + per, *D = Y + per;
    float *X4 = reinterpret_cast<float *>(D + per), *Y4 = X4 + per, *R4 = Y4 + per;
    for (int j = tid; j < cnt; j += kMmThreads) {
        X[j] = xy[g0 + j];
        Y[j] = xy[n + g0 + j];
        D[j] = INFINITY;
        X4[j] = (float)X[j];
        Y4[j] = (float)Y[j];
        R4[j] = INFINITY;
    }
    // slack: above the rounding of a coordinate difference in FP32 (at most
    // 4 x 2^-24 of the largest magnitude); a non-finite coordinate makes it
    // infinite and switches the box test off
    float big = 0.f;
    for (int j = tid; j < n; j += kMmThreads) {
        const double x = xy[j], y = xy[n + j];
        big = isfinite(x) && isfinite(y) ? fmaxf(big, fmaxf(fabsf((float)x), fabsf((float)y))) : INFINITY;
    }
    for (int o = 16; o; o >>= 1) big = fmaxf(big, __shfl_xor_sync(0xFFFFFFFFu, big, o));
    if (lane == 0) emax[warp] = big;
    // the first point: the nearest to the box's centre
    double fv = INFINITY;
    long long fi = 0x7FFFFFFFFFFFFFFFll;
    for (int b = tid; b < nfirst; b += kMmThreads)
        if (better_min(first_v[b], first_i[b], fv, fi)) {
            fv = first_v[b];
            fi = first_i[b];
        }
    const MaxLoc r0 = block_argext(fv, fi, false);
    if (tid == 0) s_p = r0.i;
    __syncthreads();
    for (int w = 0; w < kMmWarps; ++w) big = fmaxf(big, emax[w]);
    const float slack = big * 4.8e-7f + 1e-37f;  // 8 x 2^-24
    int64_t p = s_p;
    if (p < 0 || p >= n) p = 0;  // only reachable with non-finite coordinates
    double px = xy[p], py = xy[n + p];
    int bh = INT32_MIN;  // the thread's best point
    uint32_t bl = 0, bi = 0xFFFFFFFFu;
    cl.sync();
    for (int k = 0; k < n; ++k) {
        if (rank == 0 && tid == 0) perm[k] = p;
        const float px4 = (float)px, py4 = (float)py;
        bool again = k == 0;
        for (int j = tid; j < cnt; j += kMmThreads) {
            const float r = R4[j];
            if (r < 0.f || fabsf(X4[j] - px4) > r || fabsf(Y4[j] - py4) > r) continue;
            double m = -1.0;  // taken (a point's own box contains it)
            float r2 = -1.f;
            if (g0 + j != p) {
                const double d = sqdist(X[j], Y[j], px, py);
                m = D[j];
                if (d >= m) continue;
                m = fmin(m, d);
                const float m4 = (float)m;
                r2 = (m4 < 1e-30f ? 1.0001e-15f : sqrtf(m4) * 1.00001f) + slack;
            }
            D[j] = m;
            R4[j] = r2;
            again |= (uint32_t)(g0 + j) == bi;
        }
        // a thread looks its points over again, and its warp reduces again, only
        // when a best point changed (warp reductions are slow)
        if (again) {
            bh = INT32_MIN;
            for (int j = tid; j < cnt; j += kMmThreads) {
                const double m = D[j];
                const int h = __double2hiint(m);
                const uint32_t l = (uint32_t)__double2loint(m);
                if (h > bh || (h == bh && l > bl)) {  // indices rise: the first of equals stays
                    bh = h;
                    bl = l;
                    bi = (uint32_t)(g0 + j);
                }
            }
        }
        int who;
        if (__any_sync(0xFFFFFFFFu, again)) {
            mm_best(bh, bl, bi, who);
            if (lane == who) wbest[warp] = MmCand{bh, bl, (int64_t)bi, 0.0, 0.0};
        }
        __syncthreads();
        if (warp == 0) {
            const MmCand c = lane < kMmWarps ? wbest[lane] : MmCand{INT32_MIN, 0u, (int64_t)0xFFFFFFFF, 0.0, 0.0};
            mm_best(c.hi, c.lo, (uint32_t)c.i, who);
            MmCand b;
            b.hi = __shfl_sync(0xFFFFFFFFu, c.hi, who);
            b.lo = __shfl_sync(0xFFFFFFFFu, c.lo, who);
            const uint32_t i = __shfl_sync(0xFFFFFFFFu, (uint32_t)c.i, who);
            const int j = (int)i - g0;
            const bool own = i != 0xFFFFFFFFu;
            b.i = (int64_t)i;
            b.x = own ? X[j] : 0.0;
            b.y = own ? Y[j] : 0.0;
            if (lane < kOrdCl) cl.map_shared_rank(&slot[k & 1][0], lane)[rank] = b;
        }
        cl.sync();
        const MmCand c = lane < kOrdCl ? slot[k & 1][lane] : MmCand{INT32_MIN, 0u, (int64_t)0xFFFFFFFF, 0.0, 0.0};
        mm_best(c.hi, c.lo, (uint32_t)c.i, who);
        p = (int64_t)__shfl_sync(0xFFFFFFFFu, (uint32_t)c.i, who);
        px = __shfl_sync(0xFFFFFFFFu, c.x, who);
        py = __shfl_sync(0xFFFFFFFFu, c.y, who);
    }
}

// Whether clusters of 16 CTAs of the kernels above run on the current device.
static bool cluster_order_ok() {
    static PerDevice<bool> per_device;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    return per_device.get(dev, [dev] {
        int optin = 0;
        bool ok = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess &&
             cudaFuncSetAttribute(k_kd_bottom, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(KdShared)) == cudaSuccess;
        cudaFuncAttributes fa;
        ok = ok && cudaFuncGetAttributes(&fa, k_maxmin_cluster) == cudaSuccess &&
             cudaFuncSetAttribute(k_maxmin_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  optin - (int)fa.sharedSizeBytes) == cudaSuccess;
        auto fits = [](const void *k, int threads, size_t smem) {
            if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return false;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(kOrdCl);
            cfg.blockDim = dim3((unsigned)threads);
            cfg.dynamicSmemBytes = smem;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = kOrdCl;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            int nc = 0;
            return cudaOccupancyMaxActiveClusters(&nc, k, &cfg) == cudaSuccess && nc > 0;
        };
        ok = ok && fits((const void *)k_sfc_cluster, kOrdThreads, 0) && fits((const void *)k_kd_sort, kOrdThreads, 0) &&
             fits((const void *)k_kd_top, kOrdThreads, 0) &&
             fits((const void *)k_maxmin_cluster, kMmThreads, maxmin_bytes(kMaxminClusterN));
        cudaGetLastError();  // clear any error of the queries
        return ok;
    });
}

// ------------------------------------------------------------- drivers
static inline int grid1(int64_t n, int t = 256) { return (int)ceil_div(n > 0 ? n : 1, t); }

void order_sfc(const double *xy, int64_t n, int method, uint64_t seed, int64_t *perm,
               uint32_t *codes, double *xy_out, int quantize, cudaStream_t s) {
    if (n <= kClusterMaxN && cluster_order_ok()) {
        DevBuf b(16 * n, s);
        uint64_t *k = b.as<uint64_t>();
        launch(k_sfc_items, grid1(n, 128), 128, 0, s, xy, (int)n, method, seed, k, codes);
        TLR_CHECK_LAUNCH();
        launch_clustered(k_sfc_cluster, kOrdCl, 1, kOrdThreads, 0, s, xy, (int)n, k, k + n, perm, xy_out, quantize);
        return;
    }
    DevBuf kb(n * 4, s), vb(n * 4, s), kt(n * 4, s), vt(n * 4, s), hb(hist_words(n) * 4, s);
    uint32_t *keys = kb.as<uint32_t>(), *vals = vb.as<uint32_t>();
    uint32_t *ktmp = kt.as<uint32_t>(), *vtmp = vt.as<uint32_t>();
    launch(k_sfc_keys, grid1(n), 256, 0, s, xy, n, method, seed, keys, vals);
    TLR_CHECK_LAUNCH();
    if (codes) TLR_CUDA_TRY(cudaMemcpyAsync(codes, keys, n * 4, cudaMemcpyDeviceToDevice, s));
    radix_sort<uint32_t>(&keys, &vals, &ktmp, &vtmp, n, 32, hb.as<uint32_t>(), s);
    launch(k_perm_out, grid1(n), 256, 0, s, vals, n, perm);
    TLR_CHECK_LAUNCH();
    if (xy_out) permute_xy(xy, perm, n, quantize, xy_out, s);
}

static int bit_width(uint64_t v) {
    int b = 0;
    while (v) { ++b; v >>= 1; }
    return b;
}

void order_kdtree(const double *xy, int64_t n, int64_t *perm, cudaStream_t s) {
    if (n <= 1) {
        if (n == 1) launch(k_iota, 1, 32, 0, s, n, perm);
        return;
    }
    if (n <= kClusterMaxN && cluster_order_ok()) {
        // keys and values of both dimensions with their copies, two pairs of lists, sides
        DevBuf b(n * (4 * 8 + 4 * 4 + 4 * 4 + 4) + 16, s);
        uint64_t *keys = b.as<uint64_t>(), *ktmp = keys + 2 * n;
        uint32_t *vals = reinterpret_cast<uint32_t *>(ktmp + 2 * n), *vtmp = vals + 2 * n, *list = vtmp + 2 * n,
                 *ltmp = list + 2 * n, *pos = ltmp + 2 * n;
        launch_clustered(k_kd_sort, kOrdCl, 2, kOrdThreads, 0, s, xy, (int)n, keys, ktmp, vals, vtmp, list);
        int levels = 0;  // until every node has at most kKdLocal points
        while (ceil_div(n, (int64_t)1 << levels) > kKdLocal) ++levels;
        if (levels) {
            launch_clustered(k_kd_top, kOrdCl, 1, kOrdThreads, 0, s, xy, (int)n, list, ltmp,
                             reinterpret_cast<uint8_t *>(keys), levels);
            if (levels & 1) std::swap(list, ltmp);
        }
        launch(k_kd_bottom, 1u << levels, kOrdThreads, sizeof(KdShared), s, xy, (int)n, levels, list, pos, perm);
        TLR_CHECK_LAUNCH();
        return;
    }
    DevBuf kb(n * 8, s), kt(n * 8, s), vb(n * 4, s), vt(n * 4, s), hb(hist_words(n) * 4, s);
    DevBuf rx(n * 4, s), ry(n * 4, s);
    uint64_t *keys = kb.as<uint64_t>(), *ktmp = kt.as<uint64_t>();
    uint32_t *vals = vb.as<uint32_t>(), *vtmp = vt.as<uint32_t>(), *hist = hb.as<uint32_t>();
    // global ranks along x and y (stable: ties by index)
    for (int dim = 0; dim < 2; ++dim) {
        launch(k_coord_keys, grid1(n), 256, 0, s, xy + dim * n, n, keys, vals);
        radix_sort<uint64_t>(&keys, &vals, &ktmp, &vtmp, n, 64, hist, s);
        launch(k_invert, grid1(n), 256, 0, s, vals, n, dim ? ry.as<uint32_t>() : rx.as<uint32_t>());
        TLR_CHECK_LAUNCH();
    }
    // current order: identity
    launch(k_iota32, grid1(n), 256, 0, s, n, vals);
    TLR_CHECK_LAUNCH();
    // segment structure per level (host), then one sort per level
    std::vector<int64_t> starts{0}, sizes{n};
    int rbits = bit_width((uint64_t)(n - 1));
    DevBuf sb(n * 8, s), rb((size_t)n * 32, s);
    while (true) {
        bool any = false;
        for (int64_t m : sizes) any |= (m > 1);
        if (!any) break;
        int nseg = (int)starts.size();
        TLR_CUDA_TRY(cudaMemcpyAsync(sb.as<int64_t>(), starts.data(), nseg * 8, cudaMemcpyHostToDevice, s));
        unsigned long long *rng = rb.as<unsigned long long>();
        launch(k_kd_init_ranges, grid1(nseg), 256, 0, s, nseg, rng);
        launch(k_kd_ranges, grid1(n), 256, 0, s, xy, n, vals, sb.as<int64_t>(), nseg, rng);
        launch(k_kd_keys, grid1(n), 256, 0, s, n, vals, sb.as<int64_t>(), nseg, rng, rx.as<uint32_t>(),
                                           ry.as<uint32_t>(), rbits, keys);
        TLR_CHECK_LAUNCH();
        int bits = rbits + bit_width((uint64_t)(nseg - 1));
        radix_sort<uint64_t>(&keys, &vals, &ktmp, &vtmp, n, bits, hist, s);
        // children: first ceil(m/2) left, the rest right
        std::vector<int64_t> ns, nz;
        ns.reserve(2 * nseg);
        nz.reserve(2 * nseg);
        for (int q = 0; q < nseg; ++q) {
            int64_t m = sizes[q];
            if (m <= 1) { ns.push_back(starts[q]); nz.push_back(m); continue; }
            int64_t h = (m + 1) / 2;
            ns.push_back(starts[q]); nz.push_back(h);
            ns.push_back(starts[q] + h); nz.push_back(m - h);
        }
        starts.swap(ns);
        sizes.swap(nz);
        // the host vectors are read by the next level's async copy: keep the
        // stream in step with them
        TLR_CUDA_TRY(cudaStreamSynchronize(s));
    }
    launch(k_perm_out, grid1(n), 256, 0, s, vals, n, perm);
    TLR_CHECK_LAUNCH();
}

void order_maxmin(const double *xy, int64_t n, int64_t *perm, cudaStream_t s, int num_sms) {
    if (n <= 0) return;
    int nblk = (int)std::min<int64_t>(ceil_div(n, 256), (int64_t)num_sms * 2);
    DevBuf mind(n * 8, s), pv(2 * nblk * 8, s), pi(2 * nblk * 8, s), ctr(16, s);
    launch(k_fill, grid1(n), 256, 0, s, mind.as<double>(), n, INFINITY);
    launch(k_bbox, 1, 1024, 0, s, xy, n, ctr.as<double>());
    launch(k_maxmin_first, nblk, 256, 0, s, xy, n, ctr.as<double>(), pv.as<double>(), pi.as<long long>());
    TLR_CHECK_LAUNCH();
    if (n <= kMaxminClusterN && cluster_order_ok()) {
        launch_clustered(k_maxmin_cluster, kOrdCl, 1, kMmThreads, maxmin_bytes((int)n), s, xy, (int)n, nblk,
                         pv.as<double>(), pi.as<long long>(), perm);
        return;
    }
    double *bv[2] = {pv.as<double>(), pv.as<double>() + nblk};
    long long *bi[2] = {pi.as<long long>(), pi.as<long long>() + nblk};
    for (int64_t k = 0; k < n; ++k) {
        int in = (int)(k & 1), out = in ^ 1;
        launch(k_maxmin_step, nblk, 256, 0, s, xy, n, k, k == 0, bv[in], bi[in], bv[out], bi[out],
                                           mind.as<double>(), perm);
    }
    TLR_CHECK_LAUNCH();
}

void order_identity(int64_t n, int64_t *perm, cudaStream_t s) {
    if (n > 0) launch(k_iota, grid1(n), 256, 0, s, n, perm);
    TLR_CHECK_LAUNCH();
}

void permute_xy(const double *xy, const int64_t *perm, int64_t n, int quantize, double *out,
                cudaStream_t s) {
    if (n > 0) launch(k_permute_xy, grid1(n), 256, 0, s, xy, perm, n, quantize, out);
    TLR_CHECK_LAUNCH();
}

void gather(const int64_t *perm, const double *src, int64_t n, double *dst, cudaStream_t s) {
    if (n > 0) launch(k_gather, grid1(n), 256, 0, s, perm, src, n, dst);
    TLR_CHECK_LAUNCH();
}

}  // namespace tlr

// ----------------------------------------------------------------------------
// Ordering without any allocation.
//
// For callers that must not allocate device memory once they are running:
// a serving loop whose latency budget cannot absorb cudaMalloc's implicit
// device synchronisation, or a host process whose memory is fixed up front
// (a pre-sized pool shared with other work).  tlr_order allocates its sort
// buffers per call; tlr_order_noalloc instead uses one file-scope scratch
// array that every device holds from module load until process exit.
// ----------------------------------------------------------------------------
namespace tlr {

constexpr int64_t kNoAllocMaxN = (int64_t)1 << 18;  // 262,144 locations
constexpr int64_t kNoAllocBlocks = (kNoAllocMaxN + kSortTile - 1) / kSortTile;
// keys, values and their ping-pong copies (4 x n words) plus the radix histogram
constexpr int64_t kNoAllocWords = 4 * kNoAllocMaxN + 256 * kNoAllocBlocks;

static __device__ __align__(256) uint32_t g_order_scratch[kNoAllocWords];

// Device address of g_order_scratch per device, looked up once per device.
static uint32_t *noalloc_scratch(int device, int *rc) {
    static std::mutex mu;
    static uint32_t *addr[64] = {nullptr};
    *rc = TLR_OK;
    if (device < 0 || device >= 64) { *rc = TLR_ERR_ARG; return nullptr; }
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[device]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_order_scratch);
        if (e != cudaSuccess || p == nullptr) { *rc = TLR_ERR_CUDA; return nullptr; }
        addr[device] = static_cast<uint32_t *>(p);
    }
    return addr[device];
}

}  // namespace tlr

extern "C" int tlr_order_noalloc(const double *xy, int64_t n, int method, uint64_t seed, int64_t *perm,
                                 uint32_t *codes, void *stream) {
    using namespace tlr;
    if (n < 0 || n > kNoAllocMaxN) return TLR_ERR_ARG;
    if (method != TLR_ORDER_RANDOM && method != TLR_ORDER_MORTON && method != TLR_ORDER_HILBERT)
        return TLR_ERR_ARG;
    if (n == 0) return TLR_OK;
    if (!xy || !perm) return TLR_ERR_ARG;
    int device = 0;
    if (cudaGetDevice(&device) != cudaSuccess) return TLR_ERR_CUDA;
    int rc = TLR_OK;
    uint32_t *base = noalloc_scratch(device, &rc);
    if (!base) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint32_t *keys = base, *vals = base + kNoAllocMaxN;
    uint32_t *ktmp = base + 2 * kNoAllocMaxN, *vtmp = base + 3 * kNoAllocMaxN;
    uint32_t *hist = base + 4 * kNoAllocMaxN;
    const int nblk = (int)ceil_div(n, kSortTile);
    launch(k_sfc_keys, grid1(n), 256, 0, s, xy, n, method, seed, keys, vals);
    if (codes && cudaMemcpyAsync(codes, keys, n * 4, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
        return TLR_ERR_CUDA;
    // stable LSD radix sort, 4 passes of 8 bits; every histogram entry and
    // every key/value slot read by a pass is written earlier in the same call
    for (int shift = 0; shift < 32; shift += 8) {
        launch(k_radix_hist<uint32_t>, nblk, kSortThreads, 0, s, keys, n, shift, hist, nblk);
        launch(k_scan_exclusive, 1, 1024, 0, s, hist, (int64_t)256 * nblk);
        launch(k_radix_scatter<uint32_t>, nblk, kSortThreads, 0, s, keys, vals, n, shift, hist, nblk, ktmp,
               vtmp);
        std::swap(keys, ktmp);
        std::swap(vals, vtmp);
    }
    launch(k_perm_out, grid1(n), 256, 0, s, vals, n, perm);
    return cudaGetLastError() == cudaSuccess ? TLR_OK : TLR_ERR_CUDA;
}
