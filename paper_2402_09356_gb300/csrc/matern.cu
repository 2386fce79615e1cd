// a2: Matern covariance tiles (Eq. 1.1, Eq. 4.2) and the per-theta constants
// of the device K_nu.
#include <cmath>

#include "common.cuh"
#include "matern.cuh"

namespace tlr {

// zeta(2) .. zeta(40) to quadruple precision.  (Summed anew for every theta,
// 1,000 long-double powers each, they took 53 ms of host time per call on a
// CPU whose long double is software.)
static const long double kZeta[] = {
    1.6449340668482264364724151666460251892L, 1.2020569031595942853997381615114499908L,
    1.0823232337111381915160036965411679028L, 1.0369277551433699263313654864570341681L,
    1.0173430619844491397145179297909205279L, 1.0083492773819228268397975498497967596L,
    1.0040773561979443393786852385086524653L, 1.0020083928260822144178527692324120605L,
    1.000994575127818085337145958900319017L, 1.0004941886041194645587022825264699365L,
    1.000246086553308048298637998047739671L, 1.0001227133475784891467518365263573957L,
    1.0000612481350587048292585451051353337L, 1.0000305882363070204935517285106450626L,
    1.000015282259408651871732571487636722L, 1.0000076371976378997622736002935630292L,
    1.0000038172932649998398564616446219397L, 1.0000019082127165539389256569577951014L,
    1.0000009539620338727961131520386834493L, 1.000000476932986787806463116719604373L,
    1.000000238450502727732990003648186753L, 1.0000001192199259653110730677887188823L,
    1.0000000596081890512594796124402079358L, 1.0000000298035035146522801860637050694L,
    1.0000000149015548283650412346585066307L, 1.0000000074507117898354294919810041706L,
    1.0000000037253340247884570548192040184L, 1.0000000018626597235130490064039099454L,
    1.000000000931327432419668182871764735L, 1.0000000004656629065033784072989233251L,
    1.0000000002328311833676505492001455976L, 1.0000000001164155017270051977592973835L,
    1.0000000000582077208790270088924368599L, 1.0000000000291038504449709968692942523L,
    1.0000000000145519218910419842359296322L, 1.000000000007275959835057481014520869L,
    1.0000000000036379795473786511902372364L, 1.0000000000018189896503070659475848321L,
    1.0000000000009094947840263889282533118L,
};

// Temme's Gamma1(mu) = (1/Gamma(1-mu) - 1/Gamma(1+mu)) / (2 mu) and
// Gamma2(mu) = (1/Gamma(1-mu) + 1/Gamma(1+mu)) / 2 for |mu| <= 1/2.
// For small |mu| the difference cancels, so there both come from
// ln Gamma(1+z) = -gamma z + sum_{k>=2} (-1)^k zeta(k) z^k / k: with
// E = -sum_{k even} zeta(k) mu^k / k and O = gamma mu + sum_{k odd>=3} zeta(k) mu^k / k,
// 1/Gamma(1 -+ mu) = e^E e^(-+O), so Gamma1 = -e^E sinh(O)/mu and Gamma2 = e^E cosh(O).
static void temme_gammas(double mu, double *g1, double *g2) {
    long double m = mu;
    if (fabsl(m) >= 0.2L) {
        long double a = 1.0L / tgammal(1.0L - m), b = 1.0L / tgammal(1.0L + m);
        *g1 = (double)((a - b) / (2.0L * m));
        *g2 = (double)((a + b) / 2.0L);
        return;
    }
    const long double euler = 0.57721566490153286060651209008240243L;
    long double E = 0.0L, Om = euler;  // Om = O / mu
    long double prev = m;              // mu^(k-1)
    for (int k = 2; k <= 40; ++k) {
        long double cur = prev * m;    // mu^k
        const long double z = kZeta[k - 2];
        if (k % 2 == 0) E -= z * cur / k;
        else Om += z * prev / k;
        prev = cur;
    }
    long double O = Om * m;
    long double shr = (fabsl(O) < 1e-12L) ? 1.0L + O * O / 6.0L : sinhl(O) / O;  // sinh(O)/O
    *g1 = (double)(-expl(E) * shr * Om);
    *g2 = (double)(expl(E) * coshl(O));
}

bool make_matern_params(double sigma2, double beta, double nu, MaternParams *P) {
    if (!(sigma2 > 0) || !(beta > 0) || !(nu > 0) || !std::isfinite(sigma2) || !std::isfinite(beta) ||
        !std::isfinite(nu) || nu > 50.0)
        return false;
    P->sigma2 = sigma2;
    P->inv_beta = 1.0 / beta;
    P->tab = nullptr;
    P->nu = nu;
    int m = (int)std::floor(nu + 0.5);
    double mu = nu - m;
    P->m = m;
    P->mu = mu;
    P->lead = (double)(powl(2.0L, 1.0L - (long double)nu) / tgammal((long double)nu));
    temme_gammas(mu, &P->g1, &P->g2);
    P->gp = (double)tgammal(1.0L + (long double)mu);
    P->gm = (double)tgammal(1.0L - (long double)mu);
    long double mpi = (long double)mu * 3.14159265358979323846264338327950288L;
    P->mupi_sin = (fabsl(mpi) < 1e-6L) ? (double)(1.0L + mpi * mpi / 6.0L) : (double)(mpi / sinl(mpi));
    P->inv_gmu1 = (double)(1.0L / tgammal((long double)mu + 1.0L));
    P->inv_gmu2 = (double)(1.0L / tgammal((long double)mu + 2.0L));
    for (int k = 0; k <= kTemmeTerms; ++k) {
        long double kk = k;
        P->tf[k] = k ? (double)(1.0L / (kk * kk - (long double)mu * mu)) : 0.0;
        P->tp[k] = k ? (double)(1.0L / (kk - mu)) : 0.0;
        P->tq[k] = k ? (double)(1.0L / (kk + mu)) : 0.0;
        P->tk[k] = k ? (double)(1.0L / kk) : 0.0;
    }
    for (int k = 0; k <= kISeriesTerms; ++k) {
        long double kk = k;
        P->ti0[k] = k ? (double)(1.0L / (kk * (kk + mu))) : 0.0;
        P->ti1[k] = k ? (double)(1.0L / (kk * (kk + mu + 1.0L))) : 0.0;
    }
    for (int k = 0; k <= kAsymTerms; ++k) {
        long double kk = k, a = 4.0L * mu * mu, b = 4.0L * (mu + 1.0L) * (mu + 1.0L);
        long double o = (2.0L * kk - 1.0L) * (2.0L * kk - 1.0L);
        P->ta0[k] = k ? (double)((a - o) / (8.0L * kk)) : 0.0;
        P->ta1[k] = k ? (double)((b - o) / (8.0L * kk)) : 0.0;
    }
    return true;
}

// Packed lower-triangular tiles: blockIdx.y = packed tile index, each block
// fills a 32 x 32 sub-block; threads run down the columns (coalesced stores).
__global__ void k_generate_tiles(const double *__restrict__ xy, int64_t n, int nb, int nt,
                                 MaternParams P, double *__restrict__ tiles) {
    int sub = nb / 32 + (nb % 32 != 0);
    int64_t t = (int64_t)blockIdx.x / (sub * sub);
    int sb = (int)((int64_t)blockIdx.x % (sub * sub));
    // tile (i, j) from packed index t = i (i + 1) / 2 + j
    int i = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);  // corrected below
    while ((int64_t)(i + 1) * (i + 2) / 2 <= t) ++i;
    while ((int64_t)i * (i + 1) / 2 > t) --i;
    int j = (int)(t - (int64_t)i * (i + 1) / 2);
    int br = sb % sub, bc = sb / sub;
    int r = br * 32 + (threadIdx.x & 31);
    int c0 = bc * 32 + (threadIdx.x >> 5) * 4;
    int64_t gr = (int64_t)i * nb + r;
    double *T = tiles + t * (int64_t)nb * nb;
    bool rv = r < nb && gr < n;
    double xr = rv ? xy[gr] : 0.0, yr = rv ? xy[n + gr] : 0.0;
    for (int q = 0; q < 4; ++q) {
        int c = c0 + q;
        if (c >= nb || r >= nb) continue;
        int64_t gc = (int64_t)j * nb + c;
        double v = 0.0;
        if (rv && gc < n) v = matern_cov(xr, yr, xy[gc], xy[n + gc], P);
        T[(int64_t)c * nb + r] = v;
    }
    (void)nt;
}

// A column panel of the covariance: T[c * ld + r] = C(s_{ri0 + r}, s_{ci0 + c})
// for r < rows, c < cols; rows or columns past n give 0.  Each block fills a
// 32-row x 32-column sub-block, threads down the columns (coalesced stores).
__global__ void k_generate_panel(const double *__restrict__ xy, int64_t n, int64_t ri0, int64_t ci0, int rows,
                                 int cols, MaternParams P, double *__restrict__ T, int ld) {
    const int r = blockIdx.x * 32 + (threadIdx.x & 31);
    const int c0 = blockIdx.y * 32 + (threadIdx.x >> 5) * 4;
    if (r >= rows) return;
    const int64_t gr = ri0 + r;
    const bool rv = gr < n;
    const double xr = rv ? xy[gr] : 0.0, yr = rv ? xy[n + gr] : 0.0;
    for (int q = 0; q < 4; ++q) {
        const int c = c0 + q;
        if (c >= cols) break;
        const int64_t gc = ci0 + c;
        T[(int64_t)c * ld + r] = (rv && gc < n) ? matern_cov(xr, yr, xy[gc], xy[n + gc], P) : 0.0;
    }
}

__global__ void k_matern_vec(const double *__restrict__ d, int64_t m, MaternParams P,
                             double *__restrict__ out) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= m) return;
    double v = d[k];
    if (v == 0.0) out[k] = P.sigma2;
    else if (P.tab) out[k] = P.sigma2 * matern_corr_s(v * v, P);
    else out[k] = P.sigma2 * matern_corr_x(v * P.inv_beta, P);
}

// Table nodes: log2 C/sigma2 at the Chebyshev points of every interval.
__global__ void k_table_nodes(MaternParams P, double *__restrict__ g) {
    int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= kTabIntervals * kTabCoef) return;
    int iv = q / kTabCoef, k = q % kTabCoef;
    int e = kTabEmin + iv / kTabSub, sub = iv % kTabSub;
    double lo = ldexp(1.0 + (double)sub / kTabSub, e), hi = ldexp(1.0 + (double)(sub + 1) / kTabSub, e);
    double node = cospi((k + 0.5) / kTabCoef);
    double sv = lo + 0.5 * (node + 1.0) * (hi - lo);
    double c = matern_corr_x(sqrt(sv) * P.inv_beta, P);
    g[q] = (c > 1e-280) ? log2(c) : __longlong_as_double(0x7FF8000000000000ll);
}

// Coefficients a_i of the interpolant in powers of t, from the Chebyshev
// coefficients c_j = (2/N) sum_k g_k cos(j pi (k + 1/2) / N), c_0 halved, and
// T_{j+1} = 2 t T_j - T_{j-1}; an interval with a non-finite node value keeps
// a_0 = NaN (direct evaluation).  The last entries are 2^(j/32).
__global__ void k_table_coefs(const double *__restrict__ g, double *__restrict__ tab) {
    const int iv = blockIdx.x * blockDim.x + threadIdx.x;
    if (iv < kTabExp) tab[kTabIntervals * kTabCoef + iv] = exp2((double)iv / kTabExp);
    if (iv >= kTabIntervals) return;
    double gi[kTabCoef], a[kTabCoef], t0[kTabCoef], t1[kTabCoef];
    bool bad = false;
#pragma unroll
    for (int k = 0; k < kTabCoef; ++k) {
        gi[k] = g[iv * kTabCoef + k];
        bad |= !(gi[k] == gi[k]);
        a[k] = t0[k] = t1[k] = 0.0;
    }
    t0[0] = 1.0;
    t1[1] = 1.0;
    for (int j = 0; j < kTabCoef; ++j) {
        double c = 0.0;
#pragma unroll
        for (int k = 0; k < kTabCoef; ++k) c += gi[k] * cospi((double)j * (k + 0.5) / kTabCoef);
        c *= (j ? 2.0 : 1.0) / kTabCoef;
        // t0 = T_j, t1 = T_{j+1}
#pragma unroll
        for (int i = 0; i < kTabCoef; ++i) a[i] += c * t0[i];
#pragma unroll
        for (int i = kTabCoef - 1; i >= 0; --i) {
            const double n = (i > 0 ? 2.0 * t1[i - 1] : 0.0) - t0[i];
            t0[i] = t1[i];
            t1[i] = n;
        }
    }
#pragma unroll
    for (int i = 0; i < kTabCoef; ++i)
        tab[iv * kTabCoef + i] = bad && i == 0 ? __longlong_as_double(0x7FF8000000000000ll) : a[i];
}

void build_matern_table(MaternParams *P, double *tab, cudaStream_t s) {
    const int cnt = kTabIntervals * kTabCoef;
    double *g = tab + kTabDoubles;  // scratch: the caller provides kTabBuild doubles
    MaternParams direct = *P;
    direct.tab = nullptr;
    launch(k_table_nodes, (unsigned)ceil_div(cnt, 64), 64, 0, s, direct, g);
    launch(k_table_coefs, (unsigned)ceil_div(kTabIntervals, 64), 64, 0, s, g, tab);
    TLR_CHECK_LAUNCH();
    P->tab = tab;
}

void generate_tiles(const double *xy, int64_t n, int nb, const MaternParams &P, double *tiles,
                    cudaStream_t s) {
    int nt = (int)ceil_div(n, nb);
    int64_t ntiles = (int64_t)nt * (nt + 1) / 2;
    int sub = (int)ceil_div(nb, 32);
    launch(k_generate_tiles, (unsigned)(ntiles * sub * sub), 256, 0, s, xy, n, nb, nt, P, tiles);
    TLR_CHECK_LAUNCH();
}

void generate_panel(const double *xy, int64_t n, int64_t ri0, int64_t ci0, int rows, int cols,
                    const MaternParams &P, double *T, int ld, cudaStream_t s) {
    if (rows <= 0 || cols <= 0) return;
    launch(k_generate_panel, dim3((unsigned)ceil_div(rows, 32), (unsigned)ceil_div(cols, 32)), 256, 0, s, xy, n, ri0,
           ci0, rows, cols, P, T, ld);
    TLR_CHECK_LAUNCH();
}

void matern_vec(const double *d, int64_t m, const MaternParams &P, double *out, cudaStream_t s) {
    if (m > 0) launch(k_matern_vec, (unsigned)ceil_div(m, 256), 256, 0, s, d, m, P, out);
    TLR_CHECK_LAUNCH();
}

}  // namespace tlr
