// series.h -- E = exp(delta (kappa h - mu)) as a polynomial of the sparse
// hopping h (host part; the device functions are in fp64_path.cuh and
// series_cg.cuh).
//
// h has three neighbours per site and its eigenvalues lie in [-3, 3], so with
// rho = 3 |delta kappa| a polynomial of degree K reaches a given accuracy once
// the Chebyshev tail 2 (rho / 2)^(K+1) / (K+1)! is below it: K = 11 for FP64
// and 6 for FP32 at delta kappa = 1/8, on every lattice size, against V
// multiply-adds per site for the dense product.  Horner's form
//     E v = c0 y_1,  y_{K+1} = v,  y_k = v + ratio_k h y_{k+1}
// costs two additions and one multiply-add per site, component and degree.
#pragma once

#include <math.h>
#include <stddef.h>

#ifdef __CUDACC__
#define HMC_HD __host__ __device__
#else
#define HMC_HD
#endif

namespace hmc {

constexpr int kSerMax64 = 40;   // largest degree kept (FP64)
constexpr int kSerMax32 = 24;   // largest degree kept (FP32)

struct HopSeries {
    int ok;                     // the series may be used (0: the dense E only)
    int k64, k32;               // degrees
    double c0;                  // FP64 polynomial's constant, includes e^{-delta mu}
    float c0f;                  // FP32 polynomial's constant, likewise
    double r64[kSerMax64];      // r64[k-1] = c_k / c_{k-1}
    float r32[kSerMax32];
};

// Largest rho the series is used for (beyond it the degree and the growth
// e^rho of the terms make the dense product the better choice), and the
// largest L (4 cells per thread of a 256-thread block).
constexpr double kSerMaxRho = 4.0;
constexpr int kSerMaxL = 32;

// Whether the FP64 series beats the dense form, whose tiles pad V to chunks of 32
// sites: 6 k64 FP64 instructions per site, in 2 k64 steps that wait for one
// another, against 64 per chunk.  Dense / series, microseconds per CG iteration:
//   L = 5 (2 chunks)  29.8 / 28.8 at degree 11, 32.7 at 14, 36.7 at 17
//   L = 6 (3)         39.3 / 28.5 at 11, 36.3 at 17, 41.6 at 21, 46.9 at 25
//   L = 7 (4)         53.0 / 29.0 at 11, 47.0 at 25
// and of one application, which the dense form does in two launches:
//   L = 5             16.5 / 14.4 at 14, 16.5 at 17, 18.5 at 21
//   L = 6             20.6 / 16.5 at 17, 18.5 at 21, 20.5 at 23
// Up to 32 sites a slice fills a third of a warp and the dense form is ahead.
HMC_HD inline bool series_pays64(int V, int k64, bool solve) {
    return V > 32 && 2 * k64 <= (solve ? 13 : 14) * ((V + 31) / 32);
}

// Whether a solve or trajectory of Nt slices of LL cells, which could have T CTAs,
// runs on one cluster (of at most 16).  A global team's CTAs hold fewer cells, but
// its exchange grows with T, as every CTA reads every other's word.  Milliseconds of
// a solve to 1e-10 on one cluster / a global team, by the cells a CTA is spared:
//   T = 18    81 (L = 9) 1.38 / 1.42   100 (10) 1.35 / 1.35   144 (12) 1.66 / 1.57
//   T = 24    81 (9) 1.60 / 1.69       121 (11) 1.73 / 1.71   144 (12) 1.82 / 1.69
//   T = 36   128 (8) 1.87 / 1.92       162 (9) 2.24 / 2.10    288 (12) 2.88 / 2.37
//   T = 64   108 (6) 2.88 / 3.00       192 (8) 2.55 / 2.51    432 (12) 5.03 / 3.54
//   T = 96   180 (6) 3.67 / 3.74       245 (7) 2.89 / 2.61
//   T = 128  252 (6) 5.71 / 6.26       343 (7) 3.43 / 3.09
//   T = 150  324 (6) 7.20 / 7.38
// (trajectories the same to 2 %).  With at most 16 CTAs either way the cluster is
// ahead (5 to 15 %) up to 324 cells a CTA and level at 576; beyond 608 a thread has
// two cells.
constexpr int kSerCluster = 16;
HMC_HD inline bool series_on_cluster(int LL, int Nt, int T) {
    const int Tc = T < kSerCluster ? T : kSerCluster;
    if (Tc < 2) return false;
    const long long S = (Nt + Tc - 1) / Tc, Sg = (Nt + T - 1) / T;
    return S * LL <= 600 && 4 * (S - Sg) * LL <= (T > kSerCluster ? 300 + 7 * T : 0);
}

// The message numbers of a launch start after `first`: 0 for a cluster, whose boxes
// are cleared before each launch (a number that had come round to 0 would match a
// cleared box), else where the context's last launch ended -- the boxes in global
// memory then hold numbers just before it, also when it comes round.
HMC_HD inline unsigned series_first(bool cluster, unsigned last) { return cluster ? 0u : last; }

// Whether a CG vector of S slices of V sites (8 bytes each) still fits a shared
// memory of `bytes` whose first `top` are taken.  In 64 bits: one CTA may own 2^30
// site-slices.
HMC_HD inline bool vector_fits(size_t top, int S, int V, size_t bytes) {
    return top + (size_t)S * (size_t)V * 8 <= bytes;
}

// Economised power series of exp(rho t) on |t| <= 1: from the Taylor
// coefficients rho^m / m!, each power t^m above the degree is replaced by its
// best lower-degree approximation t^m - 2^{1-m} T_m(t), highest first, which
// costs 2^{1-m} times its coefficient.  Returns the smallest degree <= most
// whose dropped terms stay below tol (-1: none), coefficients in b.
inline int series_degree(double rho, double tol, int most, double* b) {
    constexpr int M = 96;       // rho <= 4: rho^96 / 96! < 1e-91
    double a[M + 1];
    a[0] = 1.0;
    for (int m = 1; m <= M; ++m) a[m] = a[m - 1] * rho / m;
    double err = 0.0;
    int K = M;
    while (K > 0) {
        const double cost = ldexp(fabs(a[K]), 1 - K);
        if (err + cost > tol) break;
        err += cost;
        // t^K = 2^{1-K} T_K - sum_{j>=1} 2^{1-K} tc_j t^{K-2j}, with the
        // coefficient of t^{K-2j} in T_K:
        //   tc_j = (-1)^j (K/2) (K-j-1)! / (j! (K-2j)!) 2^{K-2j}
        // (ratio of consecutive ones below)
        double tc = ldexp(1.0, K - 1);
        for (int j = 1; 2 * j <= K; ++j) {
            tc *= -(double)(K - 2 * j + 2) * (K - 2 * j + 1) / (4.0 * j * (K - j));
            a[K - 2 * j] -= a[K] * ldexp(tc, 1 - K);
        }
        --K;
    }
    if (K > most) return -1;
    for (int m = 0; m <= K; ++m) b[m] = a[m];
    return K;
}

// Series of exp(dk h) times f on an L x L lattice.
inline void hop_series_build(int L, double dk, double f, HopSeries* s) {
    *s = HopSeries{};
    s->c0 = f;
    const double rho = 3.0 * fabs(dk);
    if (!(rho <= kSerMaxRho) || L > kSerMaxL) return;
    double b[97];
    // tolerances relative to the smallest singular value e^{-rho} of E: a
    // tenth of a rounding of the result in each precision
    const int k64 = series_degree(rho, 2e-17 * exp(-rho), kSerMax64, b);
    if (k64 < 0) return;
    const double sg = dk < 0.0 ? -1.0 : 1.0;
    s->c0 = f * b[0];
    for (int k = 1; k <= k64; ++k) s->r64[k - 1] = sg * b[k] / b[k - 1] / 3.0;
    const int k32 = series_degree(rho, 6e-9 * exp(-rho), kSerMax32, b);
    if (k32 < 0) return;
    s->c0f = (float)(f * b[0]);
    for (int k = 1; k <= k32; ++k) s->r32[k - 1] = (float)(sg * b[k] / b[k - 1] / 3.0);
    s->k64 = k64;
    s->k32 = k32;
    s->ok = 1;
}

}  // namespace hmc
