// fp64_path.cuh -- FP64 fermion-matrix application on CUDA cores and the
// solver / force / trajectory steps built on it (device functions).
//
// Operator (exponential-hopping form of the fermion matrix, Eq. (2.2)):
//   (M psi)_t     = psi_t - s_t     E (e^{i phi_{t-1}} psi_{t-1})
//   (M^dag psi)_t = psi_t - s_{t+1} e^{-i phi_t} (E psi_{t+1}),   s_0 = -1.
//
// Two forms of E u, both bound by the FP64 issue rate of this part (2
// multiply-adds per clock and SM):
//   series  E as a polynomial of degree K of the sparse hopping (series.h),
//           6 K FP64 instructions per site (K = 11 at delta kappa = 1/8); a
//           tile is a few whole slices, hopped in shared memory;
//   dense   the real V x V times complex V x Nt product, 2 V instructions
//           per site; an output tile is TI sites x TT slices, K runs over all
//           sites in chunks of KC.  E is symmetric, so the chunk
//           E[i0.., k0..] is read as rows k of E (coalesced) and stored
//           k-major in shared memory.
// The series is used where it exists (c.ser.ok), its hop buffer fits and it pays
// (series_form); the dense form serves small lattices, an E given from
// outside, 3 |delta kappa| > 4 (at L = 5 and 6 from degree 14 or 20 on) and
// L > 27 (persistent kernels) or 32.
// Measured, one application / one CG iteration, dense -> series: L = 6,
// Nt = 32 18.3 -> 10.7 us / 41.6 -> 25.7 us; L = 12, Nt = 64 46.3 -> 13.8 /
// 95.8 -> 31; L = 24, Nt = 96 477 -> 38 / 940 -> 71; but L = 3, Nt = 8 8.1 ->
// 10.4 us, and a trajectory 13.3 -> 30 ms: nine cells fill a third of one warp,
// an FP64 instruction of a warp takes 64 clocks whatever its lanes (measured),
// and the slices' CTAs then wait for one another.
#pragma once

#include "common.cuh"
#include "ctx.h"

namespace hmc {
namespace f64 {

constexpr int TI = 32;     // sites per tile (= lanes of a warp)
constexpr int TT = 8;      // slices per tile (= warps of the CTA)
constexpr int KC = 32;     // K chunk
constexpr int NTHR = TI * TT;
static_assert(NTHR == KC * TT && (KC * TI) % NTHR == 0, "FP64 tile: chunk loads per thread");

struct Smem {
    double Et[KC][TI];     // Et[kk][ii] = E[k0+kk][i0+ii] = E[i0+ii][k0+kk]
    double2 U[TT][KC];     // source vectors of the tile's slices
};
// The dense tile's operands double as the hop buffer of the series tile.
constexpr int kHopDoubles = sizeof(Smem) / sizeof(double);

// Epilogue modes of a tile.
enum Epi : int {
    EPI_STORE = 0,       // out = M(in) (or M^dag); optional partial |out|^2
    EPI_CG_UPDATE = 1,   // M q -> Ap; x += alpha p; r -= alpha Ap; partial |r|^2
    EPI_DIRECTION = 5,   // in = r: M^dag acts on p = r + beta p_old, formed where
                         //   it is read; p and q = M^dag p stored; partial |q|^2
    EPI_RESIDUAL = 2,    // r = chi - M(in); partial |r|^2
    EPI_FORCE = 3,       // M^dag x -> y; F = phi/(dU) + 2 Im(x conj y);
                         //   store F if F != null; pi -= kick * F if pi != null
    EPI_RATIO = 4,       // M_g^dag x -> y; pi -= kick * (-2 Im(conj(y - x) chi)):
                         //   the M_g part of the ratio force of mass preconditioning
};

struct EpiArgs {
    double alpha, beta;
    double2* x;
    double2* r;
    const double2* p;      // EPI_DIRECTION: p_old
    double2* p_new;
    const double2* chi;
    const double* phi;
    double* F;
    double* pi;
    double kick;
    double inv_dU;   // 1 / (delta U)
    double hop_m1;   // hop - 1: the contraction is scaled by hop (M_g of mass
                     // preconditioning uses hop = g; 0 here is the plain M)
};

__device__ __forceinline__ int num_tiles(const ChainView& c) {
    return ((c.V + TI - 1) / TI) * ((c.Nt + TT - 1) / TT);
}

// Source element e of M / M^dag before the phase.
template <int EPI>
__device__ __forceinline__ double2 source(const double2* in, const EpiArgs& ea, size_t e) {
    const double2 v = in[e];
    if (EPI != EPI_DIRECTION) return v;
    const double2 pv = ea.p[e];
    return make_double2(fma(ea.beta, pv.x, v.x), fma(ea.beta, pv.y, v.y));
}

// What a tile does with w = E u at element o = t V + i (slice t), `hop` its
// scale, `ph` = e^{i phi} there (M^dag only).  Returns the element's share of
// the reduction.
template <bool DAG, int EPI>
__device__ __forceinline__ double finish(const ChainView& c, int t, size_t o, double2 w,
                                         double hop, double2 ph, const double2* in, double2* out,
                                         const EpiArgs& ea) {
    double sgn;
    if (DAG) {
        sgn = (t == c.Nt - 1) ? -hop : hop;
        w = cmulc(ph, w);
    } else {
        sgn = (t == 0) ? -hop : hop;
    }
    const double2 src = source<EPI>(in, ea, o);
    const double2 res = make_double2(src.x - sgn * w.x, src.y - sgn * w.y);
    if (EPI == EPI_STORE) {
        out[o] = res;
        return res.x * res.x + res.y * res.y;
    } else if (EPI == EPI_CG_UPDATE) {
        const double2 pv = ea.p[o];
        double2 xv = ea.x[o], rv = ea.r[o];
        xv.x = fma(ea.alpha, pv.x, xv.x);
        xv.y = fma(ea.alpha, pv.y, xv.y);
        rv.x = fma(-ea.alpha, res.x, rv.x);
        rv.y = fma(-ea.alpha, res.y, rv.y);
        ea.x[o] = xv;
        ea.r[o] = rv;
        return rv.x * rv.x + rv.y * rv.y;
    } else if (EPI == EPI_DIRECTION) {
        ea.p_new[o] = src;
        out[o] = res;
        return res.x * res.x + res.y * res.y;
    } else if (EPI == EPI_RESIDUAL) {
        const double2 ch = ea.chi[o];
        const double2 rv = make_double2(ch.x - res.x, ch.y - res.y);
        ea.r[o] = rv;
        return rv.x * rv.x + rv.y * rv.y;
    } else if (EPI == EPI_FORCE) {  // in = x, res = y = M^dag x
        const double f0 = ea.phi[o];
        // Im(x conj(y)) = x.y*y.x - x.x*y.y
        const double f = f0 * ea.inv_dU + 2.0 * (src.y * res.x - src.x * res.y);
        if (ea.F) ea.F[o] = f;
        if (ea.pi) ea.pi[o] -= ea.kick * f;
        return f * f;
    } else {  // EPI_RATIO: in = x, res = y = M_g^dag x, d = y - x
        const double2 ch = ea.chi[o];
        const double dx = res.x - src.x, dy = res.y - src.y;
        // Im(conj(d) chi) = d.x*chi.y - d.y*chi.x
        const double f = -2.0 * (dx * ch.y - dy * ch.x);
        ea.pi[o] -= ea.kick * f;
        return f * f;
    }
}


// ---------------------------------------------------------------- series
// A thread's cells of the tile (cell j = tid + j blockDim of the tile's
// slices, both sublattices): the A site's index in the hop buffer and those of
// the neighbours that are not in the cell.
template <int NC>
struct Cells {
    int n;                                    // cells of the tile
    int a[NC];                                // A site (its B site: a + LL)
    int bm1[NC], bm2[NC];                     // B(m1-1, m2), B(m1, m2-1)
    int ap1[NC], ap2[NC];                     // A(m1+1, m2), A(m1, m2+1)
    __device__ __forceinline__ bool has(int j) const {
        return (int)(threadIdx.x + j * blockDim.x) < n;
    }
    __device__ __forceinline__ void init(int L, int ns) {
        const int LL = L * L, V = 2 * LL;
        n = ns * LL;
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            const int cell = threadIdx.x + j * blockDim.x;
            if (!has(j)) continue;
            const int s = cell / LL, cc = cell - s * LL, m1 = cc / L, m2 = cc - m1 * L;
            const int A = s * V, B = A + LL;
            a[j] = A + cc;
            bm1[j] = B + (m1 == 0 ? L - 1 : m1 - 1) * L + m2;
            bm2[j] = B + m1 * L + (m2 == 0 ? L - 1 : m2 - 1);
            ap1[j] = A + (m1 == L - 1 ? 0 : m1 + 1) * L + m2;
            ap2[j] = A + m1 * L + (m2 == L - 1 ? 0 : m2 + 1);
        }
    }
};

// Horner on one component of the tile's cells: vA, vB hold the source and
// receive the result (without c0).  y: the tile's sites, used in place, so each
// degree has a barrier between its reads and its writes (30 clocks, against 384
// and more for a warp's six FP64 instructions per cell).  E is real, so the two
// components are independent; one at a time halves the registers and the
// buffer.
template <int NC>
__device__ __forceinline__ void hop_horner(const HopSeries& hs, const Cells<NC>& cl, int LL,
                                           double* y, double (&vA)[NC], double (&vB)[NC]) {
    double yA[NC], yB[NC];
    __syncthreads();
#pragma unroll
    for (int j = 0; j < NC; ++j)
        if (cl.has(j)) {
            yA[j] = vA[j];
            yB[j] = vB[j];
            y[cl.a[j]] = yA[j];
            y[cl.a[j] + LL] = yB[j];
        }
    for (int k = hs.k64; k >= 1; --k) {
        const double r = hs.r64[k - 1];
        __syncthreads();
#pragma unroll
        for (int j = 0; j < NC; ++j)
            if (cl.has(j)) {
                const double sA = (yB[j] + y[cl.bm1[j]]) + y[cl.bm2[j]];
                const double sB = (yA[j] + y[cl.ap1[j]]) + y[cl.ap2[j]];
                yA[j] = fma(r, sA, vA[j]);
                yB[j] = fma(r, sB, vB[j]);
            }
        if (k == 1) break;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < NC; ++j)
            if (cl.has(j)) {
                y[cl.a[j]] = yA[j];
                y[cl.a[j] + LL] = yB[j];
            }
    }
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        vA[j] = yA[j];
        vB[j] = yB[j];
    }
}

// solve: in a persistent kernel, on the hop buffer of its shared operands; else a
// standalone application, whose buffer has the slice's size.
__host__ __device__ inline bool series_form(const ChainView& c, bool solve) {
    return c.ser.ok && series_pays64(c.V, c.ser.k64, solve) && (!solve || c.V <= kHopDoubles);
}

// Slices per series tile on a hop buffer of `doubles`: enough to give every
// CTA of the team a tile, at most what the buffer and the threads take.
__device__ __forceinline__ int series_slices(const ChainView& c, int team, int doubles, int cells) {
    const int LL = c.V / 2;
    const int most = min(cells * (int)blockDim.x / LL, doubles / c.V);
    return max(1, min(most, (c.Nt + team - 1) / team));
}

// One tile of ns slices from t0 on by the series.  PHASES: e^{i phi} is
// computed here from ea.phi (standalone applications) instead of read from
// c.cis.  buf: ns V doubles.
template <bool DAG, int EPI, int NC, bool PHASES = false>
__device__ double series_tile(const ChainView& c, int t0, int ns, const double2* in, double2* out,
                              const EpiArgs& ea, double* buf) {
    const int V = c.V, LL = V / 2, Nt = c.Nt;
    Cells<NC> cl;
    cl.init(c.L, ns);
    auto phase = [&](size_t o) {
        if (!PHASES) return c.cis[o];
        double sn, cs;
        sincos(ea.phi[o], &sn, &cs);
        return make_double2(cs, sn);
    };
    double2 vA[NC], vB[NC];
#pragma unroll
    for (int j = 0; j < NC; ++j)
        if (cl.has(j)) {
            const int s = ns == 1 ? 0 : cl.a[j] / V, t = t0 + s;
            const int ts = DAG ? (t + 1 == Nt ? 0 : t + 1) : (t == 0 ? Nt - 1 : t - 1);
            const size_t o = (size_t)ts * V + (cl.a[j] - s * V);
            vA[j] = source<EPI>(in, ea, o);
            vB[j] = source<EPI>(in, ea, o + LL);
            if (!DAG) {
                vA[j] = cmul(phase(o), vA[j]);
                vB[j] = cmul(phase(o + LL), vB[j]);
            }
        }
    double a[NC], b[NC];
#pragma unroll
    for (int j = 0; j < NC; ++j) { a[j] = vA[j].x; b[j] = vB[j].x; }
    hop_horner(c.ser, cl, LL, buf, a, b);
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        vA[j].x = a[j]; vB[j].x = b[j];
        a[j] = vA[j].y; b[j] = vB[j].y;
    }
    hop_horner(c.ser, cl, LL, buf, a, b);
#pragma unroll
    for (int j = 0; j < NC; ++j) { vA[j].y = a[j]; vB[j].y = b[j]; }
    const double hop = (1.0 + ea.hop_m1) * c.ser.c0;
    double acc = 0.0;
#pragma unroll
    for (int j = 0; j < NC; ++j)
        if (cl.has(j)) {
            const int s = ns == 1 ? 0 : cl.a[j] / V, t = t0 + s;
            const size_t o = (size_t)t0 * V + cl.a[j];
            const double2 none = make_double2(1.0, 0.0);
            acc += finish<DAG, EPI>(c, t, o, vA[j], hop, DAG ? phase(o) : none, in, out, ea);
            acc += finish<DAG, EPI>(c, t, o + LL, vB[j], hop, DAG ? phase(o + LL) : none, in, out,
                                    ea);
        }
    return acc;
}

// ---------------------------------------------------------------- dense
// One output tile.  `in` is the vector M (DAG=false) or M^dag (DAG=true)
// acts on.  Returns this thread's contribution to the tile's reduction.
template <bool DAG, int EPI>
__device__ double apply_tile(const ChainView& c, int tile, const double2* __restrict__ in,
                             double2* __restrict__ out, const EpiArgs& ea, Smem& sm) {
    const int V = c.V, Nt = c.Nt;
    const int nti = (V + TI - 1) / TI;
    const int i0 = (tile % nti) * TI, t0 = (tile / nti) * TT;
    const int ii = threadIdx.x & (TI - 1), tt = threadIdx.x / TI;
    const double* __restrict__ E = c.E;
    const double2* __restrict__ cis = c.cis;
    // Chunk k0's E block and source values are loaded into registers while
    // the previous chunk is contracted from shared memory (one buffer: the
    // registers are the second stage), so the L2 latency of a chunk hides
    // behind the FP64 arithmetic of the one before.  The summation order is
    // that of a plain loop over k.
    constexpr int kEPer = KC * TI / NTHR;   // E elements per thread and chunk
    const int ukk = threadIdx.x % KC, us = threadIdx.x / KC;
    double ev[kEPer];
    double2 uv;
    auto fetch = [&](int k0) {
#pragma unroll
        for (int j = 0; j < kEPer; ++j) {
            const int e = threadIdx.x + j * NTHR;
            const int kk = e / TI, cc = e % TI;
            const int k = k0 + kk, i = i0 + cc;
            ev[j] = (k < V && i < V) ? E[(size_t)k * V + i] : 0.0;
        }
        const int k = k0 + ukk, tq = t0 + us;
        uv = make_double2(0.0, 0.0);
        if (k < V && tq < Nt) {
            if (DAG) {
                const int ts = (tq + 1 == Nt) ? 0 : tq + 1;
                uv = source<EPI>(in, ea, (size_t)ts * V + k);
            } else {
                const int ts = (tq == 0) ? Nt - 1 : tq - 1;
                uv = cmul(cis[(size_t)ts * V + k], in[(size_t)ts * V + k]);
            }
        }
    };
    double ar = 0.0, ai = 0.0;
    fetch(0);
    for (int k0 = 0; k0 < V; k0 += KC) {
#pragma unroll
        for (int j = 0; j < kEPer; ++j) {
            const int e = threadIdx.x + j * NTHR;
            sm.Et[e / TI][e % TI] = ev[j];
        }
        sm.U[us][ukk] = uv;
        __syncthreads();
        if (k0 + KC < V) fetch(k0 + KC);
#pragma unroll 8
        for (int kk = 0; kk < KC; ++kk) {
            const double e = sm.Et[kk][ii];
            const double2 u = sm.U[tt][kk];
            ar = fma(e, u.x, ar);
            ai = fma(e, u.y, ai);
        }
        __syncthreads();
    }
    const int i = i0 + ii, t = t0 + tt;
    if (i >= V || t >= Nt) return 0.0;
    const size_t o = (size_t)t * V + i;
    return finish<DAG, EPI>(c, t, o, make_double2(ar, ai), 1.0 + ea.hop_m1,
                            DAG ? cis[o] : make_double2(1.0, 0.0), in, out, ea);
}

// Which form of E a kernel is compiled with: FORM_EITHER decides per chain;
// FORM_WIDE is the series in blocks of up to 640 threads with at least half a
// thread per cell of a slice (series_cg.cuh).
enum Form : int { FORM_DENSE = 0, FORM_SERIES = 1, FORM_EITHER = 2, FORM_WIDE = 3 };

template <bool DAG, int EPI>
__device__ __forceinline__ double dense_team(const ChainView& c, const Team& tm,
                                             const double2* in, double2* out,
                                             const EpiArgs& ea, Smem& sm) {
    double acc = 0.0;
    const int nt = num_tiles(c);
    for (int tile = tm.rank; tile < nt; tile += tm.size)
        acc += apply_tile<DAG, EPI>(c, tile, in, out, ea, sm);
    return acc;
}

// Not inlined: the persistent kernels apply M and M^dag in many places, and a
// copy of the series tile in each spilled 2-8 KB of stack per thread.  The
// chain view is a __grid_constant__ parameter and the team goes by value, so
// the call leaves neither in the caller's local memory.
template <int FORM, bool DAG, int EPI>
__device__ __noinline__ double series_team(const ChainView& c, const Team tm, const double2* in,
                                           double2* out, const EpiArgs& ea, Smem& sm) {
    if (FORM == FORM_EITHER && !series_form(c, true))
        return dense_team<DAG, EPI>(c, tm, in, out, ea, sm);
    double acc = 0.0;
    // (V <= kHopDoubles: at most 768 cells; 256 threads, or at least half of
    // the cells)
    constexpr int NC = FORM == FORM_WIDE ? 2 : 3;
    const int ns = series_slices(c, tm.size, kHopDoubles, NC);
    for (int t0 = tm.rank * ns; t0 < c.Nt; t0 += tm.size * ns)
        acc += series_tile<DAG, EPI, NC>(c, t0, min(ns, c.Nt - t0), in, out, ea, &sm.Et[0][0]);
    return acc;
}

// All tiles of one application, spread over the team.
template <int FORM, bool DAG, int EPI>
__device__ __forceinline__ double apply_team(const ChainView& c, const Team& tm,
                                             const double2* in, double2* out,
                                             const EpiArgs& ea, Smem& sm) {
    if constexpr (FORM == FORM_DENSE)
        return dense_team<DAG, EPI>(c, tm, in, out, ea, sm);
    else
        return series_team<FORM, DAG, EPI>(c, tm, in, out, ea, sm);
}

#define HMC_TEAM_ELEMS(e, c, tm) \
    for (int e = (tm).rank * blockDim.x + threadIdx.x; e < (c).N; e += (tm).size * blockDim.x)

struct CgResult {
    int iterations;
    double true_res;   // |chi - M M^dag x| / |chi|
    int status;
};

// Conjugate gradient on M M^dag (FP64; with hop_m1 != 0 on M_g M_g^dag, the
// contraction scaled by 1 + hop_m1), CG vectors in the chain workspace
// (r, p, q), from x = 0 or (warm) from the x given, whose residual
// chi - M M^dag x then starts the iteration.  cis must hold exp(i phi).
// The new direction p = r + beta p is formed inside the M^dag application, where
// it is read and (into a second buffer) where it is owned, so an iteration has
// two team sums and no barrier of its own for the direction (series).
// Ends with the FP64 true residual, which leaves chi - M M^dag x in r and
// M^dag x in q.
template <int FORM>
__device__ inline bool cg_solve(const ChainView& c, Team& tm, const double2* chi, double2* x,
                         double tol, int max_iter, CgResult& res, Smem& sm,
                         bool warm = false, double hop_m1 = 0.0) {
    double2 *r = c.r, *p = c.p, *pn = c.p2, *q = c.q;
    double v1[1] = {0.0};
    HMC_TEAM_ELEMS(e, c, tm) {
        const double2 ch = chi[e];
        if (!warm) {
            x[e] = make_double2(0.0, 0.0);
            r[e] = ch;
            p[e] = FORM == FORM_DENSE ? ch : make_double2(0.0, 0.0);
        }
        v1[0] += ch.x * ch.x + ch.y * ch.y;
    }
    if (!team_sum<1>(tm, v1)) return false;
    const double chi2 = v1[0];
    double rr = chi2;
    res.iterations = 0;
    res.status = HMC_OK;
    res.true_res = 0.0;
    if (!(chi2 > 0.0)) {
        if (!finite_d(chi2)) res.status = HMC_ERR_NONFINITE;
        return true;
    }
    const double stop = tol * tol * chi2;
    EpiArgs ea = {};
    ea.x = x;
    ea.r = r;
    ea.p = p;
    ea.hop_m1 = hop_m1;
    if (warm) {
        // r = chi - M (M^dag x), p = r
        apply_team<FORM, true, EPI_STORE>(c, tm, x, q, ea, sm);
        if (!team_barrier(tm)) return false;
        ea.chi = chi;
        double vr[1] = {apply_team<FORM, false, EPI_RESIDUAL>(c, tm, q, nullptr, ea, sm)};
        if (!team_sum<1>(tm, vr)) return false;
        rr = vr[0];
        HMC_TEAM_ELEMS(e, c, tm) p[e] = FORM == FORM_DENSE ? r[e] : make_double2(0.0, 0.0);
        if (!team_barrier(tm)) return false;
        if (!finite_d(rr)) res.status = HMC_ERR_NONFINITE;
    }
    int it = 0;
    bool conv = res.status == HMC_OK && rr <= stop;
    while (!conv && res.status == HMC_OK && it < max_iter) {
        double vq[1];
        ea.p = p;
        if constexpr (FORM == FORM_DENSE) {
            vq[0] = apply_team<FORM, true, EPI_STORE>(c, tm, p, q, ea, sm);   // q = M^dag p
            if (!team_sum<1>(tm, vq)) return false;
        } else {
            // p = r + beta p, q = M^dag p
            ea.p_new = pn;
            vq[0] = apply_team<FORM, true, EPI_DIRECTION>(c, tm, r, q, ea, sm);
            if (!team_sum<1>(tm, vq)) return false;
            pn = p;
            p = ea.p_new;
            ea.p = p;
        }
        const double qq = vq[0];
        if (!finite_d(qq) || !(qq > 0.0)) { res.status = HMC_ERR_NONFINITE; break; }
        ea.alpha = rr / qq;
        double vr[1] = {apply_team<FORM, false, EPI_CG_UPDATE>(c, tm, q, nullptr, ea, sm)};
        if (!team_sum<1>(tm, vr)) return false;
        const double rr_new = vr[0];
        ++it;
        if (!finite_d(rr_new)) { res.status = HMC_ERR_NONFINITE; break; }
        if (rr_new <= stop) { conv = true; break; }
        ea.beta = rr_new / rr;
        rr = rr_new;
        if constexpr (FORM == FORM_DENSE) {
            // (the dense kernels run small lattices on one CTA: a barrier is cheap
            // there, forming p twice in FP64 is not: 1.5 % of an L = 3 trajectory)
            HMC_TEAM_ELEMS(e, c, tm) {
                const double2 rv = r[e], pv = p[e];
                p[e] = make_double2(fma(ea.beta, pv.x, rv.x), fma(ea.beta, pv.y, rv.y));
            }
            if (!team_barrier(tm)) return false;
        }
    }
    res.iterations = it;
    if (res.status == HMC_OK && !conv) res.status = HMC_ERR_CG_NOT_CONVERGED;
    // FP64 true residual r = chi - M (M^dag x)
    if (!team_barrier(tm)) return false;
    apply_team<FORM, true, EPI_STORE>(c, tm, x, q, ea, sm);
    if (!team_barrier(tm)) return false;
    ea.chi = chi;
    double vt[1] = {apply_team<FORM, false, EPI_RESIDUAL>(c, tm, q, nullptr, ea, sm)};
    if (!team_sum<1>(tm, vt)) return false;
    res.true_res = sqrt(vt[0] / chi2);
    if (!finite_d(res.true_res)) res.status = HMC_ERR_NONFINITE;
    return true;
}

}  // namespace f64
}  // namespace hmc
