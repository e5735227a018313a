// mixed_path.cuh -- the mixed-precision solver and trajectory, for every kind
// of FP32 iteration: FP32 conjugate gradient with FP64 reliable updates, and
// the HMC trajectory built on it.  FP64 stays for the true residual, chi = M rho,
// the force, the Hamiltonian sums and Metropolis.
#pragma once

#include "cg_scalars.cuh"
#include "fp64_path.cuh"
#include "launch.h"
#include "series_cg.cuh"
#include "small_cg.cuh"
#include "tc_splitk.cuh"
#include "tc_tile.cuh"
#include "tc_wide.cuh"

namespace hmc {
namespace tc {

// ---------------------------------------------------------------- epilogues
// Each epilogue splits into load (global reads of what output (t, i) needs)
// and store (arithmetic and writes), so the tile can batch the reads.
template <bool DAG>
struct EpiStore {
    const float2* in;
    float2* out;
    const float2* cis;
    int V, Nt;
    float acc;   // per-thread partial |out|^2 (at most 32 terms; FP32 suffices)
    struct In {
        float2 s, ph;
    };
    __device__ __forceinline__ In load(int i, int t) const {
        const size_t o = (size_t)t * V + i;
        In v;
        v.s = in[o];
        v.ph = DAG ? cis[o] : make_float2(1.f, 0.f);
        return v;
    }
    __device__ __forceinline__ void store(int i, int t, const In& v, float2 w) {
        float sg;
        if (DAG) {
            sg = (t == Nt - 1) ? -1.f : 1.f;
            w = cmulcf(v.ph, w);
        } else {
            sg = (t == 0) ? -1.f : 1.f;
        }
        const float2 r = make_float2(v.s.x - sg * w.x, v.s.y - sg * w.y);
        out[(size_t)t * V + i] = r;
        acc = fmaf(r.x, r.x, fmaf(r.y, r.y, acc));
    }
    // sites i, i+1 (i even) with 16-byte accesses
    struct In2 {
        float4 s, ph;
    };
    __device__ __forceinline__ In2 load2(int i, int t) const {
        const size_t o = (size_t)t * V + i;
        In2 v;
        v.s = *reinterpret_cast<const float4*>(in + o);
        v.ph = DAG ? *reinterpret_cast<const float4*>(cis + o) : make_float4(1.f, 0.f, 1.f, 0.f);
        return v;
    }
    __device__ __forceinline__ void store2(int i, int t, const In2& v, float2 w0, float2 w1) {
        float sg;
        if (DAG) {
            sg = (t == Nt - 1) ? -1.f : 1.f;
            w0 = cmulcf(make_float2(v.ph.x, v.ph.y), w0);
            w1 = cmulcf(make_float2(v.ph.z, v.ph.w), w1);
        } else {
            sg = (t == 0) ? -1.f : 1.f;
        }
        const float4 r = make_float4(v.s.x - sg * w0.x, v.s.y - sg * w0.y, v.s.z - sg * w1.x,
                                     v.s.w - sg * w1.y);
        *reinterpret_cast<float4*>(out + (size_t)t * V + i) = r;
        acc = fmaf(r.x, r.x, fmaf(r.y, r.y, acc));
        acc = fmaf(r.z, r.z, fmaf(r.w, r.w, acc));
    }
};

// M q -> Ap; x_f += alpha p; r_f -= alpha Ap; accumulates |r_f|^2.
struct EpiCgUpdate {
    const float2* q;
    const float2* p;
    float2* x;
    float2* r;
    float alpha;
    int V;
    float acc;   // per-thread partial |r|^2
    struct In {
        float2 q, p, x, r;
    };
    __device__ __forceinline__ In load(int i, int t) const {
        const size_t o = (size_t)t * V + i;
        In v;
        v.q = q[o];
        v.p = p[o];
        v.x = x[o];
        v.r = r[o];
        return v;
    }
    __device__ __forceinline__ void store(int i, int t, const In& v, float2 w) {
        const size_t o = (size_t)t * V + i;
        const float sg = (t == 0) ? -1.f : 1.f;
        const float2 ap = make_float2(v.q.x - sg * w.x, v.q.y - sg * w.y);
        float2 xv = v.x, rv = v.r;
        xv.x = fmaf(alpha, v.p.x, xv.x);
        xv.y = fmaf(alpha, v.p.y, xv.y);
        rv.x = fmaf(-alpha, ap.x, rv.x);
        rv.y = fmaf(-alpha, ap.y, rv.y);
        x[o] = xv;
        r[o] = rv;
        acc = fmaf(rv.x, rv.x, fmaf(rv.y, rv.y, acc));
    }
    struct In2 {
        float4 q, p, x, r;
    };
    __device__ __forceinline__ In2 load2(int i, int t) const {
        const size_t o = (size_t)t * V + i;
        In2 v;
        v.q = *reinterpret_cast<const float4*>(q + o);
        v.p = *reinterpret_cast<const float4*>(p + o);
        v.x = *reinterpret_cast<const float4*>(x + o);
        v.r = *reinterpret_cast<const float4*>(r + o);
        return v;
    }
    __device__ __forceinline__ void store2(int i, int t, const In2& v, float2 w0, float2 w1) {
        const size_t o = (size_t)t * V + i;
        const float sg = (t == 0) ? -1.f : 1.f;
        const float4 ap = make_float4(v.q.x - sg * w0.x, v.q.y - sg * w0.y, v.q.z - sg * w1.x,
                                      v.q.w - sg * w1.y);
        const float4 xv = make_float4(fmaf(alpha, v.p.x, v.x.x), fmaf(alpha, v.p.y, v.x.y),
                                      fmaf(alpha, v.p.z, v.x.z), fmaf(alpha, v.p.w, v.x.w));
        const float4 rv = make_float4(fmaf(-alpha, ap.x, v.r.x), fmaf(-alpha, ap.y, v.r.y),
                                      fmaf(-alpha, ap.z, v.r.z), fmaf(-alpha, ap.w, v.r.w));
        *reinterpret_cast<float4*>(x + o) = xv;
        *reinterpret_cast<float4*>(r + o) = rv;
        acc = fmaf(rv.x, rv.x, fmaf(rv.y, rv.y, acc));
        acc = fmaf(rv.z, rv.z, fmaf(rv.w, rv.w, acc));
    }
};

// CG direction step fused into M^dag: at the tile's own (t, i) form
// p_new = r + beta p_old (r from the FP64 residual after a reliable update,
// which is then also stored as the new FP32 r), store p_new, and
// q = M^dag p_new = p_new - s_{t+1} e^{-i phi_t} w; accumulates |q|^2.
struct EpiDirection {
    SrcDirection d;
    float2* p_new;
    float2* r_out;     // written when d.refresh
    float2* q;
    const float2* cis;
    int Nt;
    float acc;   // per-thread partial |q|^2
    struct In {
        float2 r, p, ph;
    };
    __device__ __forceinline__ In load(int i, int t) const {
        const size_t o = (size_t)t * d.V + i;
        In v;
        if (d.refresh) {
            const double2 r64 = d.r64[o];
            v.r = make_float2((float)r64.x, (float)r64.y);
        } else {
            v.r = d.r[o];
        }
        v.p = d.p_old[o];
        v.ph = cis[o];
        return v;
    }
    __device__ __forceinline__ void store(int i, int t, const In& v, float2 w) {
        const size_t o = (size_t)t * d.V + i;
        const float2 pv = make_float2(fmaf(d.beta, v.p.x, v.r.x), fmaf(d.beta, v.p.y, v.r.y));
        if (d.refresh) r_out[o] = v.r;
        p_new[o] = pv;
        const float sg = (t == Nt - 1) ? -1.f : 1.f;
        w = cmulcf(v.ph, w);
        const float2 qv = make_float2(pv.x - sg * w.x, pv.y - sg * w.y);
        q[o] = qv;
        acc = fmaf(qv.x, qv.x, fmaf(qv.y, qv.y, acc));
    }
    struct In2 {
        float4 r, p, ph;
    };
    __device__ __forceinline__ In2 load2(int i, int t) const {
        const size_t o = (size_t)t * d.V + i;
        In2 v;
        if (d.refresh) {
            const double2 a = d.r64[o], b = d.r64[o + 1];
            v.r = make_float4((float)a.x, (float)a.y, (float)b.x, (float)b.y);
        } else {
            v.r = *reinterpret_cast<const float4*>(d.r + o);
        }
        v.p = *reinterpret_cast<const float4*>(d.p_old + o);
        v.ph = *reinterpret_cast<const float4*>(cis + o);
        return v;
    }
    __device__ __forceinline__ void store2(int i, int t, const In2& v, float2 w0, float2 w1) {
        const size_t o = (size_t)t * d.V + i;
        const float4 pv = make_float4(fmaf(d.beta, v.p.x, v.r.x), fmaf(d.beta, v.p.y, v.r.y),
                                      fmaf(d.beta, v.p.z, v.r.z), fmaf(d.beta, v.p.w, v.r.w));
        if (d.refresh) *reinterpret_cast<float4*>(r_out + o) = v.r;
        *reinterpret_cast<float4*>(p_new + o) = pv;
        const float sg = (t == Nt - 1) ? -1.f : 1.f;
        w0 = cmulcf(make_float2(v.ph.x, v.ph.y), w0);
        w1 = cmulcf(make_float2(v.ph.z, v.ph.w), w1);
        const float4 qv = make_float4(pv.x - sg * w0.x, pv.y - sg * w0.y, pv.z - sg * w1.x,
                                      pv.w - sg * w1.y);
        *reinterpret_cast<float4*>(q + o) = qv;
        acc = fmaf(qv.x, qv.x, fmaf(qv.y, qv.y, acc));
        acc = fmaf(qv.z, qv.z, fmaf(qv.w, qv.w, acc));
    }
};

__device__ __forceinline__ void tile_coords(int tile, int nti, int ns_tile, int Nt, int& i0,
                                            int& t0, int& ns) {
    i0 = (tile % nti) * TM;
    t0 = (tile / nti) * ns_tile;
    ns = min(ns_tile, Nt - t0);
}

// All tensor-core tiles of one application, spread over the team.
template <bool DAG, class Src, class Epi>
__device__ bool apply_team(const ChainView& c, const Team& tm, TcState& st,
                           const CUtensorMap* mhi, const CUtensorMap* mlo, int ns_tile,
                           const Src& src, float scale, float inv, Epi& epi,
                           bool res_b = false) {
    const int nti = c.Vr / TM, ntt = (c.Nt + ns_tile - 1) / ns_tile;
    // tiles are dealt round robin over the team; in resident mode the team
    // size is a multiple of the site blocks, so a CTA only meets tiles of
    // its own site block (rank mod nti), whose rows of E it holds.  With a
    // resident B, slice tiles go round robin and a CTA runs all site blocks
    // of each of its slice tiles, building that B once.  One call site of
    // the tile keeps it inlined once.
    for (int j = 0;; ++j) {
        int i0, t0, ns, rflag = 0;
        if (res_b) {
            const int stl = tm.rank + (j / nti) * tm.size, rb = j % nti;
            if (stl >= ntt) break;
            i0 = rb * TM;
            t0 = stl * ns_tile;
            ns = min(ns_tile, c.Nt - t0);
            rflag = rb == 0 ? 1 : 2;
        } else {
            const int tile = tm.rank + j * tm.size;
            if (tile >= nti * ntt) break;
            tile_coords(tile, nti, ns_tile, c.Nt, i0, t0, ns);
        }
        if (!tc_tile<DAG>(st, mhi, mlo, c.V, c.Nt, c.Vp, i0, t0, ns, src, scale, inv, epi, rflag))
            return false;
    }
    return true;
}

// All slice-major tiles of one application (W sites x ns_tile slices each),
// dealt round robin over the team.
template <bool DAG, class Src, class Epi>
__device__ bool apply_team_w(const ChainView& c, const Team& tm, TcState& st, int W,
                             const CUtensorMap* mhi, const CUtensorMap* mlo, int ns_tile,
                             const Src& src, float scale, float inv, Epi& epi) {
    const WideGeom g = wide_geom(W);
    const int nsi = (c.V + W - 1) / W, ntt = (c.Nt + ns_tile - 1) / ns_tile;
    for (int tile = tm.rank; tile < nsi * ntt; tile += tm.size) {
        const int i0 = (tile % nsi) * W, t0 = (tile / nsi) * ns_tile;
        const int ns = min(ns_tile, c.Nt - t0);
        if (!tc_wtile<DAG>(st, g, mhi, mlo, c.V, c.Nt, c.Vp, i0, t0, ns, src, scale, inv,
                           c.e_inv, epi))
            return false;
    }
    return true;
}

// ---------------------------------------------------------------- mixed CG
struct MixedResult {
    int iterations;
    int reliable_updates;
    double true_res;
    int status;
    int fp64_iterations;   // iterations of the FP64 fallback (0 if it did not run)
};

struct PersistentArgs {
    int ns_tile;
    int inner;         // CTAs of the FP32 inner loop
    int cluster;       // > 1: launched in clusters of this size, the inner team is cluster 0
    int res_b;         // streaming layout: resident B per slice tile (apply_team)
    int mode;          // OperandMode: resident needs inner a multiple of the site blocks
    int wide_W;        // kSlice: sites per slice-major tile
    int vec_resident;  // resident mode with one CTA: FP32 CG vectors in shared memory
    double tol;
    int max_iter;
    double ru_delta;
    int ru_every;      // reliable update after this many FP32 iterations at the latest
    int sk_C;          // kSplitK: CTAs per cluster splitting K (ns_tile: slices per n-group)
};

// Form of E in the FP64 steps of a kernel of kind KIND: the tensor-core tiles
// whose FP32 loop is inlined keep the dense form, because a kernel with the
// series in it gives that loop fewer registers (10-20 % of its time); the
// split-K loop is a function of its own and takes the series where it exists.
// Kernel kinds of the FP32 iterations: site-major tensor-core tiles, the
// CUDA-core cluster solver, slice-major and split-K tensor-core tiles, and the
// polynomial of the sparse hopping (series_cg.cuh).
enum TileKind : int { kKindSite = 0, kKindSmall = 1, kKindSlice = 2, kKindSplitK = 3,
                      kKindSeries = 4 };
template <int KIND>
constexpr int kForm = KIND == kKindSeries   ? f64::FORM_WIDE
                      : KIND == kKindSplitK ? f64::FORM_EITHER
                                            : f64::FORM_DENSE;

// FP64 true residual of x64: r64 = chi - M (M^dag x64); returns |r64|^2.
template <int FORM>
__device__ bool f64_residual(const ChainView& c, Team& tm, f64::Smem& sm, const double2* chi,
                             double2* x64, double& rr, double gm1 = 0.0) {
    f64::EpiArgs ea = {};
    ea.hop_m1 = gm1;   // M_g = 1 - g S E D with g = 1 + gm1 (mass preconditioning)
    f64::apply_team<FORM, true, f64::EPI_STORE>(c, tm, x64, c.q, ea, sm);
    if (!team_barrier(tm)) return false;
    ea.chi = chi;
    ea.r = c.r;
    double v[1] = {f64::apply_team<FORM, false, f64::EPI_RESIDUAL>(c, tm, c.q, nullptr, ea, sm)};
    if (!team_sum<1>(tm, v)) return false;
    rr = v[0];
    return true;
}

// FP32 CG on the tensor-core operator with FP64 reliable updates
// (Sleijpen-van der Vorst style, as used in lattice QCD solvers): whenever
// the iterated residual has dropped by ru_delta since the last update, or
// claims convergence, the FP32 increment is folded into the FP64 solution,
// the true residual chi - M M^dag x is recomputed in FP64 and replaces the
// iterated one; the search direction is kept.  Stops on the FP64 true
// residual.
//
// Two teams: the FP32 iterations run on the first `inner` CTAs (one CTA
// for small lattices, so an iteration needs no inter-CTA barrier), the FP64
// steps on all CTAs of the launch (FP64 is ~1/1700 of the tensor rate, so it
// is spread over as many SMs as possible).  The other CTAs wait at the
// outer barrier while the inner loop runs.  Two inner synchronisations per
// iteration: the direction update p = r + beta p happens inside the M^dag
// application (operand build and epilogue, into a second p buffer), the
// x / r update inside the M one.  Needs c.cis and c.cis_f of the current phi.
// FP32 CG iterations of one segment (until a reliable update, max_iter or
// a non-finite norm) on split-K tiles with E' resident: M^dag contracts r
// (G = E r + beta G carried by the owners), M contracts u = e^{i phi} q.
// The owner vectors live in shared memory for the segment: r is loaded from
// the FP32 residual (or, refresh, the FP64 residual, also written back as
// FP32), p and G start at zero in the first segment of a solve and carry
// over otherwise, x (the FP32 increment) starts at zero and is folded into
// x64 by its owner at the end.
//
// Each application: wait for the owners of this CTA's K range (their posted
// words), copy and split the source with the scale from their largest
// exponent, issue the MMAs; meanwhile warp 0 sums the norm that the previous
// epilogue posted and thread 0 updates the scalars (alpha after |q|^2;
// beta, or the end of the segment, after |r|^2); then stage the partial,
// and, unless the segment ends, sync the cluster, reduce and run the
// epilogue, which writes the next source and posts its norm.  The decision
// to end the segment therefore comes after the next M^dag's MMAs are issued;
// their result is drained and dropped.  Returns the segment's end reason,
// or -1 if a bounded wait failed.  Not inlined into the persistent kernels:
// the iteration gets its own register budget.
static __device__ __noinline__ int sk_segment(const ChainView& c, Team& ti, TcState& st,
                                       const PersistentArgs& pa, ClusterSync* ics,
                                       CgScalars& s_cg, bool refresh, bool first,
                                       const float2* cisf, double2* x64, float hop) {
    int reason = kSegMaxIter;
    const SkGeom g = sk_geom(ti.rank, pa.sk_C, pa.ns_tile, c.V, c.Nt, c.Vr, c.Vp);
    Team tcl = ti;
    tcl.rank = g.rank;
    tcl.size = g.C;
    tcl.cs = ics;
    SkOwner ow;
    ow.init(st.base, g);
    // the CTAs whose posts this CTA waits for: owners of the M^dag source (r)
    // and of the M source (u), and the other members of its cluster
    __shared__ int s_own[2][kSkMaxOwners];
    __shared__ int s_nown[2];
    __shared__ unsigned s_mexp;
    const CUtensorMap* maps = reinterpret_cast<const CUtensorMap*>(c.sk_maps);
    if (threadIdx.x == 0) {
        s_nown[0] = sk_owner_list(g, c.V, c.Nt, true, s_own[0], ti.rank);
        s_nown[1] = sk_owner_list(g, c.V, c.Nt, false, s_own[1], ti.rank);
        if (s_nown[0] < 0 || s_nown[1] < 0 || !maps) set_status(ti.status, HMC_ERR_UNSUPPORTED);
        if (maps)
            for (int m = 0; m < 6; ++m)
                asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(maps + m)
                             : "memory");
    }
    float2* rh = c.rh_f;   // r with the halo rows (source of M^dag)
    float mx = 0.f;
    HMC_SK_OWNED(o, oi, g, c) {
        float2 rv;
        if (refresh) {
            const double2 d = c.r[o];
            rv = make_float2((float)d.x, (float)d.y);
        } else {
            rv = c.r_f[o];
        }
        mx = fmaxf(mx, fmaxf(fabsf(rv.x), fabsf(rv.y)));
        const int t = (int)(o / (size_t)c.V);
        rh[o + c.V] = rv;                                        // row t + 1
        if (t == 0) rh[o + (size_t)(c.Nt + 1) * c.V] = rv;      // row Nt + 1
        ow.r[oi] = rv;
        ow.x[oi] = make_float2(0.f, 0.f);
        if (first) {
            ow.p[oi] = make_float2(0.f, 0.f);
            ow.G[oi] = make_float2(0.f, 0.f);
        }
    }
    sk_post(ti, c.gslots, ++st.gseq, 0.f, mx);   // r ready (no norm: beta is the caller's)
    if (team_failed(ti)) return -1;
    bool have_rr = false;
    const int warp = threadIdx.x >> 5;
    // Predicted operand exponents: s_pe[k] for the next source of kind k
    // (0: r, 1: u) from the team's largest exponent of its last one (every
    // CTA computes the same value from the same slots); s_pw[k]: the exponent
    // the owners used for the FP16 split of the last posted source of kind
    // k, or kNoPe if they wrote none (the segment's first r is FP32 only).
    constexpr int kNoPe = -1000;
    __shared__ int s_pe[2], s_pw[2];
    if (threadIdx.x == 0) {
        if (first) s_pe[0] = s_pe[1] = kNoPe;
        s_pw[0] = s_pw[1] = kNoPe;
    }
    // (the post above ended with a block barrier; these are read after the next)
    __half_raw* const b16 = c.sk_b16;
    const size_t plane = (size_t)2 * (c.Nt + 2) * c.Vp;
    // One application of kind `list` (0: M^dag, source r, halo rows t0 + 2 ..;
    // 1: M, source u, rows t0 ..): wait for the owners' words of seq; take
    // the owners' FP16 split by TMA when its exponent is known and the
    // owners' largest component scaled by it is in [2^4, 2^15) (no overflow,
    // full precision), else the FP32 source by TMA split here with the scale
    // from the owners' exponent; issue the MMAs.  Warp 1 sums the norm of seq
    // (into *out) and the team's largest exponent (into *gm) meanwhile.
    auto contract = [&](int list, float* out, unsigned* gm, float& inv) -> bool {
        if (warp == 0) {
            unsigned m = 0;
            const bool ok =
                sk_wait_owners(ti, c.gslots, st.gseq, s_own[list], s_nown[list], 0u, m);
            if ((threadIdx.x & 31) == 0) s_mexp = ok ? m : 0xffffffffu;
        }
        __syncthreads();
        const unsigned mexp = s_mexp;
        if (mexp == 0xffffffffu) return false;
        SkSum ss;
        if (warp == 1) sk_sum_begin(ti, c.gslots, st.gseq, ss);
        const int pw = s_pw[list];
        const int top = (int)mexp - 127 + pw;
        const bool fast = b16 && pw != kNoPe && mexp != 0xffu && (mexp == 0u || (top >= 4 && top <= 14));
        bool ok = true;
        const int row0 = list == 0 ? g.t0 + 2 : g.t0;
        if (fast) {
            inv = __int_as_float((127 - pw) << 23);
            sk_issue_b16(st, g, maps + 2 + 2 * list, maps + 3 + 2 * list, 2 * row0,
                         st.bars->tmem_base);
        } else {
            float sc;
            sk_scale(mexp, sc, inv);
            sk_issue_source(st, g, maps + list, row0);
            ok = sk_convert_and_issue(st, g, sc, st.bars->tmem_base);
        }
        if (ok && warp == 1) {
            float v = 0.f;
            unsigned gmx = 0;
            const bool oks = sk_sum_end(ti, c.gslots, st.gseq, ss, v, gmx);
            if ((threadIdx.x & 31) == 0) {
                *out = oks ? v : __int_as_float(0x7fc00000);
                *gm = gmx;
            }
        }
        return ok;
    };
    // predicted exponent of the next source of a kind whose largest
    // component had biased exponent gm: that component times 2^e in [2^12, 2^13)
    auto predict = [](unsigned gm) -> int {
        if (gm == 0u || gm == 0xffu) return kNoPe;
        return max(-120, min(120, 12 - ((int)gm - 127)));
    };
    __shared__ float s_norm;
    __shared__ unsigned s_gm;
    while (s_cg.it < pa.max_iter) {
        float inv;
        // ---- M^dag p' (p' = r + beta p): contract r
        if (!contract(0, &s_norm, &s_gm, inv)) return -1;
        __syncthreads();
        if (threadIdx.x == 0) {
            s_pe[0] = predict(s_gm);
            if (have_rr) {
                cg_after_r(s_cg, s_norm);
                if (s_cg.reason == 0 && s_cg.it >= pa.max_iter) s_cg.reason = kSegMaxIter;
            }
        }
        if (!sk_stage(st, g, inv)) return -1;   // its barrier publishes s_cg, s_pe
        if (team_failed(ti)) return -1;
        if (have_rr && s_cg.reason != 0) { reason = s_cg.reason; break; }
        const int pu = s_pe[1];
        SkEpiDag ed{ow, c.u_f, pu != kNoPe ? b16 + 2 * plane : nullptr, b16 + 3 * plane,
                    __int_as_float((127 + (pu != kNoPe ? pu : 0)) << 23), c.Vp,
                    cisf, s_cg.beta, hop, c.V, c.Nt, 0.f, 0.f};
        if (!sk_reduce<false>(st, g, tcl, c.V, c.e_inv, ed)) return -1;
        if (threadIdx.x == 0) s_pw[1] = b16 ? pu : kNoPe;
        sk_post(ti, c.gslots, ++st.gseq, ed.acc, ed.mx);   // u ready, |q|^2
        // ---- M q: contract u = e^{i phi} q
        if (!contract(1, &s_norm, &s_gm, inv)) return -1;
        __syncthreads();
        if (threadIdx.x == 0) {
            s_pe[1] = predict(s_gm);
            cg_after_q(s_cg, s_norm);
        }
        if (!sk_stage(st, g, inv)) return -1;
        if (team_failed(ti)) return -1;
        if (s_cg.reason != 0) { reason = s_cg.reason; break; }
        const int pr = s_pe[0];
        SkEpiM em{ow, rh, pr != kNoPe ? b16 : nullptr, b16 + plane,
                  __int_as_float((127 + (pr != kNoPe ? pr : 0)) << 23), c.Vp,
                  s_cg.alpha, hop, c.V, c.Nt, 0.f, 0.f};
        if (!sk_reduce<false>(st, g, tcl, c.V, c.e_inv, em)) return -1;
        if (threadIdx.x == 0) s_pw[0] = b16 ? pr : kNoPe;
        sk_post(ti, c.gslots, ++st.gseq, em.acc, em.mx);   // r ready, |r|^2
        have_rr = true;
    }
    if (reason != kSegNonfinite) {
        HMC_SK_OWNED(o, oi, g, c) {
            const float2 d = ow.x[oi];
            double2 xv = x64[o];
            xv.x += (double)d.x;
            xv.y += (double)d.y;
            x64[o] = xv;
        }
    }
    return reason;
}

template <int KIND>
__device__ bool cg_mixed(const ChainView& c, Team& tm, TcState& st, f64::Smem& sm64,
                         const CUtensorMap* mhi, const CUtensorMap* mlo,
                         const PersistentArgs& pa, ClusterSync* ics, const double2* chi,
                         double2* x64, MixedResult& res, bool warm = false, double gm1 = 0.0) {
    // the heavy operator M_g of mass preconditioning (gm1 = g - 1 != 0) is
    // built into the split-K tiles' epilogues only
    if (gm1 != 0.0 && KIND != kKindSplitK) {
        set_status(tm.status, HMC_ERR_UNSUPPORTED);
        return false;
    }
    constexpr bool SMALL = KIND == kKindSmall;
    float2 *rf = c.r_f, *pf = c.p_f, *pn = c.p2_f, *qf = c.q_f, *xf = c.x_f;
    const int inner_size = min(max(pa.inner, 1), tm.size);
    const bool in_inner = tm.rank < inner_size;
    Team ti = tm;
    if constexpr (KIND != kKindSeries) {   // (whose inner team is the whole team)
    ti.size = inner_size;
    ti.slots = tm.slots + kTeamWords;
    ti.gen = tm.gen + 1;
    // inner team = cluster 0: its barriers stay inside the cluster
    ti.cs = (ics && pa.cluster > 1 && inner_size == pa.cluster) ? ics : nullptr;
    }
    // FP64 solution and |chi|^2 on all CTAs
    double v1[1] = {0.0};
    HMC_TEAM_ELEMS(e, c, tm) {
        const double2 ch = chi[e];
        if (!warm) x64[e] = make_double2(0.0, 0.0);
        v1[0] += ch.x * ch.x + ch.y * ch.y;
    }
    if (!team_sum<1>(tm, v1)) return false;
    const double chi2 = v1[0];
    res.iterations = 0;
    res.reliable_updates = 0;
    res.status = HMC_OK;
    res.true_res = 0.0;
    if (!(chi2 > 0.0)) {
        if (!finite_d(chi2)) res.status = HMC_ERR_NONFINITE;
        return true;
    }
    const double stop = pa.tol * pa.tol * chi2;
    // warm start (a later solve of a trajectory: same chi, the field moved by
    // one MD step): the FP64 true residual of the given x64 is the starting
    // residual of the FP32 iteration
    double rr_true = chi2;
    const double2* r0 = chi;
    if (warm) {
        if (!f64_residual<kForm<KIND>>(c, tm, sm64, chi, x64, rr_true, gm1)) return false;
        ++res.reliable_updates;
        if (!finite_d(rr_true)) {
            res.status = HMC_ERR_NONFINITE;
            return true;
        }
        if (rr_true <= stop) {
            res.true_res = sqrt(rr_true / chi2);
            return true;
        }
        r0 = c.r;
    }
    // FP32 iterates on the inner team (their owners).  A chain solved by one
    // CTA with E resident keeps them in shared memory: r, p, p', q, x and the
    // FP32 phase table, six vectors after the B ring.
    double rr = 0.0;
    const float2* cisf = c.cis_f;
    SmallCg sm;
    if constexpr (SMALL) {
      if (in_inner) {
        // small lattice: FP32 iterates of the cluster's slices in shared memory
        small_init_view(sm, st.base, tm.rank, inner_size, c.V, c.Nt);
        double v2[1] = {small_setup(sm, c, r0)};
        if (!team_sum<1>(ti, v2)) return false;
        rr = v2[0];
      }
    } else if constexpr (KIND == kKindSeries) {
        double v2[1] = {0.0};
        HMC_TEAM_ELEMS(e, c, ti) {
            const double2 ch = r0[e];
            const float2 rv = make_float2((float)ch.x, (float)ch.y);
            rf[e] = rv;
            pf[e] = make_float2(0.f, 0.f);
            c.g_f[e] = make_float2(0.f, 0.f);
            v2[0] += (double)rv.x * rv.x + (double)rv.y * rv.y;
        }
        if (!team_sum<1>(ti, v2)) return false;
        rr = v2[0];
    } else if constexpr (KIND == kKindSplitK) {
      if (in_inner) {
        // split-K: this CTA's part of E' stays resident for the whole launch
        if (!st.sk_loaded) {
            const SkGeom g = sk_geom(tm.rank, pa.sk_C, pa.ns_tile, c.V, c.Nt, c.Vr, c.Vp);
            if (!sk_load_E(st, g, mhi, mlo)) return false;
            st.sk_loaded = 1;
        }
        double v2[1] = {0.0};
        HMC_TEAM_ELEMS(e, c, ti) {
            const double2 ch = r0[e];
            const float2 rv = make_float2((float)ch.x, (float)ch.y);
            rf[e] = rv;
            pf[e] = make_float2(0.f, 0.f);
            xf[e] = make_float2(0.f, 0.f);
            c.g_f[e] = make_float2(0.f, 0.f);
            v2[0] += (double)rv.x * rv.x + (double)rv.y * rv.y;
        }
        if (!team_sum<1>(ti, v2)) return false;
        rr = v2[0];
      }
    } else if (in_inner) {
        if (pa.mode == kResident) {
            if (!tc_load_resident(st, mhi, mlo, (tm.rank % (c.Vr / TM)) * TM, c.Vp / KCH))
                return false;
        } else {
            tc_set_layout(st, kStreaming, 0);
        }
        if (pa.vec_resident) {
            float2* sv = reinterpret_cast<float2*>(st.free_area());
            rf = sv;
            pf = sv + c.N;
            pn = sv + 2 * c.N;
            qf = sv + 3 * c.N;
            xf = sv + 4 * c.N;
            float2* cs = sv + 5 * c.N;
            for (int e = threadIdx.x; e < c.N; e += blockDim.x) cs[e] = c.cis_f[e];
            cisf = cs;
        }
        double v2[1] = {0.0};
        HMC_TEAM_ELEMS(e, c, ti) {
            const double2 ch = r0[e];
            const float2 rv = make_float2((float)ch.x, (float)ch.y);
            rf[e] = rv;
            pf[e] = make_float2(0.f, 0.f);
            xf[e] = make_float2(0.f, 0.f);
            v2[0] += (double)rv.x * rv.x + (double)rv.y * rv.y;
        }
        if (!team_sum<1>(ti, v2)) return false;
        rr = v2[0];
    }
    __shared__ CgScalars s_cg;
    bool refresh = false;
    if (threadIdx.x == 0) {
        s_cg.rr = (float)rr;
        s_cg.pp = (float)rr;
        s_cg.rmax = (float)rr;
        s_cg.beta = 0.f;
        s_cg.stop = (float)stop;
        s_cg.ru2 = (float)(pa.ru_delta * pa.ru_delta);
        s_cg.it = 0;
        s_cg.it0 = 0;
        s_cg.every = pa.ru_every > 0 ? pa.ru_every : 1000;
        vector_scale(rr, s_cg.sc, s_cg.inv);
    }
    __syncthreads();
    bool conv = false;
    bool sk_first = true;   // split-K: the first segment starts p and G at zero
    // progress of the FP64 true residual between reliable updates: two
    // updates in a row that did not halve it mean the FP32 recursion has
    // stalled (near a singular M); the rest of the solve then runs in FP64
    double rr_last = rr_true;
    int stalls = 0;
    bool fallback = false;
    res.fp64_iterations = 0;
    volatile double* seg = c.scalars + 12;   // [0] end reason, [1] iterations
    for (;;) {
        if constexpr (KIND == kKindSeries) {
            const int reason =
                ser::run_segment(c, ti, *static_cast<const ser::Work*>(st.ser), s_cg, refresh,
                                 pa.max_iter, x64);
            if (reason < 0) return false;
            refresh = false;
            if (tm.rank == 0 && threadIdx.x == 0) {
                seg[0] = reason;
                seg[1] = s_cg.it;
            }
        } else if constexpr (SMALL) {
          if (in_inner) {
            // small lattice: each half iteration is epilogue -> partial norm
            // out -> contraction -> boundary column out -> wait (byte-counted)
            __shared__ SmallSum s_ss;
            int reason = 0;
            if (refresh) {
                small_refresh_r(sm, c.r);
                refresh = false;
            }
            __syncthreads();
            small_load_ud(sm);
            __syncthreads();
            small_matvec_any(sm, sm.v(sm.l.ud));
            __syncthreads();
            small_send_boundary_plain(sm);
            if (!team_barrier(ti)) return false;   // boundary columns published
            unsigned kk = ti.cs ? ti.cs->count_tx : 0u;   // exchange phase
            const uint32_t xbytes = (uint32_t)(4 * ti.size + 8 * c.V);
            if (s_cg.it >= pa.max_iter) reason = kSegMaxIter;
            while (reason == 0) {
                float qq, rr_new;
                // q = M^dag p', p' = r + beta p; then E e^{i phi} q
                small_sum_begin(ti, s_ss, kk, small_dag_epilogue(sm, s_cg.beta));
                small_matvec_any(sm, sm.v(sm.l.um));
                __syncthreads();
                small_send_boundary(sm, ti.cs, kk, sm.S - 1, sm.l.bm, sm.next);
                if (!small_sum_end(ti, s_ss, kk, xbytes, qq)) return false;
                ++kk;
                if (threadIdx.x == 0) cg_after_q(s_cg, qq);
                __syncthreads();
                if (s_cg.reason != 0) { reason = s_cg.reason; break; }
                // x += alpha p', r -= alpha M q; then E r
                small_sum_begin(ti, s_ss, kk, small_m_epilogue(sm, s_cg.alpha));
                small_matvec_any(sm, sm.v(sm.l.ud));
                __syncthreads();
                small_send_boundary(sm, ti.cs, kk, 0, sm.l.bd, sm.prev);
                if (!small_sum_end(ti, s_ss, kk, xbytes, rr_new)) return false;
                ++kk;
                if (threadIdx.x == 0) {
                    cg_after_r(s_cg, rr_new);
                    if (s_cg.reason == 0 && s_cg.it >= pa.max_iter) s_cg.reason = kSegMaxIter;
                }
                __syncthreads();
                if (s_cg.reason != 0) { reason = s_cg.reason; break; }
            }
            if (threadIdx.x == 0 && ti.cs) ti.cs->count_tx = kk;
            if (reason != kSegNonfinite) small_fold_x(sm, x64);
            if (tm.rank == 0 && threadIdx.x == 0) {
                seg[0] = reason;
                seg[1] = s_cg.it;
            }
          }
        } else if constexpr (KIND == kKindSplitK) {
          if (in_inner) {
            const int reason = sk_segment(c, ti, st, pa, ics, s_cg, refresh, sk_first, cisf, x64,
                                          (float)(1.0 + gm1));
            if (reason < 0) return false;
            refresh = false;
            sk_first = false;
            if (tm.rank == 0 && threadIdx.x == 0) {
                seg[0] = reason;
                seg[1] = s_cg.it;
            }
          }
        } else if (in_inner) {
            int reason = kSegMaxIter;
            while (s_cg.it < pa.max_iter) {
                // p_new = r + beta p; q = M^dag p_new
                SrcDirection dir{rf, c.r, pf, s_cg.beta, refresh, c.V};
                EpiDirection ed{dir, pn, rf, qf, cisf, c.Nt, 0.f};
                bool aok;
                if constexpr (KIND == kKindSlice)
                    aok = apply_team_w<true>(c, ti, st, pa.wide_W, mhi, mlo, pa.ns_tile, dir,
                                             s_cg.sc, s_cg.inv, ed);
                else
                    aok = apply_team<true>(c, ti, st, mhi, mlo, pa.ns_tile, dir, s_cg.sc,
                                           s_cg.inv, ed, pa.res_b != 0);
                if (!aok) return false;
                float qq;
                if (!team_sum_f(ti, ed.acc, qq)) return false;
                float2* t = pf;
                pf = pn;
                pn = t;
                refresh = false;
                if (threadIdx.x == 0) cg_after_q(s_cg, qq);
                __syncthreads();
                if (s_cg.reason != 0) { reason = s_cg.reason; break; }
                // Ap = M q; x += alpha p; r -= alpha Ap
                SrcPhase srcq{qf, cisf, c.V};
                EpiCgUpdate eu{qf, pf, xf, rf, s_cg.alpha, c.V, 0.f};
                if constexpr (KIND == kKindSlice)
                    aok = apply_team_w<false>(c, ti, st, pa.wide_W, mhi, mlo, pa.ns_tile, srcq,
                                              s_cg.sc, s_cg.inv, eu);
                else
                    aok = apply_team<false>(c, ti, st, mhi, mlo, pa.ns_tile, srcq, s_cg.sc,
                                            s_cg.inv, eu, pa.res_b != 0);
                if (!aok) return false;
                float rr_new;
                if (!team_sum_f(ti, eu.acc, rr_new)) return false;
                if (threadIdx.x == 0) cg_after_r(s_cg, rr_new);
                __syncthreads();
                if (s_cg.reason != 0) { reason = s_cg.reason; break; }
            }
            // fold the FP32 increment into x64 (the inner team owns x_f)
            if (reason != kSegNonfinite) {
                HMC_TEAM_ELEMS(e, c, ti) {
                    const float2 d = xf[e];
                    double2 xv = x64[e];
                    xv.x += (double)d.x;
                    xv.y += (double)d.y;
                    x64[e] = xv;
                    xf[e] = make_float2(0.f, 0.f);
                }
            }
            if (tm.rank == 0 && threadIdx.x == 0) {
                seg[0] = reason;
                seg[1] = s_cg.it;
            }
        }
        if (!team_barrier(tm)) return false;
        const int reason = (int)seg[0];
        const int it = (int)seg[1];
        if (reason == kSegNonfinite) { res.status = HMC_ERR_NONFINITE; break; }
        // FP64 true residual on all CTAs
        if (!f64_residual<kForm<KIND>>(c, tm, sm64, chi, x64, rr_true, gm1)) return false;
        ++res.reliable_updates;
        if (!finite_d(rr_true)) { res.status = HMC_ERR_NONFINITE; break; }
        if (rr_true <= stop) { conv = true; break; }
        if (reason == kSegMaxIter) break;
        stalls = rr_true > 0.25 * rr_last ? stalls + 1 : 0;
        rr_last = rr_true;
        if (stalls >= 2) { fallback = true; break; }
        // continue from the true residual; keep the direction
        if (threadIdx.x == 0) {
            const double b = rr_true / (double)s_cg.rr;
            const double pp = rr_true + b * b * (double)s_cg.pp;
            s_cg.beta = (float)b;
            s_cg.rr = (float)rr_true;
            s_cg.rmax = (float)rr_true;
            s_cg.pp = (float)pp;
            s_cg.it = it;
            s_cg.it0 = it;
            vector_scale(pp, s_cg.sc, s_cg.inv);
        }
        __syncthreads();
        refresh = true;
    }
    res.iterations = (int)seg[1];
    if (fallback) {
        // FP64 CG on all CTAs from the current solution; its final true
        // residual leaves M^dag x in q, as the reliable update does
        f64::CgResult r64;
        if (!f64::cg_solve<kForm<KIND>>(c, tm, chi, x64, pa.tol,
                                        max(1, pa.max_iter - res.iterations), r64, sm64, true,
                                        gm1))
            return false;
        res.fp64_iterations = r64.iterations;
        res.true_res = r64.true_res;
        res.status = r64.status;
        return true;
    }
    if (!conv && res.status == HMC_OK) res.status = HMC_ERR_CG_NOT_CONVERGED;
    res.true_res = sqrt(rr_true / chi2);
    if (!finite_d(res.true_res)) res.status = HMC_ERR_NONFINITE;
    return true;
}

// Cluster launch: set up the cluster team state and check that the inner
// team's ranks are the cluster ranks of cluster 0.  A launch that is not made of
// such clusters ends at its first team sync, which is one of the whole team
// through global memory: cluster_ok after it, on every thread (the sync orders
// the status of a member before its post).
__device__ inline void cluster_begin(const PersistentArgs& pa, ClusterSync* cs, int* status) {
    if (pa.cluster <= 1) return;
    if (threadIdx.x == 0 && !cluster_matches(pa.cluster)) set_status(status, HMC_ERR_UNSUPPORTED);
    cluster_sync_init(cs, pa.cluster);
}
__device__ inline bool cluster_ok(const PersistentArgs& pa, const Team& tm) {
    return pa.cluster <= 1 || !__syncthreads_or(threadIdx.x == 0 && team_failed(tm));
}

__device__ __forceinline__ Team make_team(const ChainView& c) {
    __shared__ unsigned s_gen[2];   // syncs of the whole team and of the inner one
    if (threadIdx.x == 0) s_gen[0] = s_gen[1] = 0;
    Team tm;
    tm.rank = blockIdx.x;
    tm.size = gridDim.x + c.team_pad;
    tm.status = c.status;
    tm.slots = c.slots;
    tm.gen = s_gen;
    tm.cs = nullptr;
    return tm;
}

__device__ __forceinline__ void set_phases(const ChainView& c, const Team& tm,
                                           const double* phi) {
    HMC_TEAM_ELEMS(e, c, tm) {
        double s, co;
        sincos(phi[e], &s, &co);
        c.cis[e] = make_double2(co, s);
        c.cis_f[e] = make_float2((float)co, (float)s);
    }
}

// One HMC trajectory with the mixed solver (same steps as the FP64 one),
// run by team `tm`; results in c.scalars.  Returns false if the team failed.
template <int KIND>
__device__ bool run_trajectory(const ChainView& c, Team& tm, TcState& st, f64::Smem& sm64,
                               const CUtensorMap* mhi, const CUtensorMap* mlo,
                               const PersistentArgs& pa, ClusterSync* ics, const TrajArgs& a) {
    double* phi = a.phi;
    const double inv_dU = 1.0 / (c.delta * c.U);
    const double rsqrt2 = 0.70710678118654752440;
    double h0[3] = {0.0, 0.0, 0.0};
    HMC_TEAM_ELEMS(e, c, tm) {
        const double2 zp = normal_pair(philox_draw(a.seed, kStreamMomentum, a.traj, a.chain, e));
        const double2 zr = normal_pair(philox_draw(a.seed, kStreamNoise, a.traj, a.chain, e));
        const double ph = phi[e];
        c.pi[e] = zp.x;
        const double2 rho = make_double2(zr.x * rsqrt2, zr.y * rsqrt2);
        c.rho[e] = rho;
        c.phi_old[e] = ph;
        double s, co;
        sincos(ph, &s, &co);
        c.cis[e] = make_double2(co, s);
        c.cis_f[e] = make_float2((float)co, (float)s);
        h0[0] += ph * ph;
        h0[1] += rho.x * rho.x + rho.y * rho.y;
        h0[2] += zp.x * zp.x;
    }
    bool ok = team_sum<3>(tm, h0) && cluster_ok(pa, tm);
    const double H0 = 0.5 * h0[0] * inv_dU + h0[1] + 0.5 * h0[2];
    f64::EpiArgs ea = {};
    if (ok) {
        f64::apply_team<kForm<KIND>, false, f64::EPI_STORE>(c, tm, c.rho, c.chi, ea, sm64);
        ok = team_barrier(tm);
    }
    int iters = 0, solves = 0, rus = 0, fp64_iters = 0, status = HMC_OK;
    double max_res = 0.0;
    ea.phi = phi;
    ea.pi = c.pi;
    ea.inv_dU = inv_dU;
    const double ed = a.eps * c.delta;
    const double edrift = md_drift(a) * ed;
    const int n_stages = md_stages(a);
    // initial guesses of the solves (the solves sit at equally spaced fields):
    // the first from zero, the second from the first solution, the third
    // from the linear extrapolation 2 x_{k-1} - x_{k-2}, later ones from the
    // quadratic one 3 x_{k-1} - 3 x_{k-2} + x_{k-3}; rho, free once chi and
    // H0 are formed, keeps x_{k-2}, xh keeps x_{k-3}
    double2* xold = c.rho;
    for (int step = 0; ok && step <= n_stages; ++step) {
        if (step > 0) {
            HMC_TEAM_ELEMS(e, c, tm) {
                const double ph = fma(edrift, c.pi[e], phi[e]);
                phi[e] = ph;
                double s, co;
                sincos(ph, &s, &co);
                c.cis[e] = make_double2(co, s);
                c.cis_f[e] = make_float2((float)co, (float)s);
                const double2 x1 = c.x[e];
                if (step > 2) {
                    const double2 x2 = xold[e], x3 = c.xh[e];
                    c.x[e] = make_double2(3.0 * (x1.x - x2.x) + x3.x, 3.0 * (x1.y - x2.y) + x3.y);
                    c.xh[e] = x2;
                } else if (step > 1) {
                    const double2 x2 = xold[e];
                    c.x[e] = make_double2(2.0 * x1.x - x2.x, 2.0 * x1.y - x2.y);
                    c.xh[e] = x2;
                }
                xold[e] = x1;
            }
            if (!(ok = team_barrier(tm))) break;
        }
        MixedResult res{};
        if (!(ok = cg_mixed<KIND>(c, tm, st, sm64, mhi, mlo, pa, ics, c.chi, c.x, res, step > 0)))
            break;
        iters += res.iterations;
        rus += res.reliable_updates;
        fp64_iters += res.fp64_iterations;
        ++solves;
        max_res = fmax(max_res, res.true_res);
        if (res.status != HMC_OK && status == HMC_OK) status = res.status;
        ea.kick = md_kick(a, step) * ed;
        if (res.status == HMC_OK) {
            // the solve ended on an FP64 true residual of its final x, which
            // left q = M^dag x (same FP64 tile): the force needs no
            // application of its own
            HMC_TEAM_ELEMS(e, c, tm) {
                const double2 xv = c.x[e], y = c.q[e];
                const double f = phi[e] * inv_dU + 2.0 * (xv.y * y.x - xv.x * y.y);
                c.pi[e] -= ea.kick * f;
            }
        } else {
            f64::apply_team<kForm<KIND>, true, f64::EPI_FORCE>(c, tm, c.x, nullptr, ea, sm64);
        }
        ok = team_barrier(tm);
    }
    double h1[3] = {0.0, 0.0, 0.0};
    if (ok) {
        HMC_TEAM_ELEMS(e, c, tm) {
            const double ph = phi[e], pv = c.pi[e];
            const double2 ch = c.chi[e], xv = c.x[e];
            h1[0] += ph * ph;
            h1[1] += ch.x * xv.x + ch.y * xv.y;
            h1[2] += pv * pv;
        }
        ok = team_sum<3>(tm, h1);
    }
    if (ok) {
        const double H1 = 0.5 * h1[0] * inv_dU + h1[1] + 0.5 * h1[2];
        const double dH = H1 - H0;
        const double u =
            uniform_pair(philox_draw(a.seed, kStreamMetropolis, a.traj, a.chain, 0)).x;
        const bool accept = u < exp(-dH);
        if (!accept) {
            HMC_TEAM_ELEMS(e, c, tm) phi[e] = c.phi_old[e];
        }
        if (tm.rank == 0 && threadIdx.x == 0) {
            c.scalars[kTrajDH] = dH;
            c.scalars[kTrajH0] = H0;
            c.scalars[kTrajH1] = H1;
            c.scalars[kTrajU] = u;
            c.scalars[kTrajAccept] = accept ? 1.0 : 0.0;
            c.scalars[kTrajIters] = iters;
            c.scalars[kTrajSolves] = solves;
            c.scalars[kTrajRU] = rus;
            c.scalars[kTrajMaxRes] = max_res;
            c.scalars[kTrajStatus] = status;
            c.scalars[kTrajFp64Iters] = fp64_iters;
        }
    }
    return ok;
}

// ---------------------------------------------------------------- batched
// Many independent chains of different sizes in one persistent launch,
// chains ordered by decreasing estimated cost.  With csize == 1 every CTA
// takes the next chain from an atomic work queue and runs its whole
// trajectory as a one-CTA team.  With csize > 1 the launch is made of
// thread-block clusters of csize CTAs and the queue starts with the chains
// marked as cluster teams (the most expensive ones): while those last, rank
// 0 of a cluster takes the next chain and hands its index to every member,
// and the cluster runs it as one team (barriers and sums through
// distributed shared memory, FP64 steps over all csize CTAs).  At the first
// one-CTA chain the cluster's members go their own way: rank 0 runs that
// chain and every member takes further chains alone.  The TMEM allocation
// and the operand ring persist across chains.
struct BatchItem {
    ChainView v;
    int team;                  // > 1: run by a cluster of this many CTAs (the launch's size)
    const CUtensorMap* maps;   // [0] E_hi, [1] E_lo, [2] / [3] scaled split for the
                               // slice-major tile (global memory, 64-byte aligned)
    PersistentArgs pa;
    TrajArgs a;                // n_md, eps, tol, max_iter, chain; seed/traj/phi per call
    long long offset;          // of this chain's field in the packed array
};

struct BatchCallArgs {
    uint64_t seed;
    uint64_t traj;
    double* phi;               // packed fields of all chains
};


template <class Run>
__device__ inline void batch_run(const BatchItem& it, int ci, const BatchCallArgs* call,
                                 double* outs, Team& tm, ClusterSync* ics, bool write_out,
                                 Run&& run, bool& ok) {
    TrajArgs a = it.a;
    a.seed = call->seed;
    a.traj = call->traj;
    a.phi = call->phi + it.offset;
    ok = run(it, tm, ics, a);
    __syncthreads();
    if (write_out && threadIdx.x == 0) {
        for (int k = 0; k < kNumScalars; ++k)
            outs[(size_t)ci * kNumScalars + k] = it.v.scalars[k];
        outs[(size_t)ci * kNumScalars + kTrajStatus] =
            ok ? it.v.scalars[kTrajStatus] : (double)(*((volatile int*)it.v.status));
    }
}

// Reset a chain's status and scalars and make its tensor maps (global
// memory) visible to the TMA proxy of this CTA.  Thread 0.
__device__ inline void batch_chain_begin(const BatchItem& it, bool reset) {
    if (reset) {
        *it.v.status = 0;
        for (int k = 0; k < kNumScalars; ++k) it.v.scalars[k] = 0.0;
    }
    for (int m = 0; it.maps && m < 4; ++m)
        asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(it.maps + m)
                     : "memory");
}

// The work queue of a batch launch; run(item, team, cluster state, args) runs one
// trajectory of one chain.
template <class Run>
__device__ inline void batch_loop(const BatchItem* __restrict__ items,
                                  const int* __restrict__ order, int n, int* queue,
                                  const BatchCallArgs* call, double* outs, int csize,
                                  ClusterSync* cs, Run&& run) {
    __shared__ int s_idx;
    if (csize > 1 && !cluster_matches(csize)) {
        // launched without its clusters (every CTA alike): no chain runs
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
            outs[(size_t)i * kNumScalars + kTrajSolves] = 0.0;
            outs[(size_t)i * kNumScalars + kTrajStatus] = (double)HMC_ERR_UNSUPPORTED;
        }
        return;
    }
    const int crank = csize > 1 ? (int)cluster_ctarank() : 0;
    bool solo = csize == 1;
    bool ok = true;
    // cluster phase: one team chain per cluster at a time
    while (!solo) {
        if (crank == 0 && threadIdx.x == 0) {
            const int v = atomicAdd(queue, 1);
            if (v < n && items[order[v]].team > 1) batch_chain_begin(items[order[v]], true);
            const uint32_t la = cta_smem_u32(&s_idx);
            for (int r = 0; r < csize; ++r) {
                uint32_t ra;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(la), "r"(r));
                asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(ra), "r"(v) : "memory");
            }
        }
        cluster_barrier_all();          // the index (and the chain's reset) published
        const int idx = s_idx;
        cluster_barrier_all();          // read by every member before the next write
        if (idx >= n) break;
        const int ci = order[idx];
        const BatchItem& it = items[ci];
        if (it.team <= 1) {
            // first one-CTA chain: rank 0 runs it, then all members go alone
            solo = true;
            if (crank == 0) {
                if (threadIdx.x == 0) batch_chain_begin(it, true);
                __syncthreads();
                Team tm{};
                tm.rank = 0;
                tm.size = 1;
                tm.status = it.v.status;   // one CTA or one cluster: no slots
                tm.cs = nullptr;
                batch_run(it, ci, call, outs, tm, nullptr, true, run, ok);
            }
            break;
        }
        if (threadIdx.x == 0 && crank != 0) batch_chain_begin(it, false);
        __syncthreads();
        Team tm{};
        tm.rank = crank;
        tm.size = csize;
        tm.status = it.v.status;   // one CTA or one cluster: no slots
        tm.cs = cs;
        batch_run(it, ci, call, outs, tm, cs, crank == 0, run, ok);
        // the team's outcome, the same on every member: a failed member has
        // set the chain's status before it left its waits
        cluster_barrier_all();
        ok = *((volatile int*)it.v.status) == 0;
        if (!ok) break;
    }
    // one-CTA phase
    while (ok) {
        if (threadIdx.x == 0) s_idx = atomicAdd(queue, 1);
        __syncthreads();
        const int idx = s_idx;
        __syncthreads();
        if (idx >= n) break;
        const int ci = order[idx];
        const BatchItem& it = items[ci];
        if (threadIdx.x == 0) batch_chain_begin(it, true);
        __syncthreads();
        Team tm{};
        tm.rank = 0;
        tm.size = 1;
        tm.status = it.v.status;   // one CTA or one cluster: no slots
        tm.cs = nullptr;
        batch_run(it, ci, call, outs, tm, nullptr, true, run, ok);
        // a failed bounded wait leaves the operand ring in an unknown phase:
        // this CTA takes no further chains (they stay unprocessed, status set)
    }
}

}  // namespace tc
}  // namespace hmc
