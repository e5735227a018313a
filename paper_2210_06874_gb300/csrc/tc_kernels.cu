// tc_kernels.cu -- the mixed-precision path: tensor-core applications of
// M / M^dag (FP16 split, FP32 accumulate), FP32 conjugate gradient with FP64
// reliable updates, and the HMC trajectory built on it.  FP64 stays for the
// true residual, chi = M rho, the force, the Hamiltonian sums and Metropolis.
#include <cuda_fp16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <queue>
#include <vector>

#include "mixed_path.cuh"
#include "tc_path.h"

namespace hmc {

struct TcCtx {
    CUtensorMap map_hi, map_lo;
    int ns_apply;        // slices per tile of standalone applications
    // pre-split B operand of standalone applications: FP16 hi / lo rows
    // [2 Nt + 64][Vp] (row 2t: re, 2t+1: im of the source of target slice t;
    // the last 64 rows stay zero for tiles that run past Nt) and the
    // per-slice inverse scales
    CUtensorMap map_bhi, map_blo;
    __half* bhi;
    __half* blo;
    float* inv_col;
    int b_rows;
    // slice-major tiles (operand_mode 4): maps of the scaled split of E (box
    // rows = W / nmma), sites per tile of the solver and of standalone
    // applications, slices per standalone tile, and the maps of the
    // pre-split U (plain remainder) over bhi / blo with 128-row boxes
    CUtensorMap map_whi, map_wlo, map_uhi, map_ulo;
    int w_cg, w_apply, ns_wapply, csplit_apply;
    // split-K tiles (operand_mode 5): the scaled split of E in 128-row boxes;
    // standalone applications: the shape (C CTAs per cluster, ns slices per
    // n-group, 0 if it does not fit) and the maps of the pre-split source
    // (plain remainder) over bhi / blo with boxes of sk_nn(ns) rows
    CUtensorMap map_shi, map_slo;
    int sk_C_apply, sk_ns_apply;
    float* inv_sk;       // per (target slice, K range) inverse scales [Nt][C]
    CUtensorMap map_skb_hi, map_skb_lo;
};

namespace tc {
// TMA box rows of the pre-split U for tiles of ns slices: 2 ns rounded up
// to 16 (the swizzle atom is 8 rows; whole 1024-byte atoms), at most 128.
__host__ __device__ inline int wide_u_rows(int ns) {
    const int r = ((2 * ns + 15) / 16) * 16;
    return r > 128 ? 128 : r;
}
}  // namespace tc

namespace tc {

// ---------------------------------------------------------------- standalone
// B operand of one standalone application, split before the tiles run: for
// target slice t (one block) the source u = in_{t+1} (M^dag) or
// e^{i phi_{t-1}} in_{t-1} (M), scaled by 2^e with max |Re u|, |Im u| in
// [2^14, 2^15), written as FP16 hi = fp16(s u) and lo = fp16((s u - hi) 2^11)
// (PLAIN, for the slice-major tile: lo = fp16(s u - hi)) in rows 2t (re) and
// 2t+1 (im), zero from V to Vp; inv[t] = 2^-e.  Also writes the FP32 phase
// table of slice t (the M^dag epilogue reads it).
// Dynamic shared memory: V float2 (the source slice).  1024 threads per
// block: the work per slice is a few sites per thread, so the block's two
// passes are each about one round trip to memory.
constexpr int kSplitThreads = 1024;
template <bool DAG, bool PLAIN>
__global__ void __launch_bounds__(kSplitThreads)
    k_split(const double* __restrict__ phi, const float2* __restrict__ in,
            float2* __restrict__ cis_f, __half* __restrict__ bhi, __half* __restrict__ blo,
            float* __restrict__ inv, int V, int Vp, int Nt) {
    extern __shared__ float2 u_s[];
    __shared__ float s_max[kSplitThreads / 32];
    __shared__ int s_e;
    // the application kernel may start its set-up now (programmatic
    // dependent launch); it waits for this grid before reading B
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int t = blockIdx.x;
    const int ts = DAG ? (t + 1 == Nt ? 0 : t + 1) : (t == 0 ? Nt - 1 : t - 1);
    float mx = 0.f;
    for (int k = threadIdx.x; k < V; k += blockDim.x) {
        float sn, cs;
        sincosf((float)phi[(size_t)t * V + k], &sn, &cs);
        cis_f[(size_t)t * V + k] = make_float2(cs, sn);
        float2 u = in[(size_t)ts * V + k];
        if (!DAG) {
            sincosf((float)phi[(size_t)ts * V + k], &sn, &cs);
            u = make_float2(cs * u.x - sn * u.y, cs * u.y + sn * u.x);
        }
        u_s[k] = u;
        mx = fmaxf(mx, fmaxf(fabsf(u.x), fabsf(u.y)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_down_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        float m = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, s_max[w]);
        const int bits = __float_as_int(m), ex = (bits >> 23) & 0xff;
        int e = 0;
        if (bits > 0 && ex != 0xff) e = max(-120, min(120, 14 - (ex - 127)));
        s_e = e;
        inv[t] = __int_as_float((127 - e) << 23);
    }
    __syncthreads();
    const float sc = __int_as_float((127 + s_e) << 23);
    __half* hr = bhi + (size_t)(2 * t) * Vp;
    __half* lr = blo + (size_t)(2 * t) * Vp;
    for (int k = threadIdx.x; k < Vp; k += blockDim.x) {
        __half h0 = __float2half_rn(0.f), h1 = h0, l0 = h0, l1 = h0;
        if (k < V) {
            const float2 u = u_s[k];
            const float x = u.x * sc, y = u.y * sc;
            h0 = __float2half_rn(x);
            h1 = __float2half_rn(y);
            const float ls = PLAIN ? 1.f : kLoScale;
            l0 = __float2half_rn((x - __half2float(h0)) * ls);
            l1 = __float2half_rn((y - __half2float(h1)) * ls);
        }
        hr[k] = h0;
        hr[Vp + k] = h1;
        lr[k] = l0;
        lr[Vp + k] = l1;
    }
}

// Standalone application of M or M^dag: the tiles load E and the pre-split
// B by TMA and contract them; the epilogue forms the result.
template <bool DAG>
__global__ void __launch_bounds__(NTHR, 1)
    k_apply(const __grid_constant__ CUtensorMap mhi, const __grid_constant__ CUtensorMap mlo,
            const __grid_constant__ CUtensorMap bhi, const __grid_constant__ CUtensorMap blo,
            const __grid_constant__ ChainView c, int ns_tile, const float2* in, float2* out, const float* inv) {
    extern __shared__ __align__(1024) uint8_t dyn[];
    TcState st;
    tc_setup(st, dyn, c.status);
    EpiStore<DAG> epi{in, out, c.cis_f, c.V, c.Nt, 0.f};
    const int nti = c.Vr / TM;
    int i0, t0, ns;
    tile_coords(blockIdx.x, nti, ns_tile, c.Nt, i0, t0, ns);
    SrcSplit src{&bhi, &blo, inv, ((2 * ns_tile + 15) / 16) * 16};
    // launched as a programmatic dependent of the split: the set-up above
    // overlaps it; its B, scales and phase table are visible after this
    asm volatile("griddepcontrol.wait;" ::: "memory");
    tc_tile<DAG>(st, &mhi, &mlo, c.V, c.Nt, c.Vp, i0, t0, ns, src, 1.f, 1.f, epi);
    tc_teardown(st);
}

// Standalone application on slice-major tiles: one output tile (W sites x
// ns_tile slices) per thread-block cluster of csplit CTAs, which split its K
// chunks; E' and the pre-split U arrive by TMA.  Each CTA contracts its
// chunks into its own accumulator and stages it in shared memory; after a
// cluster barrier each takes a share of the tile's outputs, sums the csplit
// partials through distributed shared memory in rank order and runs the
// epilogue; a second cluster barrier keeps every CTA's shared memory alive
// until the others have read it.  csplit = 1 is a plain launch.
template <bool DAG>
__global__ void __launch_bounds__(NTHR, 1)
    k_apply_w(const __grid_constant__ CUtensorMap mhi, const __grid_constant__ CUtensorMap mlo,
              const __grid_constant__ CUtensorMap uhi, const __grid_constant__ CUtensorMap ulo,
              const __grid_constant__ ChainView c, int W, int ns_tile, int csplit, const float2* in, float2* out,
              const float* inv) {
    extern __shared__ __align__(1024) uint8_t dyn[];
    TcState st;
    tc_setup(st, dyn, c.status);
    EpiStore<DAG> epi{in, out, c.cis_f, c.V, c.Nt, 0.f};
    const WideGeom g = wide_geom(W);
    const int nsi = (c.V + W - 1) / W, nk = c.Vp / KCH;
    const int tile = blockIdx.x / csplit, rank = blockIdx.x % csplit;
    const int i0 = (tile % nsi) * W, t0 = (tile / nsi) * ns_tile;
    const int ns = min(ns_tile, c.Nt - t0);
    const int kc0 = nk * rank / csplit, kc1 = nk * (rank + 1) / csplit;
    SrcSplitW src{&uhi, &ulo, inv, wide_u_rows(ns_tile)};
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the split (see k_apply)
    tc_wstage<DAG>(st, g, &mhi, &mlo, c.V, c.Nt, i0, t0, ns, kc0, kc1, src, 1.f);
    cluster_barrier_all();   // every member's partial staged (release / acquire)
    if (*((volatile int*)c.status) == 0)
        tc_wepilogue(st, W, c.V, i0, t0, ns, src, 1.f, c.e_inv, epi, rank, csplit);
    cluster_barrier_all();   // the partials stay until every member has read them
    tc_teardown(st);
}

// B operand of a standalone split-K application, one block per (target
// slice t, K range r of the clusters' C CTAs): the source u of slice t
// (in_{t+1} for M^dag, e^{i phi_{t-1}} in_{t-1} for M) over the range's
// sites, scaled by 2^e with the largest |Re u|, |Im u| of the range in
// [2^14, 2^15), split into FP16 hi and plain remainder lo in rows 2t (re)
// and 2t + 1 (im); inv[t * C + r] = 2^-e (the consumer unscales its
// partial per column with it: the scale is uniform over its K range).  Also
// the FP32 phase table of slice t over the range.  One element per thread;
// one pass over memory.
constexpr int kSplitSkThreads = 256;   // >= the largest K range (4 chunks of 64)
template <bool DAG>
__global__ void __launch_bounds__(kSplitSkThreads)
    k_split_sk(const double* __restrict__ phi, const float2* __restrict__ in,
               float2* __restrict__ cis_f, __half* __restrict__ bhi, __half* __restrict__ blo,
               float* __restrict__ inv, int V, int Vp, int Nt, int C) {
    __shared__ float s_max[kSplitSkThreads / 32];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int t = blockIdx.x, r = blockIdx.y;
    const int KS = (V + 15) / 16;
    const int k0 = 16 * (KS * r / C), k1 = min(16 * (KS * (r + 1) / C), V);
    const int ts = DAG ? (t + 1 == Nt ? 0 : t + 1) : (t == 0 ? Nt - 1 : t - 1);
    const int k = k0 + (int)threadIdx.x;
    float2 u = make_float2(0.f, 0.f);
    if (k < k1) {
        float sn, cs;
        sincosf((float)phi[(size_t)t * V + k], &sn, &cs);
        cis_f[(size_t)t * V + k] = make_float2(cs, sn);
        u = in[(size_t)ts * V + k];
        if (!DAG) {
            sincosf((float)phi[(size_t)ts * V + k], &sn, &cs);
            u = make_float2(cs * u.x - sn * u.y, cs * u.y + sn * u.x);
        }
    }
    float mx = fmaxf(fabsf(u.x), fabsf(u.y));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = mx;
    __syncthreads();
    float m = 0.f;
    for (int w = 0; w < kSplitSkThreads / 32; ++w) m = fmaxf(m, s_max[w]);
    const int bits = __float_as_int(m), ex = (bits >> 23) & 0xff;
    int e = 0;
    if (bits > 0 && ex != 0xff) e = max(-120, min(120, 14 - (ex - 127)));
    if (threadIdx.x == 0) inv[t * C + r] = __int_as_float((127 - e) << 23);
    if (k < k1) {
        const float sc = __int_as_float((127 + e) << 23);
        const float x = u.x * sc, y = u.y * sc;
        const __half h0 = __float2half_rn(x), h1 = __float2half_rn(y);
        bhi[(size_t)(2 * t) * Vp + k] = h0;
        bhi[(size_t)(2 * t + 1) * Vp + k] = h1;
        blo[(size_t)(2 * t) * Vp + k] = __float2half_rn(x - __half2float(h0));
        blo[(size_t)(2 * t + 1) * Vp + k] = __float2half_rn(y - __half2float(h1));
    }
}

// Standalone application on split-K tiles (operand_mode 5): clusters of C
// CTAs, cluster (ib, ng) = site block ib x n-group ng of ns target slices;
// each CTA loads its 128 rows x K range of the scaled split of E by TMA
// (before waiting for the split pre-pass, which it does not read), then the
// pre-split source rows 2 t0 .. 2 t0 + Nn of its K range (plain FP16 hi and
// lo, one power-of-two scale per target slice and K range), one barrier per
// 64-wide K chunk, and issues each chunk's MMAs as it lands; it stages its
// partial unscaled per column by its own range's scales.  The C partials of a
// cluster are summed through distributed shared memory in rank order by the
// owners of the outputs (deterministic); a last cluster barrier keeps every
// member's shared memory alive until the others have read it.  E moves
// from L2 once per application (not once per slice tile).
template <bool DAG>
__global__ void __launch_bounds__(NTHR, 1)
    k_apply_sk(const __grid_constant__ CUtensorMap mhi, const __grid_constant__ CUtensorMap mlo,
               const __grid_constant__ CUtensorMap bhi, const __grid_constant__ CUtensorMap blo,
               const __grid_constant__ ChainView c, int C, int ns, const float2* in, float2* out, const float* inv) {
    extern __shared__ __align__(1024) uint8_t dyn[];
    TcState st;
    tc_setup(st, dyn, c.status);
    const SkGeom g = sk_geom(blockIdx.x, C, ns, c.V, c.Nt, c.Vr, c.Vp);
    TileBars& b = *st.bars;
    const uint32_t cb = 2u * (uint32_t)g.Nn * 128u;   // bytes of one stacked B chunk
    if (threadIdx.x == 0) {
        const uint32_t bar = smem_u32(&b.res_full);
        mbar_arrive_expect_tx(bar, (uint32_t)g.nch * kAChunkBytes);
        for (int j = 0; j < g.nch; ++j) {
            const uint32_t dst = smem_u32(st.base + (size_t)j * kAChunkBytes);
            const int x = 16 * g.ks0 + KCH * j;   // a multiple of 16 elements
            tma_load_2d(dst, &mhi, x, g.ib * TM, bar);
            tma_load_2d(dst + kATileBytes, &mlo, x, g.ib * TM, bar);
        }
    }
    // launched as a programmatic dependent of the split (see k_apply)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (threadIdx.x == 0) {
        for (int j = 0; j < g.nch; ++j) {
            const uint32_t bar = smem_u32(&b.skb[j]);
            const uint32_t dst = smem_u32(st.base + g.b_off + (size_t)j * cb);
            const int x = 16 * g.ks0 + KCH * j;
            mbar_arrive_expect_tx(bar, cb);
            tma_load_2d(dst, &bhi, x, 2 * g.t0, bar);
            tma_load_2d(dst + (uint32_t)g.Nn * 128u, &blo, x, 2 * g.t0, bar);
        }
        bool ok = mbar_wait(smem_u32(&b.res_full), 0, st.status);
        for (int j = 0; j < g.nch && ok; ++j) {
            ok = mbar_wait(smem_u32(&b.skb[j]), 0, st.status);
            if (ok) sk_issue_chunk(st, g, j, smem_u32(st.base + g.b_off + (size_t)j * cb),
                                   b.tmem_base);
        }
    }
    Team none = {};
    SkEpiOut<DAG> epi{in, out, c.cis_f, c.V, c.Nt};
    sk_finish<true>(st, g, none, c.V, c.e_inv, epi, inv, c.Nt);
    cluster_barrier_all();   // the partials stay until every member has read them
    tc_teardown(st);
}


// Per-launch set-up of the operand area: the tensor-core path takes its
// mbarriers and TMEM; the small (CUDA-core) mode needs only the area.
template <bool SMALL>
__device__ inline void persistent_setup(TcState& st, uint8_t* dyn, int* status) {
    if constexpr (SMALL) {
        st.base = smem_base(dyn);
        st.status = status;
        st.ntile = 0;
    } else {
        tc_setup(st, dyn, status);
    }
}
template <bool SMALL>
__device__ inline void persistent_teardown(TcState& st) {
    if constexpr (!SMALL) tc_teardown(st);
}

// scalars: [0] iterations [1] true residual [2] status [3] reliable updates
// KIND: TileKind of the FP32 iterations.
template <int KIND>
__global__ void __launch_bounds__(NTHR, 1)
    k_cg(const __grid_constant__ CUtensorMap mhi, const __grid_constant__ CUtensorMap mlo,
         const __grid_constant__ ChainView c, PersistentArgs pa, const double* phi, const double2* chi, double2* x) {
    extern __shared__ __align__(1024) uint8_t dyn[];
    __shared__ f64::Smem sm64;
    TcState st;
    persistent_setup<KIND == kKindSmall>(st, dyn, c.status);
    __shared__ ClusterSync s_cs;
    Team tm = make_team(c);
    cluster_begin(pa, &s_cs, c.status);
    set_phases(c, tm, phi);
    MixedResult res{};
    bool ok = team_barrier(tm) && cluster_ok(pa, tm);
    if (ok) ok = cg_mixed<KIND>(c, tm, st, sm64, &mhi, &mlo, pa, &s_cs, chi, x, res);
    if (ok && tm.rank == 0 && threadIdx.x == 0) {
        c.scalars[0] = res.iterations;
        c.scalars[1] = res.true_res;
        c.scalars[2] = res.status;
        c.scalars[3] = res.reliable_updates;
        c.scalars[4] = res.fp64_iterations;
    }
    persistent_teardown<KIND == kKindSmall>(st);
    if (pa.cluster > 1) cluster_barrier_all();   // no member leaves while others may push
}

// One HMC trajectory with mass preconditioning (Hasenbusch 2001) and the
// two-level nested leapfrog (Sexton and Weingarten 1992) on the mixed path:
// the same steps as f64::k_trajectory_hb, with every solve the mixed CG
// (FP32 iterations on the split-K tiles, whose epilogues scale the
// contraction by g for the heavy operator M_g = 1 - g S E D; FP64 reliable
// updates and true residuals of the same operator) and everything else in
// FP64.  Each solve's final FP64 residual leaves q = (M_g or M)^dag x, from
// which the forces are formed.  The first solve of each level starts from
// zero, the later ones from that level's previous solution (same right-hand
// side on the inner level; consecutive solves of a level sit one step of
// that level apart).  Results in c.scalars as the FP64 kernel's.
template <int KIND>
__device__ __noinline__ bool run_trajectory_hb(const ChainView& c, Team& tm, TcState& st,
                                              f64::Smem& sm64,
                                  const CUtensorMap* mhi, const CUtensorMap* mlo,
                                  const PersistentArgs& pa, ClusterSync* ics,
                                  const TrajArgs& a) {
    double* phi = a.phi;
    const double inv_dU = 1.0 / (c.delta * c.U);
    const double rsqrt2 = 0.70710678118654752440;
    const double gm1 = a.hb_gamma - 1.0;
    // 1. heat bath: momenta, the two noise vectors (rho_1 from stream 3 in
    // c.rho, rho_2 from the plain noise stream in c.xh), start energy
    double h0[3] = {0.0, 0.0, 0.0};
    HMC_TEAM_ELEMS(e, c, tm) {
        const double2 zp = normal_pair(philox_draw(a.seed, kStreamMomentum, a.traj, a.chain, e));
        const double2 z2 = normal_pair(philox_draw(a.seed, kStreamNoise, a.traj, a.chain, e));
        const double2 z1 = normal_pair(philox_draw(a.seed, kStreamHeavy, a.traj, a.chain, e));
        const double ph = phi[e];
        c.pi[e] = zp.x;
        const double2 r1 = make_double2(z1.x * rsqrt2, z1.y * rsqrt2);
        const double2 r2 = make_double2(z2.x * rsqrt2, z2.y * rsqrt2);
        c.rho[e] = r1;
        c.xh[e] = r2;
        c.phi_old[e] = ph;
        double s, co;
        sincos(ph, &s, &co);
        c.cis[e] = make_double2(co, s);
        c.cis_f[e] = make_float2((float)co, (float)s);
        h0[0] += ph * ph;
        h0[1] += r1.x * r1.x + r1.y * r1.y + r2.x * r2.x + r2.y * r2.y;
        h0[2] += zp.x * zp.x;
    }
    if (!team_sum<3>(tm, h0) || !cluster_ok(pa, tm)) return false;
    const double H0 = 0.5 * h0[0] * inv_dU + h0[1] + 0.5 * h0[2];
    int iters_in = 0, iters_out = 0, solves_in = 0, solves_out = 0, rus = 0, fp64_iters = 0;
    int status = HMC_OK;
    double max_res = 0.0;
    auto record = [&](const MixedResult& r, bool outer) {
        (outer ? iters_out : iters_in) += r.iterations;
        ++(outer ? solves_out : solves_in);
        rus += r.reliable_updates;
        fp64_iters += r.fp64_iterations;
        max_res = fmax(max_res, r.true_res);
        if (r.status != HMC_OK && status == HMC_OK) status = r.status;
    };
    // 2. chi_1 = M_g rho_1; chi_2 = M_g^dag (M_g M_g^dag)^{-1} M rho_2
    f64::EpiArgs eg = {};
    eg.hop_m1 = gm1;
    f64::EpiArgs e1 = {};
    f64::apply_team<kForm<KIND>, false, f64::EPI_STORE>(c, tm, c.rho, c.chi, eg, sm64);
    f64::apply_team<kForm<KIND>, false, f64::EPI_STORE>(c, tm, c.xh, c.phi2, e1, sm64);
    if (!team_barrier(tm)) return false;
    MixedResult res{};
    if (!cg_mixed<KIND>(c, tm, st, sm64, mhi, mlo, pa, ics, c.phi2, c.x2, res, false, gm1))
        return false;
    record(res, false);
    if (res.status == HMC_OK) {
        HMC_TEAM_ELEMS(e, c, tm) c.chi2[e] = c.q[e];   // q = M_g^dag x_2 (final residual)
    } else {
        f64::apply_team<kForm<KIND>, true, f64::EPI_STORE>(c, tm, c.x2, c.chi2, eg, sm64);
    }
    if (!team_barrier(tm)) return false;
    // 3. nested leapfrog
    const double ed = a.eps * c.delta;
    const double h = 1.0 / a.hb_inner;
    auto drift = [&](double cf) {
        HMC_TEAM_ELEMS(e, c, tm) {
            const double ph = fma(cf * ed, c.pi[e], phi[e]);
            phi[e] = ph;
            double s, co;
            sincos(ph, &s, &co);
            c.cis[e] = make_double2(co, s);
            c.cis_f[e] = make_float2((float)co, (float)s);
        }
        return team_barrier(tm);
    };
    // bosonic and heavy forces: F_B + F_1 = phi/(delta U) + 2 Im(x_1 conj(M_g^dag x_1))
    bool warm_in = false, warm_out = false;
    auto kick_inner = [&](double cf) {
        MixedResult r{};
        if (!cg_mixed<KIND>(c, tm, st, sm64, mhi, mlo, pa, ics, c.chi, c.x, r, warm_in, gm1))
            return false;
        warm_in = true;
        record(r, false);
        const double k = cf * ed;
        if (r.status == HMC_OK) {
            HMC_TEAM_ELEMS(e, c, tm) {
                const double2 xv = c.x[e], y = c.q[e];
                c.pi[e] -= k * (phi[e] * inv_dU + 2.0 * (xv.y * y.x - xv.x * y.y));
            }
        } else {
            f64::EpiArgs ef = {};
            ef.hop_m1 = gm1;
            ef.phi = phi;
            ef.pi = c.pi;
            ef.inv_dU = inv_dU;
            ef.kick = k;
            f64::apply_team<kForm<KIND>, true, f64::EPI_FORCE>(c, tm, c.x, nullptr, ef, sm64);
        }
        return team_barrier(tm);
    };
    // ratio force: F_2 = 2 Im(x_2 conj(M^dag x_2)) - 2 Im(conj(M_g^dag x_2 - x_2) chi_2)
    auto kick_outer = [&](double cf) {
        f64::apply_team<kForm<KIND>, false, f64::EPI_STORE>(c, tm, c.chi2, c.phi2, eg, sm64);   // M_g chi_2
        if (!team_barrier(tm)) return false;
        MixedResult r{};
        if (!cg_mixed<KIND>(c, tm, st, sm64, mhi, mlo, pa, ics, c.phi2, c.x2, r, warm_out, 0.0))
            return false;
        warm_out = true;
        record(r, true);
        const double k = cf * ed;
        f64::EpiArgs ef = {};
        ef.phi = phi;
        ef.pi = c.pi;
        ef.inv_dU = 0.0;          // the bosonic force sits on the inner level
        ef.kick = k;
        if (r.status == HMC_OK) {
            HMC_TEAM_ELEMS(e, c, tm) {
                const double2 xv = c.x2[e], y = c.q[e];
                c.pi[e] -= k * (2.0 * (xv.y * y.x - xv.x * y.y));
            }
        } else {
            f64::apply_team<kForm<KIND>, true, f64::EPI_FORCE>(c, tm, c.x2, nullptr, ef, sm64);
        }
        if (!team_barrier(tm)) return false;
        ef.hop_m1 = gm1;
        ef.chi = c.chi2;
        f64::apply_team<kForm<KIND>, true, f64::EPI_RATIO>(c, tm, c.x2, nullptr, ef, sm64);
        return team_barrier(tm);
    };
    if (!kick_outer(0.5)) return false;
    for (int k = 0; k < a.n_md; ++k) {
        for (int m = 0; m < a.hb_inner; ++m) {
            if (!kick_inner(m == 0 ? 0.5 * h : h)) return false;
            if (!drift(h)) return false;
        }
        if (!kick_inner(0.5 * h)) return false;
        if (!kick_outer(k + 1 < a.n_md ? 1.0 : 0.5)) return false;
    }
    // 4. end energy (the last kick of each level was at the final field) and
    // Metropolis
    double h1[4] = {0.0, 0.0, 0.0, 0.0};
    HMC_TEAM_ELEMS(e, c, tm) {
        const double ph = phi[e], pv = c.pi[e];
        const double2 c1 = c.chi[e], x1 = c.x[e], p2 = c.phi2[e], x2 = c.x2[e];
        h1[0] += ph * ph;
        h1[1] += c1.x * x1.x + c1.y * x1.y;
        h1[2] += p2.x * x2.x + p2.y * x2.y;
        h1[3] += pv * pv;
    }
    if (!team_sum<4>(tm, h1)) return false;
    const double H1 = 0.5 * h1[0] * inv_dU + h1[1] + h1[2] + 0.5 * h1[3];
    const double dH = H1 - H0;
    const double u = uniform_pair(philox_draw(a.seed, kStreamMetropolis, a.traj, a.chain, 0)).x;
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
        c.scalars[kTrajIters] = iters_in + iters_out;
        c.scalars[kTrajSolves] = solves_in + solves_out;
        c.scalars[kTrajRU] = rus;
        c.scalars[kTrajMaxRes] = max_res;
        c.scalars[kTrajStatus] = status;
        c.scalars[kTrajFp64Iters] = fp64_iters;
        c.scalars[kTrajItersOuter] = iters_out;
        c.scalars[kTrajSolvesOuter] = solves_out;
    }
    return true;
}

template <int KIND>
__global__ void __launch_bounds__(NTHR, 1)
    k_trajectory(const __grid_constant__ CUtensorMap mhi,
                 const __grid_constant__ CUtensorMap mlo, const __grid_constant__ ChainView c, PersistentArgs pa,
                 TrajArgs a) {
    extern __shared__ __align__(1024) uint8_t dyn[];
    __shared__ f64::Smem sm64;
    TcState st;
    persistent_setup<KIND == kKindSmall>(st, dyn, c.status);
    __shared__ ClusterSync s_cs;
    Team tm = make_team(c);
    cluster_begin(pa, &s_cs, c.status);
    if constexpr (KIND == kKindSplitK) {
        // (mass preconditioning: split-K tiles only; the host refuses it for
        // the other kinds)
        if (a.hb_inner > 0)
            run_trajectory_hb<KIND>(c, tm, st, sm64, &mhi, &mlo, pa, &s_cs, a);
        else
            run_trajectory<KIND>(c, tm, st, sm64, &mhi, &mlo, pa, &s_cs, a);
    } else {
        run_trajectory<KIND>(c, tm, st, sm64, &mhi, &mlo, pa, &s_cs, a);
    }
    persistent_teardown<KIND == kKindSmall>(st);
    if (pa.cluster > 1) cluster_barrier_all();   // no member leaves while others may push
}

// ---------------------------------------------------------------- batched
// One trajectory of a batch chain of kind KIND; not inlined, so each kind
// is compiled (and given registers) once, whichever phase runs it.
template <int KIND>
__device__ __noinline__ bool batch_traj(const BatchItem& it, TcState& st, f64::Smem& sm64,
                                        Team& tm, ClusterSync* ics, const TrajArgs& a) {
    const CUtensorMap* m = KIND == kKindSlice ? it.maps + 2 : it.maps;
    return run_trajectory<KIND>(it.v, tm, st, sm64, m, m + 1, it.pa, ics, a);
}

__global__ void __launch_bounds__(NTHR, 1)
    k_batch(const BatchItem* __restrict__ items, const int* __restrict__ order, int n,
            int* queue, const BatchCallArgs* call, double* outs, int csize) {
    extern __shared__ __align__(1024) uint8_t dyn[];
    __shared__ f64::Smem sm64;
    __shared__ ClusterSync s_cs;
    TcState st;
    tc_setup(st, dyn, items[0].v.status);
    if (csize > 1) cluster_sync_init(&s_cs, csize);
    batch_loop(items, order, n, queue, call, outs, csize, &s_cs,
               [&](const BatchItem& it, Team& tm, ClusterSync* ics, const TrajArgs& a) {
                   st.status = it.v.status;
                   if (it.pa.mode == kSmall)
                       return batch_traj<kKindSmall>(it, st, sm64, tm, ics, a);
                   if (it.pa.mode == kSlice)
                       return batch_traj<kKindSlice>(it, st, sm64, tm, ics, a);
                   return batch_traj<kKindSite>(it, st, sm64, tm, ics, a);
               });
    tc_teardown(st);
    if (csize > 1) cluster_barrier_all();   // no member leaves while others may push to it
}
}  // namespace tc

// ---------------------------------------------------------------- host side
static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    }
    return fn;
}

static bool splitk_shape(const hmc_ctx* c, int* C_out, int* ns_out);

static bool make_map(CUtensorMap* m, void* base, int Vr, int Vp, int box_rows = tc::TM) {
    auto enc = encode_fn();
    if (!enc) return false;
    cuuint64_t dims[2] = {(cuuint64_t)Vp, (cuuint64_t)Vr};
    cuuint64_t strides[1] = {(cuuint64_t)Vp * 2};
    cuuint32_t box[2] = {(cuuint32_t)tc::KCH, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, base, dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
           CUDA_SUCCESS;
}

// TMA map of a split-K source with halo rows: [rows][V] complex64 seen as
// 8-byte integers (the bits are copied as they are), boxes of 64 sites x
// box_rows rows, no swizzle, zero fill outside.
static bool make_map_src(CUtensorMap* m, void* base, int rows, int V, int box_rows) {
    auto enc = encode_fn();
    if (!enc) return false;
    cuuint64_t dims[2] = {(cuuint64_t)V, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)V * 8};
    cuuint32_t box[2] = {(cuuint32_t)tc::KCH, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_INT64, 2, base, dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
           CUDA_SUCCESS;
}

// Smallest slices-per-tile in {8, 16, 32, 64} with at most `slots` tiles.
static int pick_ns(int nti, int Nt, int slots) {
    int ns = 8;
    while (ns < tc::NMAX / 2 && nti * ((Nt + ns - 1) / ns) > slots) ns *= 2;
    return ns;
}

static void* dev_alloc(hmc_ctx* c, size_t bytes, bool* ok) {
    if (!*ok) return nullptr;
    void* p = nullptr;
    if (c->n_allocs >= (int)(sizeof(c->allocs) / sizeof(c->allocs[0])) ||
        cudaMalloc(&p, bytes) != cudaSuccess) {
        *ok = false;
        return nullptr;
    }
    c->allocs[c->n_allocs++] = p;
    cudaMemset(p, 0, bytes);
    return p;
}

// The FP16 splits of E, the split-K slots and the tensor maps: what only the
// tensor-core tiles use.  Contexts on the automatic choice with a series do
// without (at L = 24 they were most of the context's set-up).
static int tc_tiles_init(hmc_ctx* c) {
    ChainView& v = c->view;
    const int V = v.V;
    std::vector<double> E((size_t)V * V);
    if (cudaMemcpy(E.data(), v.E, E.size() * sizeof(double), cudaMemcpyDeviceToHost) !=
        cudaSuccess)
        return HMC_ERR_CUDA;
    // E = E_hi + 2^-11 E_lo with both parts in fp16, padded with zeros
    std::vector<__half> hi((size_t)v.Vr * v.Vp), lo((size_t)v.Vr * v.Vp);
    for (int r = 0; r < v.Vr; ++r)
        for (int k = 0; k < v.Vp; ++k) {
            const double e = (r < V && k < V) ? E[(size_t)r * V + k] : 0.0;
            const __half h = __float2half_rn((float)e);
            const double rem = (e - (double)__half2float(h)) * 2048.0;
            hi[(size_t)r * v.Vp + k] = h;
            lo[(size_t)r * v.Vp + k] = __float2half_rn((float)rem);
        }
    // slice-major tile: 2^eE E = Ew_hi + Ew_lo (plain remainder) with
    // max |2^eE E| in [2^14, 2^15)
    double emax = 0.0;
    for (size_t k = 0; k < E.size(); ++k) emax = std::max(emax, std::fabs(E[k]));
    int eE = 0;
    if (emax > 0.0 && std::isfinite(emax)) {
        int ex = 0;
        std::frexp(emax, &ex);   // emax in [2^(ex-1), 2^ex)
        eE = std::max(-100, std::min(100, 15 - ex));
    }
    const double es = std::ldexp(1.0, eE);
    std::vector<__half> whi((size_t)v.Vr * v.Vp), wlo((size_t)v.Vr * v.Vp);
    for (int r = 0; r < v.Vr; ++r)
        for (int k = 0; k < v.Vp; ++k) {
            const double e = (r < V && k < V) ? E[(size_t)r * V + k] * es : 0.0;
            const __half h = __float2half_rn((float)e);
            whi[(size_t)r * v.Vp + k] = h;
            wlo[(size_t)r * v.Vp + k] = __float2half_rn((float)(e - (double)__half2float(h)));
        }
    v.e_inv = (float)std::ldexp(1.0, -eE);
    bool ok = true;
    void* dhi = dev_alloc(c, hi.size() * sizeof(__half), &ok);
    void* dlo = dev_alloc(c, lo.size() * sizeof(__half), &ok);
    void* dwhi = dev_alloc(c, whi.size() * sizeof(__half), &ok);
    void* dwlo = dev_alloc(c, wlo.size() * sizeof(__half), &ok);
    v.sk_b16 = nullptr;
    v.sk_maps = nullptr;
    v.gslots = (unsigned long long*)dev_alloc(c, tc::kGatherSlots * sizeof(unsigned long long),
                                              &ok);
    if (!ok) return HMC_ERR_CUDA;
    if (cudaMemcpy(dhi, hi.data(), hi.size() * sizeof(__half), cudaMemcpyHostToDevice) !=
            cudaSuccess ||
        cudaMemcpy(dlo, lo.data(), lo.size() * sizeof(__half), cudaMemcpyHostToDevice) !=
            cudaSuccess ||
        cudaMemcpy(dwhi, whi.data(), whi.size() * sizeof(__half), cudaMemcpyHostToDevice) !=
            cudaSuccess ||
        cudaMemcpy(dwlo, wlo.data(), wlo.size() * sizeof(__half), cudaMemcpyHostToDevice) !=
            cudaSuccess)
        return HMC_ERR_CUDA;
    v.E_hi = dhi;
    v.E_lo = dlo;
    v.Ew_hi = dwhi;
    v.Ew_lo = dwlo;
    c->tc = new TcCtx();
    if (!make_map(&c->tc->map_hi, dhi, v.Vr, v.Vp) || !make_map(&c->tc->map_lo, dlo, v.Vr, v.Vp) ||
        !make_map(&c->tc->map_shi, dwhi, v.Vr, v.Vp) || !make_map(&c->tc->map_slo, dwlo, v.Vr, v.Vp))
        return HMC_ERR_CUDA;
    {
        // slice-major tiles: all sites in one tile up to 288; standalone
        // applications above 256 sites take tiles of 144 (one instruction,
        // same TMA box) and as many slice tiles as fill one wave
        TcCtx* t = c->tc;
        t->w_cg = tc::wide_sites(V);
        const tc::WideGeom g = tc::wide_geom(t->w_cg);
        const int box = t->w_cg / g.nmma;
        t->w_apply = V > tc::kWMaxN ? box : t->w_cg;
        // standalone tiles of up to 64 slices (balanced); each tile's K is
        // split over a cluster of up to 8 CTAs while the tiles x split fill
        // the GPU (at least one K chunk per CTA)
        const int nsi = (V + t->w_apply - 1) / t->w_apply;
        const int ntt = (v.Nt + tc::kWSlices - 1) / tc::kWSlices;
        t->ns_wapply = (v.Nt + ntt - 1) / ntt;
        if (c->params.operand_mode == 4 && c->params.tile_slices > 0)
            t->ns_wapply = c->params.tile_slices;
        const int tiles = nsi * ((v.Nt + t->ns_wapply - 1) / t->ns_wapply);
        t->csplit_apply = std::max(1, std::min(std::min(tc::kMaxClusterW, v.Vp / tc::KCH),
                                               c->num_sms / std::max(1, tiles)));
        if (!make_map(&t->map_whi, dwhi, v.Vr, v.Vp, box) ||
            !make_map(&t->map_wlo, dwlo, v.Vr, v.Vp, box))
            return HMC_ERR_CUDA;
    }
    c->tc->ns_apply = pick_ns(v.Vr / tc::TM, v.Nt, c->num_sms);
    if (c->params.tile_slices > 0 && c->params.operand_mode != 4 && c->params.operand_mode != 5)
        c->tc->ns_apply = c->params.tile_slices;
    {
        // pre-split B of standalone applications (rows padded by 64 zero rows)
        const int nb = ((2 * c->tc->ns_apply + 15) / 16) * 16;   // MMA N = TMA box rows
        c->tc->b_rows = 2 * v.Nt + 128;   // a 128-row box from any 2t stays inside
        const size_t nbh = (size_t)c->tc->b_rows * v.Vp;
        bool okb = true;
        c->tc->bhi = (__half*)dev_alloc(c, nbh * sizeof(__half), &okb);
        c->tc->blo = (__half*)dev_alloc(c, nbh * sizeof(__half), &okb);
        c->tc->inv_col = (float*)dev_alloc(c, (size_t)v.Nt * sizeof(float), &okb);
        if (!okb || !make_map(&c->tc->map_bhi, c->tc->bhi, c->tc->b_rows, v.Vp, nb) ||
            !make_map(&c->tc->map_blo, c->tc->blo, c->tc->b_rows, v.Vp, nb) ||
            !make_map(&c->tc->map_uhi, c->tc->bhi, c->tc->b_rows, v.Vp,
                      tc::wide_u_rows(c->tc->ns_wapply)) ||
            !make_map(&c->tc->map_ulo, c->tc->blo, c->tc->b_rows, v.Vp,
                      tc::wide_u_rows(c->tc->ns_wapply)))
            return HMC_ERR_CUDA;
        // split-K standalone applications (operand_mode 5)
        c->tc->sk_C_apply = 0;
        c->tc->sk_ns_apply = 0;
        int skC = 0, skns = 0;
        if (c->params.operand_mode == 5 && splitk_shape(c, &skC, &skns)) {
            if (!make_map(&c->tc->map_skb_hi, c->tc->bhi, c->tc->b_rows, v.Vp, tc::sk_nn(skns)) ||
                !make_map(&c->tc->map_skb_lo, c->tc->blo, c->tc->b_rows, v.Vp, tc::sk_nn(skns)))
                return HMC_ERR_CUDA;
            c->tc->sk_C_apply = skC;
            c->tc->sk_ns_apply = skns;
            c->tc->inv_sk = (float*)dev_alloc(c, (size_t)v.Nt * skC * sizeof(float), &okb);
            if (!okb) return HMC_ERR_CUDA;
            // the CG's sources: r and u with their halo rows, boxes of ns rows,
            // and their FP16 splits, boxes of sk_nn(ns) rows
            const int rows16 = 2 * (v.Nt + 2);
            const size_t plane = (size_t)rows16 * v.Vp;
            __half_raw* b16 = (__half_raw*)dev_alloc(c, 4 * plane * sizeof(__half), &okb);
            if (!okb) return HMC_ERR_CUDA;
            c->view.sk_b16 = b16;
            CUtensorMap hm[6];
            if (!make_map_src(&hm[0], c->view.rh_f, v.Nt + 2, V, skns) ||
                !make_map_src(&hm[1], c->view.u_f, v.Nt + 2, V, skns))
                return HMC_ERR_CUDA;
            for (int q = 0; q < 4; ++q)
                if (!make_map(&hm[2 + q], b16 + q * plane, rows16, v.Vp, tc::sk_nn(skns)))
                    return HMC_ERR_CUDA;
            void* dm = dev_alloc(c, sizeof(hm), &okb);
            if (!okb || cudaMemcpy(dm, hm, sizeof(hm), cudaMemcpyHostToDevice) != cudaSuccess)
                return HMC_ERR_CUDA;
            c->view.sk_maps = dm;
        }
        const int split_smem = V * (int)sizeof(float2);
        for (const void* k : {(const void*)tc::k_split<false, false>,
                              (const void*)tc::k_split<true, false>,
                              (const void*)tc::k_split<false, true>,
                              (const void*)tc::k_split<true, true>})
            if (split_smem > 48 * 1024 &&
                cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     split_smem) != cudaSuccess)
                return HMC_ERR_CUDA;
    }
    const void* kernels[] = {(const void*)tc::k_apply<false>,
                             (const void*)tc::k_apply<true>,
                             (const void*)tc::k_apply_sk<false>,
                             (const void*)tc::k_apply_sk<true>,
                             (const void*)tc::k_apply_w<false>,
                             (const void*)tc::k_apply_w<true>,
                             (const void*)tc::k_cg<tc::kKindSite>,
                             (const void*)tc::k_trajectory<tc::kKindSite>,
                             (const void*)tc::k_cg<tc::kKindSmall>,
                             (const void*)tc::k_trajectory<tc::kKindSmall>,
                             (const void*)tc::k_cg<tc::kKindSlice>,
                             (const void*)tc::k_trajectory<tc::kKindSlice>,
                             (const void*)tc::k_cg<tc::kKindSplitK>,
                             (const void*)tc::k_trajectory<tc::kKindSplitK>};
    for (const void* k : kernels)
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)tc::kSmemBytes) != cudaSuccess)
            return HMC_ERR_CUDA;
    // the small-lattice mode may run on clusters of up to 16 CTAs (beyond the
    // portable 8); a device that cannot co-schedule them refuses the launch
    for (const void* k : {(const void*)tc::k_cg<tc::kKindSmall>,
                          (const void*)tc::k_trajectory<tc::kKindSmall>})
        if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
            cudaSuccess)
            (void)cudaGetLastError();
    return HMC_OK;
}

// FP32 workspaces of the mixed path, and what its kernels need.
int tc_ctx_init(hmc_ctx* c) {
    ChainView& v = c->view;
    v.Vr = ((v.V + tc::TM - 1) / tc::TM) * tc::TM;
    v.Vp = ((v.V + tc::KCH - 1) / tc::KCH) * tc::KCH;
    bool ok = true;
    const size_t N = (size_t)v.N;
    v.cis_f = (float2*)dev_alloc(c, N * sizeof(float2), &ok);
    v.r_f = (float2*)dev_alloc(c, N * sizeof(float2), &ok);
    v.p_f = (float2*)dev_alloc(c, N * sizeof(float2), &ok);
    v.p2_f = (float2*)dev_alloc(c, N * sizeof(float2), &ok);
    v.q_f = (float2*)dev_alloc(c, N * sizeof(float2), &ok);
    v.x_f = (float2*)dev_alloc(c, N * sizeof(float2), &ok);
    v.g_f = (float2*)dev_alloc(c, N * sizeof(float2), &ok);
    const size_t Nh = (size_t)(v.Nt + 2) * v.V;   // split-K sources with the halo rows
    v.u_f = (float2*)dev_alloc(c, Nh * sizeof(float2), &ok);
    v.rh_f = (float2*)dev_alloc(c, Nh * sizeof(float2), &ok);
    if (!ok) return HMC_ERR_CUDA;
    return series_chosen(c) ? series_ctx_init(c) : tc_tiles_init(c);
}

void tc_ctx_free(hmc_ctx* c) {
    delete c->tc;
    c->tc = nullptr;
}

// Launch an application kernel as a programmatic dependent of the split
// that precedes it on the stream (its set-up overlaps the split; it waits
// with griddepcontrol.wait before reading the split's output), in clusters
// of `cluster` CTAs when cluster > 1.
static int launch_dependent(const void* fn, int grid, int cluster, void** args,
                            cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(tc::NTHR);
    cfg.dynamicSmemBytes = tc::kSmemBytes;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)cluster;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelExC(&cfg, fn, args) == cudaSuccess ? HMC_OK : HMC_ERR_CUDA;
}

int tc_apply(hmc_ctx* c, const double* phi, const float2* in, float2* out, bool dag,
             cudaStream_t s) {
    const ChainView& v = c->view;
    if (series_chosen(c)) return series_apply(v, phi, in, out, dag, s);
    const size_t split_smem = (size_t)v.V * sizeof(float2);
    TcCtx* t = c->tc;
    if (c->params.operand_mode == 5 && t->sk_C_apply > 0) {
        int C = t->sk_C_apply, ns = t->sk_ns_apply;
        const int grid = (v.Vr / tc::TM) * ((v.Nt + ns - 1) / ns) * C;
        const dim3 sgrid(v.Nt, C);
        if (dag)
            tc::k_split_sk<true><<<sgrid, tc::kSplitSkThreads, 0, s>>>(
                phi, in, v.cis_f, t->bhi, t->blo, t->inv_sk, v.V, v.Vp, v.Nt, C);
        else
            tc::k_split_sk<false><<<sgrid, tc::kSplitSkThreads, 0, s>>>(
                phi, in, v.cis_f, t->bhi, t->blo, t->inv_sk, v.V, v.Vp, v.Nt, C);
        if (cudaGetLastError() != cudaSuccess) return HMC_ERR_CUDA;
        ChainView vv = v;
        const float2* inp = in;
        float2* outp = out;
        const float* invp = t->inv_sk;
        void* args[] = {&t->map_shi, &t->map_slo, &t->map_skb_hi, &t->map_skb_lo, &vv,
                        &C, &ns, &inp, &outp, &invp};
        return launch_dependent(
            dag ? (const void*)tc::k_apply_sk<true> : (const void*)tc::k_apply_sk<false>, grid,
            C, args, s);
    }
    if (c->params.operand_mode == 4) {
        int W = t->w_apply, ns = t->ns_wapply, cs = t->csplit_apply;
        const int tiles = ((v.V + W - 1) / W) * ((v.Nt + ns - 1) / ns);
        if (dag)
            tc::k_split<true, true><<<v.Nt, tc::kSplitThreads, split_smem, s>>>(
                phi, in, v.cis_f, t->bhi, t->blo, t->inv_col, v.V, v.Vp, v.Nt);
        else
            tc::k_split<false, true><<<v.Nt, tc::kSplitThreads, split_smem, s>>>(
                phi, in, v.cis_f, t->bhi, t->blo, t->inv_col, v.V, v.Vp, v.Nt);
        if (cudaGetLastError() != cudaSuccess) return HMC_ERR_CUDA;
        ChainView vv = v;
        const float2* inp = in;
        float2* outp = out;
        const float* invp = t->inv_col;
        void* args[] = {&t->map_whi, &t->map_wlo, &t->map_uhi, &t->map_ulo, &vv,
                        &W, &ns, &cs, &inp, &outp, &invp};
        return launch_dependent(
            dag ? (const void*)tc::k_apply_w<true> : (const void*)tc::k_apply_w<false>,
            tiles * cs, cs, args, s);
    }
    int ns = c->tc->ns_apply;
    const int tiles = (v.Vr / tc::TM) * ((v.Nt + ns - 1) / ns);
    if (dag)
        tc::k_split<true, false><<<v.Nt, tc::kSplitThreads, split_smem, s>>>(
            phi, in, v.cis_f, t->bhi, t->blo, t->inv_col, v.V, v.Vp, v.Nt);
    else
        tc::k_split<false, false><<<v.Nt, tc::kSplitThreads, split_smem, s>>>(
            phi, in, v.cis_f, t->bhi, t->blo, t->inv_col, v.V, v.Vp, v.Nt);
    if (cudaGetLastError() != cudaSuccess) return HMC_ERR_CUDA;
    ChainView vv = v;
    const float2* inp = in;
    float2* outp = out;
    const float* invp = t->inv_col;
    void* args[] = {&t->map_hi, &t->map_lo, &t->map_bhi, &t->map_blo, &vv, &ns, &inp, &outp, &invp};
    return launch_dependent(dag ? (const void*)tc::k_apply<true> : (const void*)tc::k_apply<false>,
                            tiles, 1, args, s);
}

static int team_size(hmc_ctx* c, const void* kernel) {
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, tc::NTHR, tc::kSmemBytes) !=
            cudaSuccess ||
        occ < 1)
        return -1;
    const ChainView& v = c->view;
    const int f64_tiles = ((v.V + f64::TI - 1) / f64::TI) * ((v.Nt + f64::TT - 1) / f64::TT);
    const int tc_tiles = (v.Vr / tc::TM) * ((v.Nt + 7) / 8);
    int want = std::max(f64_tiles, tc_tiles);
    if (c->params.team_ctas > 0) want = c->params.team_ctas;
    int g = std::min(c->num_sms * occ, kMaxTeam);
    return std::max(1, std::min(g, want));
}

// Resident B per slice tile pays when a CTA runs several site blocks of the
// same slices: streaming layout, at least two site blocks, every CTA of the
// inner team with a slice tile, and the tile's B within the area after the
// E ring.
static bool res_b_ok(const ChainView& v, int mode, int ns, int inner) {
    const int nti = v.Vr / tc::TM, ntt = (v.Nt + ns - 1) / ns;
    const int N = ((2 * ns + 15) / 16) * 16;
    return mode == tc::kStreaming && nti >= 2 && inner <= ntt &&
           tc::res_b_bytes(N, v.Vp) <= tc::kResBArea;
}

// Cluster size of the small-lattice CUDA-core mode: inner_ctas when given,
// else the largest of 8, 4, 2, 1 that fits (each CTA at least 2 slices).
static int small_cluster(const hmc_ctx* c) {
    const ChainView& v = c->view;
    if (c->params.inner_ctas > 0)
        return tc::small_feasible(v.V, v.Nt, c->params.inner_ctas) ? c->params.inner_ctas : 0;
    for (int C = 16; C >= 1; C >>= 1)
        if ((C == 1 || v.Nt >= 2 * C) && tc::small_feasible(v.V, v.Nt, C)) return C;
    return 0;
}

// Split-K shape (operand_mode 5): slices per n-group (tile_slices, else the
// fewest n-groups of at most 64 slices, balanced) and CTAs per cluster
// (inner_ctas, else the smallest of 6, 8, 4, 2 whose K range fits the
// shared memory); false if the requested shape does not fit.
static bool splitk_shape(const hmc_ctx* c, int* C_out, int* ns_out) {
    const ChainView& v = c->view;
    int ns = c->params.tile_slices;
    if (ns <= 0) {
        const int nng = (v.Nt + 63) / 64;
        ns = (v.Nt + nng - 1) / nng;
    }
    if (ns < 1 || ns > 64) return false;
    const int Nn = tc::sk_nn(ns);
    const int KS = (v.V + 15) / 16;
    auto fits = [&](int C) {
        if (C < 2 || C > tc::kSkMaxCluster || C > KS) return false;
        const int steps = (KS + C - 1) / C;
        const int nch = tc::sk_chunks(steps);
        const int own_slices = (std::min(ns, v.Nt) + C - 1) / C;
        return nch <= tc::kSkMaxChunks &&
               tc::sk_smem_total(nch, Nn, own_slices) <= tc::kOperandBytes;
    };
    int C = c->params.inner_ctas;
    if (C > 0) {
        if (!fits(C)) return false;
    } else {
        C = 0;
        for (int cand : {6, 8, 4, 2})
            if (fits(cand)) { C = cand; break; }
        if (!C) return false;
    }
    *C_out = C;
    *ns_out = ns;
    return true;
}

static tc::PersistentArgs persistent_args(hmc_ctx* c, int grid, double tol, int max_iter) {
    tc::PersistentArgs pa;
    const ChainView& v = c->view;
    pa.sk_C = 0;
    if (c->params.operand_mode == 5) {
        // split-K tiles with E' resident: nib x nng clusters of C CTAs form
        // the inner team (0 CTAs if the shape does not fit)
        int C = 0, ns = 0;
        pa.mode = tc::kSplitK;
        pa.inner = 0;
        if (splitk_shape(c, &C, &ns)) {
            pa.sk_C = C;
            pa.ns_tile = ns;
            pa.inner = (v.Vr / tc::TM) * ((v.Nt + ns - 1) / ns) * C;
        }
        pa.cluster = C;
        pa.vec_resident = 0;
        pa.res_b = 0;
        pa.wide_W = 0;
        pa.tol = tol;
        pa.max_iter = max_iter;
        pa.ru_delta = c->params.ru_delta;
        pa.ru_every = c->params.ru_every;
        (void)grid;
        return pa;
    }
    if (c->params.operand_mode == 3) {
        // CUDA-core cluster solver; grid is a multiple of the cluster size
        pa.mode = tc::kSmall;
        pa.inner = small_cluster(c);
        pa.ns_tile = 8;
        pa.vec_resident = 0;
        pa.tol = tol;
        pa.max_iter = max_iter;
        pa.ru_delta = c->params.ru_delta;
        pa.ru_every = c->params.ru_every;
        pa.cluster = 0;
        pa.res_b = 0;
        pa.wide_W = 0;
        return pa;
    }
    pa.wide_W = 0;
    if (c->params.operand_mode == 4) {
        // slice-major tiles: one CTA per tile at 64 slices by default
        pa.mode = tc::kSlice;
        pa.wide_W = c->tc->w_cg;
        const int ntt64 = (v.Nt + tc::kWSlices - 1) / tc::kWSlices;
        pa.inner = std::min(grid, ((v.V + pa.wide_W - 1) / pa.wide_W) * ntt64);
        if (c->params.inner_ctas > 0) pa.inner = std::min(c->params.inner_ctas, grid);
        const int nsi = (v.V + pa.wide_W - 1) / pa.wide_W;
        // slices per tile: balanced over enough slice tiles for the team
        const int want_tt = std::max(ntt64, (pa.inner + nsi - 1) / nsi);
        pa.ns_tile = std::min(tc::kWSlices, (v.Nt + want_tt - 1) / want_tt);
        if (c->params.tile_slices > 0) pa.ns_tile = c->params.tile_slices;
        pa.vec_resident = 0;
        pa.tol = tol;
        pa.max_iter = max_iter;
        pa.ru_delta = c->params.ru_delta;
        pa.ru_every = c->params.ru_every;
        pa.cluster = 0;
        pa.res_b = 0;
        return pa;
    }
    // inner team: one CTA while the whole lattice fits in a handful of tiles
    // (a single CTA needs no inter-CTA barrier), else the whole launch
    const int nti = v.Vr / tc::TM;
    const int nk = v.Vp / tc::KCH;
    // resident E when one site block's rows (all K) fit and every site block
    // gets its own CTA; else stream E through the ring
    const bool can_resident = nk <= tc::kMaxResidentChunks && nti <= grid;
    pa.mode = (c->params.operand_mode == 2 || (c->params.operand_mode == 0 && can_resident))
                  ? tc::kResident
                  : tc::kStreaming;
    if (pa.mode == tc::kResident && !can_resident) pa.mode = tc::kStreaming;
    pa.vec_resident = 0;
    if (pa.mode == tc::kResident) {
        // one CTA per site block, or (inner_ctas) a multiple of that: the
        // extra CTAs take further slice tiles of the same block
        pa.inner = nti;
        if (c->params.inner_ctas > nti)
            pa.inner = std::min(c->params.inner_ctas / nti, grid / nti) * nti;
        pa.ns_tile = std::min(16, pick_ns(1, v.Nt, pa.inner / nti));
        const size_t free_bytes =
            tc::kOperandBytes - (size_t)nk * tc::kAChunkBytes - tc::kMaxStages * tc::kBStageSmall;
        pa.vec_resident =
            (pa.inner == 1 && 6 * sizeof(float2) * (size_t)v.N <= free_bytes) ? 1 : 0;
    } else {
        pa.inner = nti * ((v.Nt + 31) / 32) <= 2 ? 1 : grid;
        if (c->params.inner_ctas > 0) pa.inner = std::min(c->params.inner_ctas, grid);
        pa.ns_tile = pick_ns(nti, v.Nt, pa.inner);
    }
    if (c->params.tile_slices > 0) pa.ns_tile = c->params.tile_slices;
    if (pa.mode == tc::kResident && pa.ns_tile > 16) pa.ns_tile = 16;   // 8 KB B stages
    pa.tol = tol;
    pa.max_iter = max_iter;
    pa.ru_delta = c->params.ru_delta;
    pa.ru_every = c->params.ru_every;
    pa.cluster = 0;
    pa.res_b = res_b_ok(v, pa.mode, pa.ns_tile, pa.inner) ? 1 : 0;
    return pa;
}

// Cooperative launch of a persistent kernel.  An inner team of 2..8 CTAs
// that divides the grid is launched as thread-block clusters (cluster 0 is
// the inner team) unless cluster_mode says never; in automatic mode a
// refused cluster launch falls back to global-memory team barriers.
// `pa` is the object args points at.
static int launch_persistent(hmc_ctx* c, const void* fn, int grid, void** args,
                             tc::PersistentArgs& pa, cudaStream_t s) {
    int cm = c->params.cluster_mode;
    if (!control_reset(c->view, grid, s)) return HMC_ERR_CUDA;
    if (pa.mode == tc::kSmall) {
        // the small mode reads its peers' shared memory: a cluster or nothing
        if (pa.inner < 1 || grid % pa.inner != 0) return HMC_ERR_UNSUPPORTED;
        if (pa.inner > 1) {
            if (cm == 2) return HMC_ERR_UNSUPPORTED;
            cm = 1;
        }
    }
    const int max_cluster = pa.mode == tc::kSmall ? tc::kSmallMaxCluster : 8;
    const bool want = cm != 2 && pa.inner > 1 && pa.inner <= max_cluster && grid % pa.inner == 0;
    if (cm == 1 && !want) return HMC_ERR_UNSUPPORTED;
    if (want) {
        pa.cluster = pa.inner;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(grid);
        cfg.blockDim = dim3(tc::NTHR);
        cfg.dynamicSmemBytes = tc::kSmemBytes;
        cfg.stream = s;
        // the CTAs of one cluster are scheduled together, so a launch that
        // is one cluster needs no cooperative attribute; several clusters
        // take it for the team barriers between them
        cudaLaunchAttribute at[2];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)pa.inner;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        at[1].id = cudaLaunchAttributeCooperative;
        at[1].val.cooperative = 1;
        cfg.attrs = at;
        cfg.numAttrs = grid == pa.inner ? 1 : 2;
        if (cudaLaunchKernelExC(&cfg, fn, args) == cudaSuccess) return HMC_OK;
        (void)cudaGetLastError();   // a refused configuration is not sticky
        pa.cluster = 0;
        if (cm == 1) return HMC_ERR_UNSUPPORTED;
    }
    return cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(tc::NTHR), args, tc::kSmemBytes, s) ==
                   cudaSuccess
               ? HMC_OK
               : HMC_ERR_CUDA;
}

// Split-K mode: a cooperative launch of thread-block clusters of sk_C CTAs,
// as many clusters as can be resident at once (at least the inner team's;
// team_ctas caps it), with the team-sum slots cleared first.
static int launch_splitk(hmc_ctx* c, const void* fn, void** args, tc::PersistentArgs& pa,
                         cudaStream_t s) {
    if (pa.inner < 1 || pa.sk_C < 2) return HMC_ERR_UNSUPPORTED;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(tc::NTHR);
    cfg.dynamicSmemBytes = tc::kSmemBytes;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)pa.sk_C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeCooperative;
    at[1].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3(pa.inner);
    int nclu = 0;
    if (cudaOccupancyMaxActiveClusters(&nclu, fn, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return HMC_ERR_UNSUPPORTED;
    }
    int grid = std::min(nclu * pa.sk_C, kMaxTeam / pa.sk_C * pa.sk_C);
    if (c->params.team_ctas > 0)
        grid = std::min(grid, std::max(c->params.team_ctas / pa.sk_C * pa.sk_C, pa.inner));
    if (grid < pa.inner) return HMC_ERR_UNSUPPORTED;
    cfg.gridDim = dim3(grid);
    // HMC_PROFILE_NONCOOPERATIVE=1: the same launch without the cooperative
    // attribute, for profilers that refuse cooperative cluster launches.  The
    // grid is the clusters that can be resident at once, so in practice every
    // CTA runs; were one not resident, the bounded team waits would end the
    // launch with HMC_ERR_TIMEOUT.
    cfg.numAttrs = getenv("HMC_PROFILE_NONCOOPERATIVE") ? 1 : 2;
    if (!control_reset(c->view, grid, s) ||
        cudaMemsetAsync(c->view.gslots, 0, tc::kGatherSlots * sizeof(unsigned long long), s) !=
            cudaSuccess)
        return HMC_ERR_CUDA;
    pa.cluster = pa.sk_C;
    if (cudaLaunchKernelExC(&cfg, fn, args) != cudaSuccess) {
        (void)cudaGetLastError();
        return HMC_ERR_UNSUPPORTED;
    }
    return HMC_OK;
}

// Small mode: the launch is a whole number of clusters.
static int round_grid(const tc::PersistentArgs& pa, int grid) {
    if (pa.mode != tc::kSmall || pa.inner < 1) return grid;
    return std::max(pa.inner, grid / pa.inner * pa.inner);
}

int tc_cg(hmc_ctx* c, const double* phi, const double2* chi, double2* x, double tol,
          int max_iter, cudaStream_t s) {
    if (series_chosen(c)) return series_cg(c, phi, chi, x, tol, max_iter, s);
    int grid = team_size(c, (const void*)tc::k_cg<tc::kKindSite>);
    if (grid < 1) return HMC_ERR_CUDA;
    tc::PersistentArgs pa = persistent_args(c, grid, tol, max_iter);
    if (pa.mode == tc::kSmall && pa.inner < 1) return HMC_ERR_UNSUPPORTED;
    grid = round_grid(pa, grid);
    ChainView v = c->view;
    if (pa.mode == tc::kSplitK) {
        void* args[] = {&c->tc->map_shi, &c->tc->map_slo, &v, &pa, &phi, &chi, &x};
        return launch_splitk(c, (const void*)tc::k_cg<tc::kKindSplitK>, args, pa, s);
    }
    const void* fn = pa.mode == tc::kSmall   ? (const void*)tc::k_cg<tc::kKindSmall>
                     : pa.mode == tc::kSlice ? (const void*)tc::k_cg<tc::kKindSlice>
                                             : (const void*)tc::k_cg<tc::kKindSite>;
    const bool sl = pa.mode == tc::kSlice;
    void* args[] = {sl ? &c->tc->map_whi : &c->tc->map_hi, sl ? &c->tc->map_wlo : &c->tc->map_lo,
                    &v, &pa, &phi, &chi, &x};
    return launch_persistent(c, fn, grid, args, pa, s);
}

int tc_trajectory(hmc_ctx* c, const TrajArgs& a, cudaStream_t s) {
    if (series_chosen(c)) return series_trajectory(c, a, s);
    int grid = team_size(c, (const void*)tc::k_trajectory<tc::kKindSite>);
    if (grid < 1) return HMC_ERR_CUDA;
    tc::PersistentArgs pa = persistent_args(c, grid, a.tol, a.max_iter);
    if (pa.mode == tc::kSmall && pa.inner < 1) return HMC_ERR_UNSUPPORTED;
    grid = round_grid(pa, grid);
    ChainView v = c->view;
    TrajArgs av = a;
    if (pa.mode == tc::kSplitK) {
        void* args[] = {&c->tc->map_shi, &c->tc->map_slo, &v, &pa, &av};
        return launch_splitk(c, (const void*)tc::k_trajectory<tc::kKindSplitK>, args, pa, s);
    }
    const void* fn = pa.mode == tc::kSmall   ? (const void*)tc::k_trajectory<tc::kKindSmall>
                     : pa.mode == tc::kSlice ? (const void*)tc::k_trajectory<tc::kKindSlice>
                                             : (const void*)tc::k_trajectory<tc::kKindSite>;
    const bool sl = pa.mode == tc::kSlice;
    void* args[] = {sl ? &c->tc->map_whi : &c->tc->map_hi, sl ? &c->tc->map_wlo : &c->tc->map_lo,
                    &v, &pa, &av};
    return launch_persistent(c, fn, grid, args, pa, s);
}


// ---------------------------------------------------------------- batch (host)
struct TcBatch {
    int n = 0;
    int grid = 0;
    int csize = 1;                   // CTAs per cluster (> 1: team chains present)
    // the kernel: the tensor-core one, or (every chain on the automatic choice
    // and its series) the series' one
    const void* kernel = nullptr;
    bool series = false;
    int threads = 0;
    unsigned smem = 0;
    int mail_V = 0;                  // series: sites of a mail box
    std::vector<hmc_ctx*> ctxs;
    std::vector<long long> offsets;   // n + 1
    tc::BatchItem* d_items = nullptr;
    int* d_order = nullptr;
    int* d_queue = nullptr;
    tc::BatchCallArgs* d_call = nullptr;
    tc::BatchCallArgs* h_call = nullptr;   // pinned
    double* d_outs = nullptr;
    double* h_outs = nullptr;          // pinned
    CUtensorMap* d_maps = nullptr;
    cudaStream_t stream = nullptr;
    cudaEvent_t ready = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    double* graph_phi = nullptr;
};

void tc_batch_destroy(TcBatch* b) {
    if (!b) return;
    if (b->stream) cudaStreamSynchronize(b->stream);
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    if (b->ready) cudaEventDestroy(b->ready);
    if (b->stream) cudaStreamDestroy(b->stream);
    cudaFree(b->d_items);
    cudaFree(b->d_order);
    cudaFree(b->d_queue);
    cudaFree(b->d_call);
    cudaFree(b->d_outs);
    cudaFree(b->d_maps);
    if (b->h_call) cudaFreeHost(b->h_call);
    if (b->h_outs) cudaFreeHost(b->h_outs);
    for (hmc_ctx* c : b->ctxs) hmc_ctx_destroy(c);
    delete b;
}

// Makespan of a batch step as the kernel schedules it: the first k of the chains
// `order` (by decreasing cost) as cluster teams, each taken by the next free
// cluster of csize CTAs, whose CTAs then take one-CTA chains on their own.
static double series_makespan(const std::vector<double>& solo, const std::vector<double>& team,
                              const std::vector<int>& order, const std::vector<char>& is_team,
                              int clusters, int csize) {
    using Heap = std::priority_queue<double, std::vector<double>, std::greater<double>>;
    Heap clu(std::greater<double>(), std::vector<double>(clusters, 0.0));
    double end = 0.0;
    for (int i : order)
        if (is_team[i]) {
            const double t = clu.top() + team[i];
            clu.pop();
            clu.push(t);
            end = std::max(end, t);
        }
    std::vector<double> start;
    for (; !clu.empty(); clu.pop()) start.insert(start.end(), csize, clu.top());
    Heap cta(std::greater<double>(), std::move(start));
    for (int i : order)
        if (!is_team[i]) {
            const double t = cta.top() + solo[i];
            cta.pop();
            cta.push(t);
            end = std::max(end, t);
        }
    return end;
}

// Cluster teams of a series batch that asks for none (team_ctas 0 or 1 is one CTA
// when given; 0 leaves it to the library): chains whose vectors do not fit one
// CTA's shared memory may run on 8 CTAs, as many of the largest as shorten the
// step.  Clocks per half iteration, measured (L = 6, Nt = 32 and L = 12, Nt = 64
// on one CTA: 12,900 and 104,000; the latter on 8 CTAs: 14,200): 5.6 a site, plus
// 2,500 for a team's exchange; iterations grow in proportion to Nt delta.
static void plan_series_teams(TcBatch* b, std::vector<char>& is_team) {
    constexpr int kTeam = 8, kSoloSites = 2048;
    const int n = b->n;
    std::vector<double> solo(n), team(n);
    std::vector<int> order(n), cand;
    for (int i = 0; i < n; ++i) {
        const hmc_params& p = b->ctxs[i]->params;
        if (p.team_ctas > 1) return;                 // the caller chose
        const double its = p.beta * p.n_md * (p.integrator == 1 ? 2 : 1);
        const double sites = b->ctxs[i]->view.N;
        solo[i] = its * (500.0 + 5.6 * sites);
        team[i] = its * (2500.0 + 5.6 * sites / kTeam);
        order[i] = i;
    }
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return solo[x] > solo[y]; });
    for (int i : order)
        if (b->ctxs[i]->params.team_ctas == 0 && b->ctxs[i]->view.N > kSoloSites &&
            b->ctxs[i]->params.Nt >= kTeam)
            cand.push_back(i);
    if (cand.empty()) return;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(b->ctxs[0]->num_sms / kTeam * kTeam);
    cfg.blockDim = dim3(b->threads);
    cfg.dynamicSmemBytes = b->smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kTeam;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, b->kernel, &cfg) != cudaSuccess ||
        clusters < 1) {
        (void)cudaGetLastError();
        return;
    }
    // without teams every SM takes one-CTA chains
    std::vector<char> none(n, 0);
    double best = series_makespan(solo, team, order, none, b->ctxs[0]->num_sms, 1);
    size_t best_k = 0;
    const size_t step = std::max<size_t>(1, cand.size() / 48);
    std::vector<char> flags(n, 0);
    for (size_t k = 0; k < cand.size();) {
        for (size_t q = 0; q < step && k < cand.size(); ++q) flags[cand[k++]] = 1;
        const double m = series_makespan(solo, team, order, flags, clusters, kTeam);
        if (m < best) {
            best = m;
            best_k = k;
        }
    }
    for (size_t k = 0; k < best_k; ++k) {
        is_team[cand[k]] = 1;
        b->ctxs[cand[k]]->params.team_ctas = kTeam;
    }
}

int tc_batch_create(const hmc_params* p, int n, TcBatch** out) {
    TcBatch* b = new TcBatch();
    b->n = n;
    int st = HMC_OK;
    // one context per chain (workspaces); chains with the same lattice,
    // delta*kappa and delta*mu share the first such context's E, its splits
    // and maps
    std::vector<int> leader(n);
    std::vector<int> map_slot(n);
    int n_maps = 0;
    for (int i = 0; i < n && st == HMC_OK; ++i) {
        if (p[i].precision != HMC_PREC_MIXED || p[i].operand_mode == 5) st = HMC_ERR_UNSUPPORTED;
        hmc_ctx* c = nullptr;
        if (st == HMC_OK) st = hmc_ctx_create(&p[i], &c);
        if (st != HMC_OK) break;
        b->ctxs.push_back(c);
        leader[i] = i;
        for (int j = 0; j < i; ++j)
            if (p[j].L == p[i].L &&
                p[j].beta / p[j].Nt * p[j].kappa == p[i].beta / p[i].Nt * p[i].kappa &&
                p[j].beta / p[j].Nt * p[j].mu == p[i].beta / p[i].Nt * p[i].mu) {
                leader[i] = leader[j];
                break;
            }
        map_slot[i] = (leader[i] == i) ? n_maps++ : map_slot[leader[i]];
    }
    if (st != HMC_OK) {
        tc_batch_destroy(b);
        return st;
    }
    b->series = true;
    for (hmc_ctx* c : b->ctxs)   // (a team's ring needs a slice on every CTA)
        b->series = b->series && series_chosen(c) && c->params.team_ctas <= c->params.Nt;
    b->kernel = (const void*)tc::k_batch;
    b->threads = tc::NTHR;
    b->smem = (unsigned)tc::kSmemBytes;
    if (b->series) {
        b->kernel = series_batch_kernel(&b->smem, &b->threads);
        if (!b->kernel) {
            tc_batch_destroy(b);
            return HMC_ERR_CUDA;
        }
    }
    std::vector<char> auto_team(n, 0);
    if (b->series) plan_series_teams(b, auto_team);
    std::vector<CUtensorMap> maps(4 * n_maps);
    for (int i = 0; i < n && !b->series; ++i)
        if (!b->ctxs[i]->tc && tc_tiles_init(b->ctxs[i]) != HMC_OK) {
            tc_batch_destroy(b);
            return HMC_ERR_CUDA;
        }
    for (int i = 0; i < n && !b->series; ++i)
        if (leader[i] == i) {
            maps[4 * map_slot[i]] = b->ctxs[i]->tc->map_hi;
            maps[4 * map_slot[i] + 1] = b->ctxs[i]->tc->map_lo;
            maps[4 * map_slot[i] + 2] = b->ctxs[i]->tc->map_whi;
            maps[4 * map_slot[i] + 3] = b->ctxs[i]->tc->map_wlo;
        }
    // chains asking for a team (team_ctas >= 2) run on a thread-block
    // cluster of that many CTAs; all such chains of a batch use one size
    for (int i = 0; i < n; ++i) {
        const int tmc = b->ctxs[i]->params.team_ctas;
        if (tmc <= 1) continue;
        if (tmc > tc::kMaxClusterW || (b->csize > 1 && tmc != b->csize)) {
            tc_batch_destroy(b);
            return HMC_ERR_UNSUPPORTED;
        }
        b->csize = tmc;
    }
    std::vector<tc::BatchItem> items(n);
    b->offsets.assign(n + 1, 0);
    std::vector<double> cost(n);
    for (int i = 0; i < n; ++i) {
        hmc_ctx* c = b->ctxs[i];
        const ChainView& lv = b->ctxs[leader[i]]->view;
        tc::BatchItem& it = items[i];
        it.v = c->view;
        it.v.E = lv.E;
        it.v.E_hi = lv.E_hi;
        it.v.E_lo = lv.E_lo;
        it.v.Ew_hi = lv.Ew_hi;
        it.v.Ew_lo = lv.Ew_lo;
        it.v.e_inv = lv.e_inv;
        it.team = c->params.team_ctas > 1 ? c->params.team_ctas : 1;
        it.pa.inner = 1;
        it.pa.cluster = 0;
        if (it.team > 1 && auto_team[i]) {
            it.pa = tc::PersistentArgs{};
            it.pa.inner = it.pa.cluster = it.team;
        } else if (it.team > 1) {
            // a cluster team: the launch shape of a single-chain run on
            // team CTAs with an inner team of all of them, as one cluster
            if (c->params.inner_ctas == 0) c->params.inner_ctas = it.team;
            it.pa = persistent_args(c, it.team, c->params.cg_tol, c->params.cg_max_iter);
            if (it.pa.inner != it.team || (it.pa.mode == tc::kSmall && it.pa.inner < 1)) {
                tc_batch_destroy(b);
                return HMC_ERR_UNSUPPORTED;
            }
            it.pa.cluster = it.team;
        } else {
            // one CTA per chain: E resident when the chain has one site block
            const int nti = it.v.Vr / tc::TM, nk = it.v.Vp / tc::KCH;
            const bool res = nti == 1 && nk <= tc::kMaxResidentChunks &&
                             c->params.operand_mode != 1;
            it.pa.mode = res ? tc::kResident : tc::kStreaming;
            it.pa.ns_tile = pick_ns(nti, it.v.Nt, 1);
            if (c->params.tile_slices > 0) it.pa.ns_tile = c->params.tile_slices;
            it.pa.vec_resident = 0;
            if (res) {
                it.pa.ns_tile = std::min(it.pa.ns_tile, 16);
                const size_t free_bytes = tc::kOperandBytes - (size_t)nk * tc::kAChunkBytes -
                                          tc::kMaxStages * tc::kBStageSmall;
                it.pa.vec_resident = 6 * sizeof(float2) * (size_t)it.v.N <= free_bytes;
            }
            // operand_mode 3: the CUDA-core solver on the chain's one CTA
            if (c->params.operand_mode == 3 && tc::small_feasible(it.v.V, it.v.Nt, 1)) {
                it.pa.mode = tc::kSmall;
                it.pa.vec_resident = 0;
            }
            it.pa.res_b = res_b_ok(it.v, it.pa.mode, it.pa.ns_tile, 1) ? 1 : 0;
            it.pa.wide_W = 0;
            // operand_mode 4: slice-major tiles, balanced slices of at most 64
            if (c->params.operand_mode == 4) {
                it.pa.mode = tc::kSlice;
                it.pa.wide_W = c->tc->w_cg;
                const int ntt = (it.v.Nt + tc::kWSlices - 1) / tc::kWSlices;
                it.pa.ns_tile = (it.v.Nt + ntt - 1) / ntt;
                if (c->params.tile_slices > 0) it.pa.ns_tile = c->params.tile_slices;
                it.pa.res_b = 0;
                it.pa.vec_resident = 0;
            }
        }
        if (it.team > 1) it.pa.res_b = 0;
        it.pa.tol = c->params.cg_tol;
        it.pa.max_iter = c->params.cg_max_iter;
        it.pa.ru_delta = c->params.ru_delta;
        it.pa.ru_every = c->params.ru_every;
        std::memset(&it.a, 0, sizeof(it.a));
        it.a.chain = (uint32_t)i;
        it.a.n_md = c->params.n_md;
        it.a.integrator = c->params.integrator;
        it.a.eps = c->params.traj_length / c->params.n_md;
        it.a.tol = c->params.cg_tol;
        it.a.max_iter = c->params.cg_max_iter;
        it.a.ru_delta = c->params.ru_delta;
        it.offset = b->offsets[i];
        b->offsets[i + 1] = b->offsets[i] + it.v.N;
        // cost proxy: tile work of one application times Nt (CG iterations
        // grow with beta = Nt * delta)
        // (series: the work per site does not depend on V)
        cost[i] = (b->series ? (double)it.v.V : (double)it.v.Vr * it.v.Vp) * it.v.Nt * it.v.Nt;
        if (b->series && it.team > 1) b->mail_V = std::max(b->mail_V, it.v.V);
    }
    std::vector<int> order(n);
    for (int i = 0; i < n; ++i) order[i] = i;
    // team chains first (the cluster phase of the kernel), then by cost
    std::stable_sort(order.begin(), order.end(), [&](int a, int c) {
        if ((items[a].team > 1) != (items[c].team > 1)) return items[a].team > 1;
        return cost[a] > cost[c];
    });
    bool ok = true;
    auto alloc = [&](void** ptr, size_t bytes) {
        if (ok && cudaMalloc(ptr, bytes) != cudaSuccess) ok = false;
    };
    alloc((void**)&b->d_maps, sizeof(CUtensorMap) * maps.size());
    alloc((void**)&b->d_items, sizeof(tc::BatchItem) * n);
    alloc((void**)&b->d_order, sizeof(int) * n);
    alloc((void**)&b->d_queue, sizeof(int));
    alloc((void**)&b->d_call, sizeof(tc::BatchCallArgs));
    alloc((void**)&b->d_outs, sizeof(double) * kNumScalars * n);
    if (ok && (cudaMallocHost((void**)&b->h_call, sizeof(tc::BatchCallArgs)) != cudaSuccess ||
               cudaMallocHost((void**)&b->h_outs, sizeof(double) * kNumScalars * n) !=
                   cudaSuccess))
        ok = false;
    if (ok) {
        for (int i = 0; i < n; ++i)
            items[i].maps = b->series ? nullptr : b->d_maps + 4 * map_slot[i];
        ok = cudaMemcpy(b->d_maps, maps.data(), sizeof(CUtensorMap) * maps.size(),
                        cudaMemcpyHostToDevice) == cudaSuccess &&
             cudaMemcpy(b->d_items, items.data(), sizeof(tc::BatchItem) * n,
                        cudaMemcpyHostToDevice) == cudaSuccess &&
             cudaMemcpy(b->d_order, order.data(), sizeof(int) * n, cudaMemcpyHostToDevice) ==
                 cudaSuccess &&
             cudaFuncSetAttribute(b->kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)b->smem) == cudaSuccess &&
             cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) == cudaSuccess &&
             cudaEventCreateWithFlags(&b->ready, cudaEventDisableTiming) == cudaSuccess;
    }
    int occ = 0;
    if (ok && (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, b->kernel, b->threads,
                                                             b->smem) != cudaSuccess ||
               occ < 1))
        ok = false;
    if (!ok) {
        tc_batch_destroy(b);
        return HMC_ERR_CUDA;
    }
    b->grid = std::min(n, b->ctxs[0]->num_sms * occ);
    if (b->csize > 1) {
        // whole clusters, as many as can be resident at once
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(b->ctxs[0]->num_sms / b->csize * b->csize);
        cfg.blockDim = dim3(b->threads);
        cfg.dynamicSmemBytes = b->smem;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)b->csize;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int nclus = 0;
        if (cudaOccupancyMaxActiveClusters(&nclus, b->kernel, &cfg) !=
                cudaSuccess ||
            nclus < 1) {
            (void)cudaGetLastError();
            tc_batch_destroy(b);
            return HMC_ERR_UNSUPPORTED;
        }
        b->grid = nclus * b->csize;
    }
    *out = b;
    return HMC_OK;
}

void tc_batch_offsets(const TcBatch* b, long long* off) {
    for (int i = 0; i <= b->n; ++i) off[i] = b->offsets[i];
}

int tc_batch_size(const TcBatch* b) { return b->n; }

// One trajectory of every chain: the launch is captured once into a CUDA
// graph on the batch's own stream (H2D of the call arguments from pinned
// memory, queue reset, the persistent kernel, D2H of the results) and
// replayed; it is ordered after the caller's stream by an event.
int tc_batch_trajectory(TcBatch* b, double* phi, uint64_t seed, uint64_t traj,
                        hmc_traj_out* out, cudaStream_t caller) {
    if (!b->exec || b->graph_phi != phi) {
        if (b->exec) cudaGraphExecDestroy(b->exec);
        if (b->graph) cudaGraphDestroy(b->graph);
        b->exec = nullptr;
        b->graph = nullptr;
        cudaStream_t s = b->stream;
        if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
            return HMC_ERR_CUDA;
        cudaMemcpyAsync(b->d_call, b->h_call, sizeof(tc::BatchCallArgs), cudaMemcpyHostToDevice, s);
        cudaMemsetAsync(b->d_queue, 0, sizeof(int), s);
        // (a chain that no CTA gets to, once every one of them has failed, reports
        // no solves instead of the last call's results)
        cudaMemsetAsync(b->d_outs, 0, sizeof(double) * kNumScalars * b->n, s);
        {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(b->grid);
            cfg.blockDim = dim3(b->threads);
            cfg.dynamicSmemBytes = b->smem;
            cfg.stream = s;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = (unsigned)b->csize;
            at[0].val.clusterDim.y = 1;
            at[0].val.clusterDim.z = 1;
            cfg.attrs = at;
            cfg.numAttrs = b->csize > 1 ? 1 : 0;
            const tc::BatchItem* ip = b->d_items;
            const int* op = b->d_order;
            int nn = b->n, cs = b->csize;
            int* qp = b->d_queue;
            const tc::BatchCallArgs* cp = b->d_call;
            double* outp = b->d_outs;
            int mv = b->mail_V;
            unsigned sb = b->smem;
            void* args[] = {&ip, &op, &nn, &qp, &cp, &outp, &cs, &mv, &sb};   // (the last two:
            cudaLaunchKernelExC(&cfg, b->kernel, args);                       // series only)
        }
        cudaMemcpyAsync(b->h_outs, b->d_outs, sizeof(double) * kNumScalars * b->n,
                        cudaMemcpyDeviceToHost, s);
        if (cudaStreamEndCapture(s, &b->graph) != cudaSuccess ||
            cudaGraphInstantiate(&b->exec, b->graph, 0) != cudaSuccess)
            return HMC_ERR_CUDA;
        b->graph_phi = phi;
    }
    b->h_call->seed = seed;
    b->h_call->traj = traj;
    b->h_call->phi = phi;
    if (cudaEventRecord(b->ready, caller) != cudaSuccess ||
        cudaStreamWaitEvent(b->stream, b->ready, 0) != cudaSuccess ||
        cudaGraphLaunch(b->exec, b->stream) != cudaSuccess ||
        cudaStreamSynchronize(b->stream) != cudaSuccess)
        return HMC_ERR_CUDA;
    int first_bad = HMC_OK;
    for (int i = 0; i < b->n; ++i) {
        const double* v = b->h_outs + (size_t)i * kNumScalars;
        hmc_traj_out& o = out[i];
        o.dH = v[kTrajDH];
        o.H0 = v[kTrajH0];
        o.H1 = v[kTrajH1];
        o.u = v[kTrajU];
        o.accept = (int)v[kTrajAccept];
        o.cg_iterations = (int)v[kTrajIters];
        o.cg_solves = (int)v[kTrajSolves];
        o.reliable_updates = (int)v[kTrajRU];
        o.max_true_residual = v[kTrajMaxRes];
        o.fp64_iterations = (int)v[kTrajFp64Iters];
        o.status = (int)v[kTrajStatus];
        if (o.cg_solves == 0 && o.status == HMC_OK) o.status = HMC_ERR_TIMEOUT;  // not run
        if (o.status != HMC_OK && first_bad == HMC_OK) first_bad = o.status;
    }
    return first_bad;
}

}  // namespace hmc
