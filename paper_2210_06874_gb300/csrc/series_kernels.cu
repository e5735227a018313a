// series_kernels.cu -- kernels of the mixed path with E as a polynomial of the
// sparse hopping (series_cg.cuh), and their launchers: the automatic choice of
// the mixed path wherever the series exists.
//
//  k_apply       one application of M or M^dag in FP32, one slice per block
//  k_cg          persistent mixed solve of (M M^dag) x = chi
//  k_trajectory  persistent mixed HMC trajectory
//  k_batch       one trajectory of every chain of a batch
#include <algorithm>

#include "mixed_path.cuh"
#include "tc_path.h"

namespace hmc {
namespace ser {

constexpr int kApplyThreads = 576;   // L = 24: one cell per thread

// Standalone application, target slice blockIdx.x: the source slice's phase is
// computed here, the slice hopped in shared memory (two buffers of V float2)
// and the result formed: the vector, phi and the output each move once.
template <bool DAG, int N>
__global__ void __launch_bounds__(kApplyThreads)
    k_apply(const __grid_constant__ ChainView c, const double* __restrict__ phi,
            const float2* __restrict__ in, float2* __restrict__ out) {
    const int V = c.V, LL = V / 2, Nt = c.Nt, t = blockIdx.x;
    const int ts = DAG ? (t + 1 == Nt ? 0 : t + 1) : (t == 0 ? Nt - 1 : t - 1);
    const float2* src = in + (size_t)ts * V;
    const size_t o = (size_t)t * V;
    const double* ph = phi + (DAG ? o : (size_t)ts * V);
    Cells<N> cl;
    cl.init(c.L, 1, blockDim.x);
    float4 v[N], cis[N], self[N];
#pragma unroll
    for (int j = 0; j < N; ++j)
        if (cl.has(j)) {
            const int a = cl.cell(j);
            v[j] = field_cell(src, a, LL);
            self[j] = field_cell(in + o, a, LL);
            float sa, ca, sb, cb;
            sincosf((float)ph[a], &sa, &ca);
            sincosf((float)ph[a + LL], &sb, &cb);
            cis[j] = make_float4(ca, sa, cb, sb);
            if (!DAG) v[j] = phase4<false>(cis[j], v[j]);
        }
    int par = 0;
    hop<N>(c.ser.r32, c.ser.k32, cl, reinterpret_cast<float4*>(ser_dyn), LL, par, v, [] {});
    const float c0 = c.ser.c0f, sg = (DAG ? t == Nt - 1 : t == 0) ? c0 : -c0;
#pragma unroll
    for (int j = 0; j < N; ++j)
        if (cl.has(j)) {
            const int a = cl.cell(j);
            const float4 w = axpy4(sg, DAG ? phase4<true>(cis[j], v[j]) : v[j], self[j]);
            out[o + a] = make_float2(w.x, w.y);
            out[o + a + LL] = make_float2(w.z, w.w);
        }
}

// Per-launch set-up of a persistent kernel's team and workspace: the cluster's
// mail boxes cleared before any member can write to them, or the sequence number
// taken up where the context's last launch left it.
struct Launch {
    int cluster;        // the grid is one cluster of this many CTAs (0: global team)
    unsigned smem;      // dynamic shared memory in bytes
};
__device__ __forceinline__ bool begin(const ChainView& c, const Launch& la, ClusterSync* cs,
                                      uint64_t* norm, unsigned* seq, Work& wk, Team& tm) {
    tm = tc::make_team(c);
    wk.bytes = la.smem;
    wk.mail_V = la.cluster ? c.V : 0;
    wk.norm_smem = norm;
    wk.seq = seq;
    if (threadIdx.x == 0) *seq = series_first(la.cluster != 0, *c.ser_seq) +
                                    (blockIdx.x == 0 ? (unsigned)c.misnumber : 0u);
    if (la.cluster) {
        uint64_t* m = reinterpret_cast<uint64_t*>(ser_dyn);
        for (int i = threadIdx.x; i < (int)(mail_bytes(c.V) / 8); i += blockDim.x) m[i] = 0;
        if (threadIdx.x < 32) norm[threadIdx.x] = 0;
        if (threadIdx.x == 0 &&
            !(cluster_matches(la.cluster) && gridDim.x == (unsigned)la.cluster))
            set_status(c.status, HMC_ERR_UNSUPPORTED);
        __syncthreads();
        cluster_sync_init(cs, la.cluster);
        if (__syncthreads_or(threadIdx.x == 0 && team_failed(tm))) return false;
        tm.cs = cs;
    }
    __syncthreads();
    return true;
}
// No member leaves while others may still write to it; the context's next launch
// with its mail in global memory starts past every number any CTA can have used.
__device__ __forceinline__ void end(const ChainView& c, const Launch& la, const Work& wk) {
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0) *c.ser_seq = *wk.seq + 16u;
    if (la.cluster) cluster_barrier_all();
}

#define HMC_SER_BEGIN()                                                                   \
    __shared__ f64::Smem sm64;                                                            \
    __shared__ ClusterSync s_cs;                                                          \
    __shared__ uint64_t s_norm[32];                                                       \
    __shared__ unsigned s_seq;                                                            \
    Work wk;                                                                              \
    Team tm;                                                                              \
    if (!begin(c, la, &s_cs, s_norm, &s_seq, wk, tm)) return;                             \
    tc::TcState st;                                                                       \
    st.ser = &wk

__global__ void __launch_bounds__(kThreads, 1)
    k_cg(const __grid_constant__ ChainView c, const __grid_constant__ tc::PersistentArgs pa,
         const Launch la, const double* phi, const double2* chi, double2* x) {
    HMC_SER_BEGIN();
    tc::set_phases(c, tm, phi);
    tc::MixedResult res{};
    bool ok = team_barrier(tm);
    if (ok)
        ok = tc::cg_mixed<tc::kKindSeries>(c, tm, st, sm64, nullptr, nullptr, pa, nullptr, chi, x,
                                           res);
    if (ok && tm.rank == 0 && threadIdx.x == 0) {
        c.scalars[0] = res.iterations;
        c.scalars[1] = res.true_res;
        c.scalars[2] = res.status;
        c.scalars[3] = res.reliable_updates;
        c.scalars[4] = res.fp64_iterations;
    }
    end(c, la, wk);
}

__global__ void __launch_bounds__(kThreads, 1)
    k_trajectory(const __grid_constant__ ChainView c,
                 const __grid_constant__ tc::PersistentArgs pa, const Launch la, TrajArgs a) {
    HMC_SER_BEGIN();
    tc::run_trajectory<tc::kKindSeries>(c, tm, st, sm64, nullptr, nullptr, pa, nullptr, a);
    end(c, la, wk);
}

// Batch of chains (see batch_loop): one CTA or one cluster of csize CTAs per
// chain at a time; mail boxes of mail_V sites, cleared once.
__device__ __noinline__ bool batch_traj(const tc::BatchItem& it, tc::TcState& st,
                                        f64::Smem& sm64, Team& tm, const TrajArgs& a) {
    return tc::run_trajectory<tc::kKindSeries>(it.v, tm, st, sm64, nullptr, nullptr, it.pa,
                                               nullptr, a);
}
__global__ void __launch_bounds__(kThreads, 1)
    k_batch(const tc::BatchItem* __restrict__ items, const int* __restrict__ order, int n,
            int* queue, const tc::BatchCallArgs* call, double* outs, int csize, int mail_V,
            unsigned smem) {
    __shared__ f64::Smem sm64;
    __shared__ ClusterSync s_cs;
    __shared__ uint64_t s_norm[32];
    __shared__ unsigned s_seq;
    Work wk{smem, mail_V, s_norm, &s_seq};
    if (threadIdx.x == 0) s_seq = 0;
    uint64_t* m = reinterpret_cast<uint64_t*>(ser_dyn);
    for (int i = threadIdx.x; i < (int)(mail_bytes(mail_V) / 8); i += blockDim.x) m[i] = 0;
    if (threadIdx.x < 32) s_norm[threadIdx.x] = 0;
    __syncthreads();
    if (csize > 1) cluster_sync_init(&s_cs, csize);
    tc::TcState st;
    st.ser = &wk;
    tc::batch_loop(items, order, n, queue, call, outs, csize, &s_cs,
                   [&](const tc::BatchItem& it, Team& tm, ClusterSync*, const TrajArgs& a) {
                       return batch_traj(it, st, sm64, tm, a);
                   });
    if (csize > 1) cluster_barrier_all();
}

}  // namespace ser

// ---------------------------------------------------------------- host side
const void* series_batch_kernel(unsigned* smem, int* threads) {
    *threads = ser::kThreads;
    const void* k = (const void*)ser::k_batch;
    int dev = 0, most = 0;
    cudaFuncAttributes at;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) !=
            cudaSuccess ||
        cudaFuncGetAttributes(&at, k) != cudaSuccess)
        return nullptr;
    *smem = (unsigned)(most - (int)at.sharedSizeBytes) & ~15u;
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)*smem) ==
                   cudaSuccess
               ? k
               : nullptr;
}

bool series_chosen(const hmc_ctx* c) {
    const hmc_params& p = c->params;
    return p.operand_mode == 0 && p.cluster_mode == 0 && c->view.ser.ok &&
           c->view.V <= f64::kHopDoubles && p.hb_inner == 0;
}

static int series_ctas(const ChainView& v, int num_sms) {
    return std::min(v.Nt, std::min(num_sms, ser::kMaxTeamCtas));
}

int series_ctx_init(hmc_ctx* c) {
    ChainView& v = c->view;
    if (!series_chosen(c)) return HMC_OK;
    const size_t T = series_ctas(v, c->num_sms);
    auto alloc = [&](size_t bytes) -> void* {
        void* p = nullptr;
        if (c->n_allocs >= (int)(sizeof(c->allocs) / sizeof(c->allocs[0])) ||
            cudaMalloc(&p, bytes) != cudaSuccess)
            return nullptr;
        c->allocs[c->n_allocs++] = p;
        cudaMemset(p, 0, bytes);
        return p;
    };
    // [mail][norms][sequence number]
    const size_t mail = 2 * T * v.V * 16, norms = 2 * T * 128;
    unsigned char* p = (unsigned char*)alloc(mail + norms + 16);
    if (!p) return HMC_ERR_CUDA;
    v.ser_mail = (uint64_t*)p;
    v.ser_norm = (uint64_t*)(p + mail);
    v.ser_seq = (unsigned*)(p + mail + norms);
    int most = 0;
    if (cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device) !=
        cudaSuccess)
        return HMC_ERR_CUDA;
    for (const void* k : {(const void*)ser::k_cg, (const void*)ser::k_trajectory}) {
        cudaFuncAttributes at;
        if (cudaFuncGetAttributes(&at, k) != cudaSuccess ||
            cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 most - (int)at.sharedSizeBytes) != cudaSuccess)
            return HMC_ERR_CUDA;
        // teams of up to 16 CTAs as one cluster (beyond the portable 8); a
        // device that refuses it gets a global-memory team
        if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
            cudaSuccess)
            (void)cudaGetLastError();
    }
    return HMC_OK;
}

int series_apply(const ChainView& v, const double* phi, const float2* in, float2* out, bool dag,
                 cudaStream_t s) {
    const int LL = v.V / 2;
    const bool two = LL > ser::kApplyThreads;
    const int thr = ((two ? (LL + 1) / 2 : LL) + 31) / 32 * 32;
    const size_t smem = 2 * (size_t)v.V * sizeof(float2);
    if (dag && two) ser::k_apply<true, 2><<<v.Nt, thr, smem, s>>>(v, phi, in, out);
    else if (dag) ser::k_apply<true, 1><<<v.Nt, thr, smem, s>>>(v, phi, in, out);
    else if (two) ser::k_apply<false, 2><<<v.Nt, thr, smem, s>>>(v, phi, in, out);
    else ser::k_apply<false, 1><<<v.Nt, thr, smem, s>>>(v, phi, in, out);
    return cudaGetLastError() == cudaSuccess ? HMC_OK : HMC_ERR_CUDA;
}

// Launch a persistent series kernel: as one thread-block cluster where that is the
// quicker (series_on_cluster), else as a cooperative launch with global mail.
static int launch_series(hmc_ctx* c, const void* fn, tc::PersistentArgs& pa, ser::Launch& la,
                         void** args, cudaStream_t s) {
    const ChainView& v = c->view;
    int most = series_ctas(v, c->num_sms);
    if (c->params.team_ctas > 0) most = std::min(most, c->params.team_ctas);
    if (c->params.inner_ctas > 0) most = std::min(most, c->params.inner_ctas);
    int T = most;
    bool cluster = series_on_cluster(v.V / 2, v.Nt, most) && v.team_pad == 0;
    if (cluster) T = std::min(most, kSerCluster);
    for (;;) {
        la.cluster = cluster ? T : 0;
        pa.inner = T;
        pa.cluster = 0;
        const ser::Shape sh = ser::shape(v.L, v.Nt, T);
        cudaFuncAttributes at;
        if (cudaFuncGetAttributes(&at, fn) != cudaSuccess) return HMC_ERR_CUDA;
        const size_t want = ser::shared_bytes(v.V, cluster ? v.V : 0, sh, ser::kVecs + 1);
        la.smem = (unsigned)std::min(want, (size_t)at.maxDynamicSharedSizeBytes);
        if (!control_reset(v, T, s)) return HMC_ERR_CUDA;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(T);
        cfg.blockDim = dim3(sh.workers + 32);   // the service warp
        cfg.dynamicSmemBytes = la.smem;
        cfg.stream = s;
        cudaLaunchAttribute a[1];
        if (cluster) {
            a[0].id = cudaLaunchAttributeClusterDimension;
            a[0].val.clusterDim.x = (unsigned)T;
            a[0].val.clusterDim.y = 1;
            a[0].val.clusterDim.z = 1;
        } else {
            a[0].id = cudaLaunchAttributeCooperative;
            a[0].val.cooperative = 1;
        }
        cfg.attrs = a;
        cfg.numAttrs = 1;
        if (cudaLaunchKernelExC(&cfg, fn, args) == cudaSuccess) return HMC_OK;
        (void)cudaGetLastError();   // a refused configuration is not sticky
        if (!cluster) return HMC_ERR_CUDA;
        cluster = false;
        T = most;
    }
}

static tc::PersistentArgs series_args(const hmc_ctx* c, double tol, int max_iter) {
    tc::PersistentArgs pa{};
    pa.tol = tol;
    pa.max_iter = max_iter;
    pa.ru_delta = c->params.ru_delta;
    pa.ru_every = c->params.ru_every;
    return pa;
}

int series_cg(hmc_ctx* c, const double* phi, const double2* chi, double2* x, double tol,
              int max_iter, cudaStream_t s) {
    tc::PersistentArgs pa = series_args(c, tol, max_iter);
    ser::Launch la{};
    ChainView v = c->view;
    void* args[] = {&v, &pa, &la, &phi, &chi, &x};
    return launch_series(c, (const void*)ser::k_cg, pa, la, args, s);
}

int series_trajectory(hmc_ctx* c, const TrajArgs& a, cudaStream_t s) {
    tc::PersistentArgs pa = series_args(c, a.tol, a.max_iter);
    ser::Launch la{};
    ChainView v = c->view;
    TrajArgs av = a;
    void* args[] = {&v, &pa, &la, &av};
    return launch_series(c, (const void*)ser::k_trajectory, pa, la, args, s);
}

}  // namespace hmc
