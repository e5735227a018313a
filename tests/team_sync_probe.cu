// Kernels of test_gpu_team_sync.py: the team barrier and sums of common.cuh on
// their own, between CTAs whose warps arrive at different times.
#include "../paper_2210_06874_gb300/csrc/common.cuh"

namespace {

using namespace hmc;

__device__ Team probe_team(const ChainView& c, ClusterSync* cs, unsigned* gen, bool cluster) {
    if (threadIdx.x == 0) *gen = 0;
    Team tm;
    tm.rank = blockIdx.x;
    tm.size = gridDim.x;
    tm.status = c.status;
    tm.slots = c.slots;
    tm.gen = gen;
    tm.cs = nullptr;
    if (cluster) {
        cluster_sync_init(cs, gridDim.x);
        tm.cs = cs;
    }
    __syncthreads();
    return tm;
}

// `rounds` times: every warp but the first waits, each another time, and
// stores one word per thread; plain barrier; every thread reads the next
// CTA's words; plain barrier.  Counts the words that were not this round's.
__global__ void k_exchange(ChainView c, unsigned* data, int rounds, int cluster, int* bad) {
    __shared__ ClusterSync cs;
    __shared__ unsigned gen;
    Team tm = probe_team(c, &cs, &gen, cluster != 0);
    const int n = blockDim.x, warp = threadIdx.x >> 5;
    const unsigned* other = data + (size_t)((tm.rank + 1) % tm.size) * n;
    bool ok = true;
    for (int r = 1; ok && r <= rounds; ++r) {
        if (warp > 0) __nanosleep(1000u * (unsigned)((warp + r + tm.rank) % 8));
        data[(size_t)tm.rank * n + threadIdx.x] = (unsigned)r;
        if (!(ok = team_barrier(tm))) break;
        if (warp > 0) __nanosleep(1000u * (unsigned)((warp + r) % 5));
        if (other[threadIdx.x] != (unsigned)r) atomicAdd(bad, 1);
        double v[2] = {1.0, (double)threadIdx.x};
        if (!(ok = team_barrier(tm))) break;
        if (!(ok = team_sum<2>(tm, v))) break;
        if (v[0] != (double)tm.size * n || v[1] != 0.5 * tm.size * n * (n - 1.0))
            atomicAdd(bad, 1);
    }
    if (!ok) atomicAdd(bad, 1 << 20);
    if (cluster) cluster_barrier_all();
}

// One CTA sets the status word before its third sync: res[rank] = the syncs
// that succeeded before one failed (kind 0: plain barriers, 1: sums of three
// values, 2: FP32 sums).
__global__ void k_status(ChainView c, int setter, int kind, int* res) {
    __shared__ unsigned gen;
    Team tm = probe_team(c, nullptr, &gen, false);
    int good = 0;
    for (; good < 8; ++good) {
        if (good == 2 && tm.rank == setter && threadIdx.x == 0)
            set_status(tm.status, HMC_ERR_UNSUPPORTED);
        double v[3] = {1.0, 2.0, 3.0};
        float f = 0.f;
        const bool ok = kind == 0   ? team_barrier(tm)
                        : kind == 1 ? team_sum<3>(tm, v)
                                    : team_sum_f(tm, 1.f, f);
        if (!ok) break;
    }
    if (threadIdx.x == 0) res[tm.rank] = good;
}

// res[CTA] = what cluster_matches says of a launch in clusters of `size`.
__global__ void k_matches(int size, int* res) {
    if (threadIdx.x == 0) res[blockIdx.x] = cluster_matches(size) ? 1 : 0;
}

}  // namespace

extern "C" int probe_status(void* control, int* res, int grid, int threads, int setter, int kind) {
    ChainView c{};
    control_bind(&c, control);
    void* args[] = {&c, &setter, &kind, &res};
    cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_status, dim3(grid), dim3(threads),
                                                args, 0, nullptr);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    return (int)e;
}

extern "C" int probe_matches(int* res, int grid, int launched, int size) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(32);
    cudaLaunchAttribute a[1];
    a[0].id = cudaLaunchAttributeClusterDimension;
    a[0].val.clusterDim.x = (unsigned)launched;
    a[0].val.clusterDim.y = a[0].val.clusterDim.z = 1;
    cfg.attrs = a;
    cfg.numAttrs = launched > 0 ? 1 : 0;
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_matches, size, res);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    return (int)e;
}

// Control block (zeroed), words (zeroed) and counter are the caller's device memory.
extern "C" int probe_exchange(void* control, unsigned* data, int* bad, int grid, int threads,
                              int rounds, int cluster) {
    ChainView c{};
    control_bind(&c, control);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cudaLaunchAttribute a[1];
    if (cluster) {
        a[0].id = cudaLaunchAttributeClusterDimension;
        a[0].val.clusterDim.x = (unsigned)grid;
        a[0].val.clusterDim.y = a[0].val.clusterDim.z = 1;
        if (grid > 8 && cudaFuncSetAttribute((const void*)k_exchange,
                                             cudaFuncAttributeNonPortableClusterSizeAllowed,
                                             1) != cudaSuccess)
            return (int)cudaGetLastError();
    } else {
        a[0].id = cudaLaunchAttributeCooperative;
        a[0].val.cooperative = 1;
    }
    cfg.attrs = a;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_exchange, c, data, rounds, cluster, bad);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    return (int)e;
}

extern "C" unsigned long long probe_control_bytes() { return kControlBytes; }
