// series_cg.cuh -- FP32 iterations of the mixed CG with E as a polynomial of
// the sparse hopping (series.h).
//
// E acts within a time slice, so each CTA owns a contiguous range of slices and
// hops them in its shared memory: per site and degree two additions and one
// multiply-add per component (degree 6 at delta kappa = 1/8) instead of the V
// multiply-adds of the dense product.  At L = 24 that is 7 MFLOP per
// application against 0.51 GFLOP, and no V x V operand moves at all.
//
// Operator: (M u)_t = u_t - s_t E D_{t-1} u_{t-1},
// (M^dag u)_t = u_t - s_{t+1} D_t^* E u_{t+1}, s_0 = -1, D_t = diag e^{i phi_t}.
//
// A half iteration is
//   epilogue -> post the partial norm -> hop the own slices -> send the result
//   of the boundary slice to its target's owner -> wait for the norms and the
//   neighbour's slice -> scalars.
// The hops depend only on r (M^dag: E p' = E r + beta E p, with E p carried per
// target slice as G) or on q (M), which are final before beta and alpha are
// known, so the hops run while the norms travel.  What travels is tagged with
// the half iteration's sequence number inside each 64-bit word {fp32, number}:
// the receiver polls the data itself, one hop through L2 (or, for a team that
// is one cluster, through distributed shared memory) with no fence and no
// flag.  One buffer per kind suffices: a CTA sends its next message of a kind
// only after an all-to-all sum that every CTA posts after reading this one.
//
// What bounds it: latency and instruction issue of one CTA per SM.  Measured
// clocks of a half iteration at L = 24, Nt = 96 (96 CTAs of one slice, 608
// threads): contraction 5,100, wait for the neighbour and the norm 2,000,
// epilogue 900, norm and scalars 600; at L = 6, Nt = 32 (a cluster of 16)
// 2,600, 900, 470 and 490.  One CG iteration, tensor-core tiles -> here: L = 24
// 41 us (split-K tiles 20) -> 8; L = 12, Nt = 64 20 -> 4.8 (64 CTAs; 6.4 on one
// cluster); L = 6, Nt = 32 19 -> 3.8-4.0.
#pragma once

#include "cg_scalars.cuh"
#include "fp64_path.cuh"

namespace hmc {
namespace ser {

constexpr int kWorkers = 608;        // most threads with cells (19 warps: L = 24's 576 cells)
constexpr int kThreads = 640;        // ... and the service warp
constexpr int kMaxTeamCtas = 160;    // norm slots read per team: 5 per lane

__host__ __device__ inline int t_lo(int rank, int Nt, int T) {
    return (int)((long long)rank * Nt / T);
}
__host__ __device__ inline int max_slices(int Nt, int T) { return (Nt + T - 1) / T; }

// Geometry of a team of T CTAs: one cell (both sublattices) per thread while the
// CTA has at most 608, else two, in blocks of whole slices.
struct Shape {
    int S;        // most slices of any CTA
    int N;        // cells per thread and block
    int SB;       // slices per block
    int workers;  // threads with cells
};
// (A team of one CTA takes all workers whatever the size, as the CTAs of a batch
// do: the same sums bit for bit.)
__host__ __device__ inline Shape shape(int L, int Nt, int T) {
    Shape s;
    const int LL = L * L;
    s.S = max_slices(Nt, T);
    s.N = s.S * LL <= kWorkers ? 1 : 2;
    const int fit = s.N * kWorkers / LL;
    s.SB = fit < s.S ? fit : s.S;
    const int need = (s.SB * LL + s.N - 1) / s.N;
    s.workers = T == 1 || s.SB < s.S ? kWorkers : (need + 31) / 32 * 32;
    return s;
}

// Dynamic shared memory: [cluster mail: 2 kinds x mail_V x 16 bytes] [hop
// buffers: 2 x SB LL float4] [Z and the vectors that fit: S LL float4 each].
// Everything here is stored by cells, {A site, B site} as one float4.
__host__ __device__ inline size_t mail_bytes(int mail_V) { return 2 * (size_t)mail_V * 16; }
__host__ __device__ inline size_t hop_bytes(int V, const Shape& s) {
    return (size_t)s.SB * V * sizeof(float4);
}

// ---------------------------------------------------------------- mail
__device__ __forceinline__ uint64_t tagged(float v, unsigned seq) {
    return ((uint64_t)seq << 32) | __float_as_uint(v);
}
__device__ __forceinline__ uint32_t peer(uint32_t addr, int rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
    return a;
}

struct Link {
    int T, rank;
    bool cluster;
    // mail boxes of this CTA's receivers and its own, per kind: cell c's two
    // 16-byte words at 32 c (shared-memory addresses in a cluster, else global)
    uint32_t to_s[2], own_s[2];
    uint64_t *to_g[2], *own_g[2];
    uint64_t* norm;    // [2 kinds][T] every 16 words (global) or [2][16] (own shared memory)

    // msg: [2 kinds][T][V] x 2 words (global) or [2][mail_V] x 2 (shared memory)
    __device__ __forceinline__ void init(const Team& tm, int V, int mail_V, uint64_t* msg,
                                         uint64_t* nrm) {
        T = tm.size;
        rank = tm.rank;
        cluster = tm.cs != nullptr;
        norm = nrm;
        const int dst[2] = {rank == 0 ? T - 1 : rank - 1, rank == T - 1 ? 0 : rank + 1};
        for (int k = 0; k < 2; ++k) {
            if (cluster) {
                own_s[k] = cta_smem_u32(msg) + 16u * (uint32_t)(k * mail_V);
                to_s[k] = peer(own_s[k], dst[k]);
            } else {
                own_g[k] = msg + 2 * ((size_t)k * T + rank) * V;
                to_g[k] = msg + 2 * ((size_t)k * T + dst[k]) * V;
            }
        }
    }
    // cell c of a boundary slice to its target's owner (kind 0: the previous CTA,
    // 1: the next)
    __device__ __forceinline__ void send(int kind, int c, float4 v, unsigned seq) const {
        const uint64_t a = tagged(v.x, seq), b = tagged(v.y, seq);
        const uint64_t d = tagged(v.z, seq), e = tagged(v.w, seq);
        if (cluster) {
            const uint32_t p = to_s[kind] + 32u * (uint32_t)c;
            asm volatile("st.relaxed.cluster.shared::cluster.v2.u64 [%0], {%1, %2};\n\t"
                         "st.relaxed.cluster.shared::cluster.v2.u64 [%0 + 16], {%3, %4};" ::"r"(p),
                         "l"(a), "l"(b), "l"(d), "l"(e)
                         : "memory");
        } else {
            asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};\n\t"
                         "st.relaxed.gpu.global.v2.u64 [%0 + 16], {%3, %4};" ::"l"(
                             to_g[kind] + 4 * (size_t)c),
                         "l"(a), "l"(b), "l"(d), "l"(e)
                         : "memory");
        }
    }
    __device__ __forceinline__ bool peek(int kind, int c, unsigned seq, float4& v) const {
        uint64_t a, b, d, e;
        if (cluster)
            asm volatile("ld.relaxed.cluster.shared::cta.v2.u64 {%0, %1}, [%4];\n\t"
                         "ld.relaxed.cluster.shared::cta.v2.u64 {%2, %3}, [%4 + 16];"
                         : "=l"(a), "=l"(b), "=l"(d), "=l"(e)
                         : "r"(own_s[kind] + 32u * (uint32_t)c)
                         : "memory");
        else
            asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%4];\n\t"
                         "ld.relaxed.gpu.global.v2.u64 {%2, %3}, [%4 + 16];"
                         : "=l"(a), "=l"(b), "=l"(d), "=l"(e)
                         : "l"(own_g[kind] + 4 * (size_t)c)
                         : "memory");
        v = make_float4(__uint_as_float((uint32_t)a), __uint_as_float((uint32_t)b),
                        __uint_as_float((uint32_t)d), __uint_as_float((uint32_t)e));
        return (unsigned)(a >> 32) == seq && (unsigned)(b >> 32) == seq &&
               (unsigned)(d >> 32) == seq && (unsigned)(e >> 32) == seq;
    }
    // warp 0: the CTA's sum to every member
    __device__ __forceinline__ void post(int kind, float v, unsigned seq) const {
        const int lane = threadIdx.x & 31;
        const uint64_t w = tagged(v, seq);
        if (cluster) {
            if (lane < T)
                asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(
                                 peer(cta_smem_u32(norm + kind * 16 + rank), lane)),
                             "l"(w)
                             : "memory");
        } else if (lane == 0) {
            asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(
                             norm + ((size_t)kind * T + rank) * 16),
                         "l"(w)
                         : "memory");
        }
    }
    __device__ __forceinline__ uint64_t peek_norm(int kind, int r) const {
        uint64_t w;
        if (cluster)
            asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];"
                         : "=l"(w)
                         : "r"(cta_smem_u32(norm + kind * 16 + r))
                         : "memory");
        else
            asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];"
                         : "=l"(w)
                         : "l"(norm + ((size_t)kind * T + r) * 16)
                         : "memory");
        return w;
    }
};

// Bounded polling: true when the time limit or the team's status says to stop.
struct Patience {
    unsigned n = 0;
    uint64_t t0 = 0;
    __device__ __forceinline__ bool out(int* status) {
        if ((++n & 255u) != 0) return false;
        if (t0 == 0) t0 = global_ns();
        if (*((volatile int*)status) != 0) return true;
        if (global_ns() - t0 > wait_limit_ns(status)) {
            set_status(status, HMC_ERR_TIMEOUT);
            return true;
        }
        return false;
    }
};

// Warp 0: the team's sum of the values posted under seq, added in a fixed
// order (lane r, r + 32, ..., then a shuffle tree); valid on every lane.
__device__ __forceinline__ bool wait_norm(const Link& lk, int* status, int kind, unsigned seq,
                                          float& sum) {
    const int lane = threadIdx.x & 31;
    constexpr int kPer = kMaxTeamCtas / 32;
    uint64_t w[kPer];
    Patience pt;
    bool ok = true;
    for (;;) {
        bool all = true;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int r = lane + 32 * i;
            w[i] = (uint64_t)seq << 32;
            if (r < lk.T) w[i] = lk.peek_norm(kind, r);
            all = all && (unsigned)(w[i] >> 32) == seq;
        }
        if (__all_sync(0xffffffffu, all || !ok)) break;
        if (ok && !all && pt.out(status)) ok = false;
    }
    float a = 0.f;
#pragma unroll
    for (int i = 0; i < kPer; ++i)
        if (32 * i < lk.T) a += __uint_as_float((uint32_t)w[i]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
    sum = __shfl_sync(0xffffffffu, a, 0);
    return __all_sync(0xffffffffu, ok);
}

// ---------------------------------------------------------------- hops
// A thread's cells of a block of slices (cell tid + j threads), and the six cells
// around each: (m1 +- 1, m2), (m1, m2 +- 1), (m1 - 1, m2 + 1), (m1 + 1, m2 - 1).
template <int N>
struct Cells {
    int n, nthr;            // cells of the block, worker threads
    int s[N];               // slice in the block
    int nb[N][6];
    __device__ __forceinline__ bool has(int j) const {
        return (int)threadIdx.x < nthr && (int)threadIdx.x + j * nthr < n;
    }
    __device__ __forceinline__ int cell(int j) const { return (int)threadIdx.x + j * nthr; }
    __device__ __forceinline__ void init(int L, int SB, int threads) {
        const int LL = L * L;
        n = SB * LL;
        nthr = threads;
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const int e = cell(j);
            s[j] = e / LL;
            const int b = s[j] * LL, m1 = (e - b) / L, m2 = (e - b) - m1 * L;
            const int p1 = b + (m1 == L - 1 ? 0 : m1 + 1) * L;
            const int q1 = b + (m1 == 0 ? L - 1 : m1 - 1) * L, r0 = b + m1 * L;
            const int p2 = m2 == L - 1 ? 0 : m2 + 1, q2 = m2 == 0 ? L - 1 : m2 - 1;
            nb[j][0] = p1 + m2;
            nb[j][1] = q1 + m2;
            nb[j][2] = r0 + p2;
            nb[j][3] = r0 + q2;
            nb[j][4] = q1 + p2;
            nb[j][5] = p1 + q2;
        }
    }
};

__device__ __forceinline__ float4 add4(float4 a, float4 b) {
    return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}
__device__ __forceinline__ float4 axpy4(float a, float4 x, float4 y) {
    return make_float4(fmaf(a, x.x, y.x), fmaf(a, x.y, y.y), fmaf(a, x.z, y.z),
                       fmaf(a, x.w, y.w));
}

// v <- E v / c0 on the block's cells (v.xy the A site, v.zw the B site), two
// degrees per barrier:
//     y <- v + r_{k-1} h (v + r_k h y) = (v + r_{k-1} h v) + r_{k-1} r_k h^2 y.
// h^2 = 3 + the six cells around, the same ones for either sublattice, so a
// neighbour is one 16-byte load; h v needs four of the twelve sites that the
// first gather reads anyway.  A phase is a store, a barrier and six loads: 112
// bytes of shared memory per cell for two degrees, and half the barriers and
// round trips of one degree at a time (which at one cell per thread took 590
// clocks per degree at L = 24, most of it latency).
// The two buffers alternate, also from call to call (par), so one barrier per
// phase suffices.  first() runs on every thread after the first barrier.
template <int N, class First>
__device__ __forceinline__ void hop(const float* ratio, int K, const Cells<N>& cl, float4* buf,
                                    int stride, int& par, float4 (&v)[N], First&& first) {
    float4 y[N], hv[N];
    bool on[N];
#pragma unroll
    for (int j = 0; j < N; ++j) {
        on[j] = cl.has(j);
        y[j] = v[j];
    }
    int k = K;
    bool head = true;
    do {
        float4* const b = buf + (par ? stride : 0);
        par ^= 1;
        // the pair of degrees of this phase (odd K: the first phase does degree K alone)
        const bool two = !head || (K & 1) == 0;
        const float r1 = k >= 1 ? ratio[two && k >= 2 ? k - 2 : k - 1] : 0.f;
        const float r2 = two && k >= 2 ? r1 * ratio[k - 1] : 0.f;
#pragma unroll
        for (int j = 0; j < N; ++j)
            if (on[j]) b[cl.cell(j)] = y[j];
        __syncthreads();
        if (head) first();
#pragma unroll
        for (int j = 0; j < N; ++j)
            if (on[j]) {
                const float4 u0 = b[cl.nb[j][0]], u1 = b[cl.nb[j][1]], u2 = b[cl.nb[j][2]];
                const float4 u3 = b[cl.nb[j][3]], u4 = b[cl.nb[j][4]], u5 = b[cl.nb[j][5]];
                if (head)
                    hv[j] = make_float4(v[j].z + u1.z + u3.z, v[j].w + u1.w + u3.w,
                                        v[j].x + u0.x + u2.x, v[j].y + u0.y + u2.y);
                const float4 h2 = axpy4(3.f, y[j], add4(add4(add4(u0, u1), add4(u2, u3)),
                                                        add4(u4, u5)));
                y[j] = axpy4(r2, h2, axpy4(r1, hv[j], v[j]));
            }
        k -= two ? 2 : 1;
        head = false;
    } while (k >= 1);
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = y[j];
}

// c * v (conj: conj(c) * v) of both sites of a cell
template <bool CONJ>
__device__ __forceinline__ float4 phase4(float4 c, float4 v) {
    const float s = CONJ ? -1.f : 1.f;
    return make_float4(c.x * v.x - s * c.y * v.y, c.x * v.y + s * c.y * v.x,
                       c.z * v.z - s * c.w * v.w, c.z * v.w + s * c.w * v.z);
}
__device__ __forceinline__ float norm4(float4 v, float acc) {
    return fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, acc))));
}

// Where the CG vectors of the CTA's slices live.
enum Store : int {
    kShared = 0,   // shared memory
    kAny = 1       // shared memory as far as it goes, then global memory
};

// Cell at A site a of a field in the natural layout [Nt][V].
__device__ __forceinline__ float4 field_cell(const float2* m, size_t a, int LL) {
    const float2 x = m[a], y = m[a + LL];
    return make_float4(x.x, x.y, y.x, y.y);
}

extern __shared__ uint4 ser_dyn4[];   // 16-byte elements: the mail is read and written so
#define ser_dyn (reinterpret_cast<uint8_t*>(ser_dyn4))

// A CG vector by cells: an offset into the dynamic shared memory (so that the
// compiler sees shared-memory accesses), or any memory.
template <int ST>
struct Vec {
    uint32_t off;
    float4* m;
    __device__ __forceinline__ float4& operator[](int c) const {
        return (ST == kAny ? m : reinterpret_cast<float4*>(ser_dyn + off))[c];
    }
};

// Workspace of a launch.
struct Work {
    size_t bytes;          // of dynamic shared memory
    int mail_V;            // sites per mail box: the cluster's mail boxes come first (place and
                           // size are the launch's, so stale words keep old numbers)
    uint64_t* norm_smem;   // [2][16], static shared memory (cluster teams)
    unsigned* seq;         // static shared memory: last half iteration's number
};

// The loop invariants of a segment (shared memory).
struct Geo {
    int LL, Nt, S, t0, SB, stride, K, it_end, max_iter;
    bool alone;
    float c0, rmax, stop, ru2;
    size_t g0;      // first element of the own slices in [Nt][V]
    int* status;
    Link lk;
};

// Vectors besides Z that a CTA keeps in memory.
constexpr int kVecs = 6;
__host__ __device__ inline size_t shared_bytes(int V, int mail_V, const Shape& s, int vecs) {
    return mail_bytes(mail_V) + hop_bytes(V, s) + (size_t)vecs * s.S * V * sizeof(float2);
}

// FP32 CG iterations of one segment (until a reliable update, max_iter or a
// non-finite norm).  r is loaded from c.r_f (or, refresh, the FP64 residual),
// p and G from c.p_f and c.g_f, which also receive them; the increment x starts
// at zero and is folded into x64 at the end.  Returns the end reason, -1 if a
// bounded wait failed.
//
// The last warp has no cells: between the same barriers as the others it adds
// the warps' sums, posts the CTA's norm during the first hop and collects the
// team's while the others wait for the boundary slice, so the norm's trip is off
// their path.  Every thread then derives the same scalars from the same total
// (one thread that did so for all of them cost 700 clocks a half iteration).
template <int ST, int N>
__device__ __noinline__ int segment(const ChainView& c, const Team tm, const Work& wk,
                                    const Shape sh, tc::CgScalars& s_cg, bool refresh,
                                    int max_iter, double2* x64) {
    if (cta_smem_u32(ser_dyn) & 15u) {   // (the mail's 16-byte accesses)
        set_status(tm.status, HMC_ERR_UNSUPPORTED);
        return -1;
    }
    // What the loop needs and never changes lives in shared memory: a spilled
    // pointer costs a trip to L2 per use (the dynamic shared memory leaves next to
    // no L1), and with the geometry in registers the L = 24 trajectory took 85
    // instead of 70 ms.
    __shared__ Geo g;
    __shared__ float s_w[kWorkers / 32];
    __shared__ float s_sum, s_ratio[kSerMax32];
    if (threadIdx.x == 0) {
        g.LL = c.V / 2;
        g.Nt = c.Nt;
        g.alone = tm.size == 1;
        g.t0 = t_lo(tm.rank, c.Nt, tm.size);
        g.S = t_lo(tm.rank + 1, c.Nt, tm.size) - g.t0;
        g.SB = min(sh.SB, g.S);
        g.stride = sh.SB * g.LL;
        g.g0 = (size_t)g.t0 * c.V;
        g.K = c.ser.k32;
        g.c0 = c.ser.c0f;
        g.rmax = s_cg.rmax;
        g.stop = s_cg.stop;
        g.ru2 = s_cg.ru2;
        g.it_end = s_cg.it0 + s_cg.every;
        g.max_iter = max_iter;
        g.status = tm.status;
        if (tm.cs)
            g.lk.init(tm, c.V, wk.mail_V, reinterpret_cast<uint64_t*>(ser_dyn), wk.norm_smem);
        else
            g.lk.init(tm, c.V, 0, c.ser_mail, c.ser_norm);
    }
    if (threadIdx.x < kSerMax32) s_ratio[threadIdx.x] = c.ser.r32[threadIdx.x];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nww = (blockDim.x >> 5) - 1;
    // the iteration's scalars, the same on every thread
    float rr = s_cg.rr, alpha = 0.f, beta = s_cg.beta;
    int it = s_cg.it, reason = tc::kSegMaxIter;
    unsigned seq = *wk.seq;
    bool have_rr = false, failed = false;
    __syncthreads();
    // after the half iteration's barrier: the new |r|^2 / |q|^2 (true: segment ends)
    auto after_r = [&]() {
        const float n = s_sum;
        ++it;
        if (!isfinite(n)) reason = tc::kSegNonfinite;
        else if (n <= g.stop || n <= g.ru2 * g.rmax || it >= g.it_end) reason = tc::kSegUpdate;
        else {
            beta = n / rr;
            rr = n;
            return it >= g.max_iter;
        }
        return true;
    };
    auto after_q = [&]() {
        const float n = s_sum;
        if (!isfinite(n) || !(n > 0.f)) {
            reason = tc::kSegNonfinite;
            return true;
        }
        alpha = rr / n;
        return false;
    };
    uint32_t top = (uint32_t)mail_bytes(wk.mail_V);
    float4* const hopbuf = reinterpret_cast<float4*>(ser_dyn + top);
    top += (uint32_t)hop_bytes(c.V, sh);
    const uint32_t vec = (uint32_t)(sh.S * c.V * sizeof(float2));   // (of one that fits)
    Vec<ST> r, p, G, q, cis, x, Z;
    auto take = [&](auto& v, float2* fallback) {
        if (ST != kAny || vector_fits(top, sh.S, c.V, wk.bytes)) {
            v.off = top;
            v.m = reinterpret_cast<float4*>(ser_dyn + top);
            top += vec;
        } else {
            v.m = reinterpret_cast<float4*>(fallback + g.g0);
        }
    };
    take(Z, c.u_f);
    take(r, c.p2_f);     // (c.r_f and c.cis_f hold the inputs in the natural layout)
    take(q, c.q_f);
    take(p, c.p_f);
    take(cis, c.rh_f);
    take(G, c.g_f);
    take(x, c.x_f);
    Cells<N> cl;
    cl.init(c.L, g.SB, blockDim.x - 32);
    int par = 0;
    // f(c, slice) for each of this thread's cells c of the CTA's slices
    auto each = [&](auto&& f) {
        for (int b = 0; b < g.S; b += g.SB) {
            cl.n = min(g.SB, g.S - b) * g.LL;
#pragma unroll
            for (int j = 0; j < N; ++j)
                if (cl.has(j)) f(cl.cell(j) + b * g.LL, b + cl.s[j]);
        }
    };
    float4* const keep_p = reinterpret_cast<float4*>(c.p_f + g.g0);
    float4* const keep_G = reinterpret_cast<float4*>(c.g_f + g.g0);
    each([&](int e, int s) {
        const size_t a = g.g0 + (size_t)e + (size_t)s * g.LL;   // A site in [Nt][V]
        float4 rv;
        if (refresh) {
            const double2 u = c.r[a], w = c.r[a + g.LL];
            rv = make_float4((float)u.x, (float)u.y, (float)w.x, (float)w.y);
        } else {
            rv = field_cell(c.r_f, a, g.LL);
        }
        r[e] = rv;
        p[e] = keep_p[e];
        G[e] = keep_G[e];
        cis[e] = field_cell(c.cis_f, a, g.LL);
        x[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    });
    __syncthreads();
    float own = 0.f;        // service warp: this CTA's sum of the pending norm
    // this warp's part of the norm
    auto give = [&](float acc) {
        if (warp == nww) return;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if (lane == 0) s_w[warp] = acc;
    };
    // E on every own slice of `src`; results to Z at their target slice or to
    // its owner (kind 0, M^dag: target t - 1; kind 1, M: target t + 1).  The
    // norm given before it is posted after the first barrier.
    auto contract = [&](int kind, bool norm, auto&& src) {
        for (int b = 0; b < g.S; b += g.SB) {
            cl.n = min(g.SB, g.S - b) * g.LL;
            float4 v[N];
#pragma unroll
            for (int j = 0; j < N; ++j)
                if (cl.has(j)) v[j] = src(cl.cell(j) + b * g.LL);
            hop<N>(s_ratio, g.K, cl, hopbuf, g.stride, par, v, [&]() {
                if (b != 0 || warp != nww || !norm) return;
                float a = lane < nww ? s_w[lane] : 0.f;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
                own = __shfl_sync(0xffffffffu, a, 0);
                if (!g.alone) g.lk.post(kind, own, seq);
            });
#pragma unroll
            for (int j = 0; j < N; ++j)
                if (cl.has(j)) {
                    const int e = cl.cell(j) + b * g.LL, s = b + cl.s[j];
                    const int last = (g.S - 1) * g.LL;
                    const bool edge = kind == 0 ? s == 0 : s == g.S - 1;
                    if (edge && !g.alone) g.lk.send(kind, kind == 0 ? e : e - last, v[j], seq);
                    else Z[kind == 0 ? (edge ? e + last : e - g.LL)
                                     : (edge ? e - last : e + g.LL)] = v[j];
                }
        }
    };
    // end of a half iteration: the neighbour's slice for the own boundary target
    // into Z, the team's norm into s_sum; false if a wait failed in the CTA
    auto finish = [&](int kind, bool norm) {
        bool ok = true;
        if (warp == nww) {
            if (norm) {
                float sum = own;
                if (!g.alone) ok = wait_norm(g.lk, g.status, kind, seq, sum);
                if (lane == 0) s_sum = sum;
            }
        } else if (!g.alone) {
            const int edge = kind == 0 ? g.S - 1 : 0;
            each([&](int e, int s) {
                if (s != edge) return;
                float4 z;
                Patience pt;
                while (!g.lk.peek(kind, e - edge * g.LL, seq, z))
                    if (!ok || pt.out(g.status)) { ok = false; break; }
                Z[e] = z;
            });
        }
        return __syncthreads_or(ok ? 0 : 1) == 0;
    };
    while (it < g.max_iter) {
        // ---- M^dag p' (p' = r + beta p): hop r
        if (!have_rr) ++seq;
        contract(0, have_rr, [&](int e) { return r[e]; });
        if (!finish(0, have_rr)) { failed = true; break; }
        if (have_rr && after_r()) break;
        float acc = 0.f;
        each([&](int e, int s) {
            const float4 pv = axpy4(beta, p[e], r[e]);
            const float4 gv = axpy4(beta, G[e], Z[e]);
            p[e] = pv;
            G[e] = gv;
            const float sg = g.t0 + s == g.Nt - 1 ? g.c0 : -g.c0;
            const float4 qv = axpy4(sg, phase4<true>(cis[e], gv), pv);
            q[e] = qv;
            acc = norm4(qv, acc);
        });
        ++seq;
        give(acc);
        // ---- M q: hop e^{i phi} q
        contract(1, true, [&](int e) { return phase4<false>(cis[e], q[e]); });
        if (!finish(1, true)) { failed = true; break; }
        if (after_q()) break;
        acc = 0.f;
        each([&](int e, int s) {
            const float sg = g.t0 + s == 0 ? g.c0 : -g.c0;
            const float4 ap = axpy4(sg, Z[e], q[e]);
            x[e] = axpy4(alpha, p[e], x[e]);
            const float4 rv = axpy4(-alpha, ap, r[e]);
            r[e] = rv;
            acc = norm4(rv, acc);
        });
        ++seq;
        have_rr = true;
        give(acc);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        *wk.seq = seq;
        s_cg.rr = rr;
        s_cg.beta = beta;
        s_cg.it = it;
    }
    if (!failed && reason != tc::kSegNonfinite)
        each([&](int e, int s) {
            const size_t a = g.g0 + (size_t)e + (size_t)s * g.LL;
            const float4 d = x[e];
            double2 u = x64[a], w = x64[a + g.LL];
            u.x += (double)d.x;
            u.y += (double)d.y;
            w.x += (double)d.z;
            w.y += (double)d.w;
            x64[a] = u;
            x64[a + g.LL] = w;
            keep_p[e] = p[e];
            keep_G[e] = G[e];
        });
    __syncthreads();
    return failed ? -1 : reason;
}

__device__ inline int run_segment(const ChainView& c, const Team& tm, const Work& wk,
                                  tc::CgScalars& s_cg, bool refresh, int max_iter,
                                  double2* x64) {
    const Shape sh = shape(c.L, c.Nt, tm.size);
    if (shared_bytes(c.V, wk.mail_V, sh, kVecs + 1) > wk.bytes)
        return segment<kAny, 2>(c, tm, wk, sh, s_cg, refresh, max_iter, x64);
    if (sh.N == 1)
        return segment<kShared, 1>(c, tm, wk, sh, s_cg, refresh, max_iter, x64);
    return segment<kShared, 2>(c, tm, wk, sh, s_cg, refresh, max_iter, x64);
}

}  // namespace ser
}  // namespace hmc
