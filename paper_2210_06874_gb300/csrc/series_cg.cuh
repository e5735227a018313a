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
// What bounds it: latency.  A half iteration at L = 24, Nt = 96 (one slice per
// CTA, 288 threads) is six hops of ~190 clocks (shared-memory bandwidth: 80
// bytes per cell and hop) and two trips through L2.
#pragma once

#include "cg_scalars.cuh"
#include "fp64_path.cuh"

namespace hmc {
namespace ser {

constexpr int kThreads = 512;        // most threads per CTA
constexpr int kMaxTeamCtas = 160;    // norm slots read per team: 5 per lane
constexpr int kMaxCells = 4;         // cells per thread and block of slices

__host__ __device__ inline int t_lo(int rank, int Nt, int T) {
    return (int)((long long)rank * Nt / T);
}
__host__ __device__ inline int max_slices(int Nt, int T) { return (Nt + T - 1) / T; }

// Geometry of a team of T CTAs of nthr threads.
struct Shape {
    int S;        // most slices of any CTA
    int N;        // cells per thread (1, 2 or kMaxCells)
    int reg;      // vectors in registers (one block of slices, N <= 2)
    int SB;       // slices per block
};
__host__ __device__ inline Shape shape(int L, int Nt, int T, int nthr) {
    Shape s;
    const int LL = L * L;
    s.S = max_slices(Nt, T);
    const int cells = s.S * LL;
    s.reg = cells <= 2 * nthr;
    s.N = cells <= nthr ? 1 : cells <= 2 * nthr ? 2 : kMaxCells;
    const int fit = s.N * nthr / LL;
    s.SB = s.reg ? s.S : (fit < s.S ? fit : s.S);
    return s;
}
// Threads for that team: one cell per thread up to 512 cells, else two.  A team
// of one CTA takes all 512, as the CTAs of a batch do: the same sums bit for bit.
__host__ __device__ inline int threads(int L, int Nt, int T) {
    if (T == 1) return kThreads;
    const int cells = max_slices(Nt, T) * L * L;
    const int want = cells <= kThreads ? cells : cells <= 2 * kThreads ? (cells + 1) / 2 : kThreads;
    return want <= 32 ? 32 : (want + 31) / 32 * 32;
}

// Dynamic shared memory: [cluster mail: 2 kinds x mail_V x 16 bytes] [hop
// buffers: 2 x SB V float2] [Z: S V float2] [vectors that fit, S V float2 each].
__host__ __device__ inline size_t mail_bytes(int mail_V) { return 2 * (size_t)mail_V * 16; }
__host__ __device__ inline size_t hop_bytes(int V, const Shape& s) {
    return 2 * (size_t)s.SB * V * sizeof(float2);
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
    int T, rank, prev, next;
    int V;             // sites of a mail box
    bool cluster;
    uint64_t* msg;     // [2 kinds][T][V] x 2 words (global) or [2][V] x 2 (own shared memory)
    uint64_t* norm;    // [2 kinds][T] every 16 words (global) or [2][16] (own shared memory)

    // value of site `site` of a boundary slice to CTA dst
    __device__ __forceinline__ void send(int kind, int dst, int site, float2 v,
                                         unsigned seq) const {
        const uint64_t a = tagged(v.x, seq), b = tagged(v.y, seq);
        if (cluster) {
            const uint32_t p = peer(cta_smem_u32(msg + 2 * ((size_t)kind * V + site)), dst);
            asm volatile("st.relaxed.cluster.shared::cluster.v2.u64 [%0], {%1, %2};" ::"r"(p),
                         "l"(a), "l"(b)
                         : "memory");
        } else {
            asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(
                             msg + 2 * (((size_t)kind * T + dst) * V + site)),
                         "l"(a), "l"(b)
                         : "memory");
        }
    }
    __device__ __forceinline__ bool peek(int kind, int site, unsigned seq, float2& v) const {
        uint64_t a, b;
        if (cluster)
            asm volatile("ld.relaxed.cluster.shared::cta.v2.u64 {%0, %1}, [%2];"
                         : "=l"(a), "=l"(b)
                         : "r"(cta_smem_u32(msg + 2 * ((size_t)kind * V + site)))
                         : "memory");
        else
            asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];"
                         : "=l"(a), "=l"(b)
                         : "l"(msg + 2 * (((size_t)kind * T + rank) * V + site))
                         : "memory");
        v = make_float2(__uint_as_float((uint32_t)a), __uint_as_float((uint32_t)b));
        return (unsigned)(a >> 32) == seq && (unsigned)(b >> 32) == seq;
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
    __device__ __forceinline__ bool out(const Team& tm) {
        if ((++n & 255u) != 0) return false;
        if (t0 == 0) t0 = global_ns();
        if (team_failed(tm)) return true;
        if (global_ns() - t0 > wait_limit_ns(tm.status)) {
            set_status(tm.status, HMC_ERR_TIMEOUT);
            return true;
        }
        return false;
    }
};

// Warp 0: the team's sum of the values posted under seq, added in a fixed
// order (lane r, r + 32, ..., then a shuffle tree); valid on every lane.
__device__ __forceinline__ bool wait_norm(const Link& lk, const Team& tm, int kind, unsigned seq,
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
        if (ok && !all && pt.out(tm)) ok = false;
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
// A thread's cells of a block of slices, in the natural layout [slice][V].
template <int N>
struct Cells {
    int n;                                       // cells of the block
    int a[N], s[N];                              // A site's index; slice in the block
    int bm1[N], bm2[N], ap1[N], ap2[N];          // neighbours outside the cell
    __device__ __forceinline__ bool has(int j) const {
        return (int)(threadIdx.x + j * blockDim.x) < n;
    }
    __device__ __forceinline__ void init(int L, int ns) {
        const int LL = L * L, V = 2 * LL;
        n = ns * LL;
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const int cell = threadIdx.x + j * blockDim.x;
            s[j] = cell / LL;
            const int cc = cell - s[j] * LL, m1 = cc / L, m2 = cc - m1 * L;
            const int A = s[j] * V, B = A + LL;
            a[j] = A + cc;
            bm1[j] = B + (m1 == 0 ? L - 1 : m1 - 1) * L + m2;
            bm2[j] = B + m1 * L + (m2 == 0 ? L - 1 : m2 - 1);
            ap1[j] = A + (m1 == L - 1 ? 0 : m1 + 1) * L + m2;
            ap2[j] = A + m1 * L + (m2 == L - 1 ? 0 : m2 + 1);
        }
    }
};

// v <- E v / c0 on the block's cells (v.xy the A site, v.zw the B site).  The
// two buffers alternate, also from call to call (par), so one barrier per
// degree suffices.
template <int N>
__device__ __forceinline__ void hop(const float* ratio, int K, const Cells<N>& cl, int LL,
                                    float2* buf, int stride, int& par, float4 (&v)[N]) {
    float4 y[N];
#pragma unroll
    for (int j = 0; j < N; ++j) y[j] = v[j];
    for (int k = K; k >= 1; --k) {
        float2* b = buf + (par ? stride : 0);
        par ^= 1;
        const float r = ratio[k - 1];
#pragma unroll
        for (int j = 0; j < N; ++j)
            if (cl.has(j)) {
                b[cl.a[j]] = make_float2(y[j].x, y[j].y);
                b[cl.a[j] + LL] = make_float2(y[j].z, y[j].w);
            }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < N; ++j)
            if (cl.has(j)) {
                const float2 b1 = b[cl.bm1[j]], b2 = b[cl.bm2[j]];
                const float2 a1 = b[cl.ap1[j]], a2 = b[cl.ap2[j]];
                const float4 s = make_float4(y[j].z + b1.x + b2.x, y[j].w + b1.y + b2.y,
                                             y[j].x + a1.x + a2.x, y[j].y + a1.y + a2.y);
                y[j] = make_float4(fmaf(r, s.x, v[j].x), fmaf(r, s.y, v[j].y),
                                   fmaf(r, s.z, v[j].z), fmaf(r, s.w, v[j].w));
            }
    }
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = y[j];
}

__device__ __forceinline__ float4 axpy4(float a, float4 x, float4 y) {
    return make_float4(fmaf(a, x.x, y.x), fmaf(a, x.y, y.y), fmaf(a, x.z, y.z),
                       fmaf(a, x.w, y.w));
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

// A CG vector of the CTA's slices: registers, or memory [S][V] float2.
template <bool REG, int N>
struct Vec {
    float4 v[REG ? N : 1];
    float2* m;
    __device__ __forceinline__ float4 get(int j, int a, int LL) const {
        if constexpr (REG) return v[j];
        const float2 x = m[a], y = m[a + LL];
        return make_float4(x.x, x.y, y.x, y.y);
    }
    __device__ __forceinline__ void set(int j, int a, int LL, float4 w) {
        if constexpr (REG) {
            v[j] = w;
        } else {
            m[a] = make_float2(w.x, w.y);
            m[a + LL] = make_float2(w.z, w.w);
        }
    }
};

// Workspace of a launch.
struct Work {
    uint8_t* smem;         // dynamic shared memory: the cluster's mail boxes first (their
    size_t bytes;          // place and size are the launch's, so stale words keep old numbers)
    int mail_V;            // sites per mail box
    uint64_t* norm_smem;   // [2][16], static shared memory (cluster teams)
    float* ratio;          // static shared memory [kSerMax32]
    unsigned* seq;         // static shared memory: last half iteration's number
};

// FP32 CG iterations of one segment (until a reliable update, max_iter or a
// non-finite norm).  r is loaded from c.r_f (or, refresh, the FP64 residual),
// p and G from c.p_f and c.g_f, which also receive them; the increment x starts
// at zero and is folded into x64 at the end.  Returns the end reason, -1 if a
// bounded wait failed.
template <bool REG, int N>
__device__ __noinline__ int segment(const ChainView& c, const Team tm, const Work& wk,
                                    const Shape sh, tc::CgScalars& s_cg, bool refresh,
                                    int max_iter, double2* x64, float hop_scale) {
    const int V = c.V, LL = V / 2, Nt = c.Nt, T = tm.size;
    const int t0 = t_lo(tm.rank, Nt, T), S = t_lo(tm.rank + 1, Nt, T) - t0;
    const size_t g0 = (size_t)t0 * V;
    Link lk;
    lk.T = T;
    lk.rank = tm.rank;
    lk.prev = tm.rank == 0 ? T - 1 : tm.rank - 1;
    lk.next = tm.rank == T - 1 ? 0 : tm.rank + 1;
    lk.cluster = tm.cs != nullptr;
    lk.V = lk.cluster ? wk.mail_V : V;
    lk.msg = lk.cluster ? reinterpret_cast<uint64_t*>(wk.smem) : c.ser_mail;
    lk.norm = lk.cluster ? wk.norm_smem : c.ser_norm;
    const bool alone = T == 1;
    // shared memory
    const int SB = min(sh.SB, S), stride = sh.SB * V;
    uint8_t* top = wk.smem + mail_bytes(wk.mail_V);
    float2* hopbuf = reinterpret_cast<float2*>(top);
    top += hop_bytes(V, sh);
    const size_t vec = (size_t)sh.S * V * sizeof(float2);
    auto take = [&](float2* fallback) {
        if (top + vec <= wk.smem + wk.bytes) {
            float2* p = reinterpret_cast<float2*>(top);
            top += vec;
            return p;
        }
        return fallback + g0;
    };
    float2* Z = take(c.u_f);
    Vec<REG, N> r, p, G, q, cis, x;
    if constexpr (!REG) {
        r.m = take(c.r_f);
        q.m = take(c.q_f);
        p.m = take(c.p_f);
        cis.m = take(c.cis_f);
        G.m = take(c.g_f);
        x.m = take(c.x_f);
    }
    Cells<N> cl;
    cl.init(c.L, SB);
    const int K = c.ser.k32;
    if ((int)threadIdx.x < K) wk.ratio[threadIdx.x] = c.ser.r32[threadIdx.x];
    const float c0 = c.ser.c0f * hop_scale;
    // f(j, a, slice) for each of this thread's cells of every block of slices
    auto each = [&](auto&& f) {
        for (int b = 0; b < S; b += SB) {
            const int nb = min(SB, S - b);
            cl.n = nb * LL;
#pragma unroll
            for (int j = 0; j < N; ++j)
                if (cl.has(j)) f(j, cl.a[j] + b * V, b + cl.s[j]);
            if (REG) break;
        }
    };
    auto load = [&](const float2* g, int a) {
        const float2 u = g[g0 + a], w = g[g0 + a + LL];
        return make_float4(u.x, u.y, w.x, w.y);
    };
    each([&](int j, int a, int) {
        float4 rv;
        if (refresh) {
            const double2 u = c.r[g0 + a], w = c.r[g0 + a + LL];
            rv = make_float4((float)u.x, (float)u.y, (float)w.x, (float)w.y);
        } else {
            rv = load(c.r_f, a);
        }
        r.set(j, a, LL, rv);
        p.set(j, a, LL, load(c.p_f, a));
        G.set(j, a, LL, load(c.g_f, a));
        cis.set(j, a, LL, load(c.cis_f, a));
        x.set(j, a, LL, make_float4(0.f, 0.f, 0.f, 0.f));
    });
    __shared__ float s_w[kThreads / 32];
    __shared__ float s_sum;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    unsigned seq = *wk.seq;
    int par = 0;
    float own = 0.f;        // warp 0: this CTA's sum of the pending norm
    // the CTA's norm: posted by warp 0 (kind 0: |r|^2, 1: |q|^2)
    auto post = [&](int kind, float acc) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if (lane == 0) s_w[warp] = acc;
        __syncthreads();
        if (warp == 0) {
            float a = lane < nw ? s_w[lane] : 0.f;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
            own = __shfl_sync(0xffffffffu, a, 0);
            if (!alone) lk.post(kind, own, seq);
        }
    };
    // E on every own slice of `src`; results to Z at their target slice or to
    // its owner (kind 0, M^dag: target t - 1; kind 1, M: target t + 1)
    auto contract = [&](int kind, auto&& src) {
        for (int b = 0; b < S; b += SB) {
            cl.n = min(SB, S - b) * LL;
            float4 v[N];
#pragma unroll
            for (int j = 0; j < N; ++j)
                if (cl.has(j)) v[j] = src(j, cl.a[j] + b * V);
            hop<N>(wk.ratio, K, cl, LL, hopbuf, stride, par, v);
#pragma unroll
            for (int j = 0; j < N; ++j)
                if (cl.has(j)) {
                    const int a = cl.a[j] + b * V, s = b + cl.s[j];
                    const float2 vA = make_float2(v[j].x, v[j].y), vB = make_float2(v[j].z, v[j].w);
                    const bool edge = kind == 0 ? s == 0 : s == S - 1;
                    if (edge && !alone) {
                        const int site = a - s * V, dst = kind == 0 ? lk.prev : lk.next;
                        lk.send(kind, dst, site, vA, seq);
                        lk.send(kind, dst, site + LL, vB, seq);
                    } else {
                        const int to = kind == 0 ? (s == 0 ? a + (S - 1) * V : a - V)
                                                 : (s == S - 1 ? a - (S - 1) * V : a + V);
                        Z[to] = vA;
                        Z[to + LL] = vB;
                    }
                }
            if (REG) break;
        }
        if (K == 0) __syncthreads();   // (kappa = 0: the hops had no barrier)
    };
    // the neighbour's slice for the own boundary target into Z
    auto receive = [&](int kind) {
        if (alone) return true;
        bool ok = true;
        each([&](int, int a, int s) {
            if (s != (kind == 0 ? S - 1 : 0)) return;
            const int site = a - s * V;
            float2 vA, vB;
            Patience pt;
            for (;;) {
                const bool ra = lk.peek(kind, site, seq, vA), rb = lk.peek(kind, site + LL, seq, vB);
                if (ra && rb) break;
                if (!ok || pt.out(tm)) { ok = false; break; }
            }
            Z[a] = vA;
            Z[a + LL] = vB;
        });
        return ok;
    };
    // end of a half iteration: the team's norm to thread 0's update, which every
    // thread sees after the barrier; false if a wait failed anywhere in the CTA
    auto finish = [&](int kind, bool ok, bool have, auto&& update) {
        if (warp == 0 && have) {
            float sum = own;
            if (!alone) ok = wait_norm(lk, tm, kind, seq, sum) && ok;
            if (lane == 0) {
                s_sum = sum;
                update(sum);
            }
        }
        return __syncthreads_or(ok ? 0 : 1) == 0;
    };
    __syncthreads();
    int reason = tc::kSegMaxIter;
    bool have_rr = false, failed = false;
    while (s_cg.it < max_iter) {
        // ---- M^dag p' (p' = r + beta p): hop r
        if (!have_rr) ++seq;
        contract(0, [&](int j, int a) { return r.get(j, a, LL); });
        bool ok = receive(0);
        if (!finish(0, ok, have_rr, [&](float rr) {
                tc::cg_after_r(s_cg, rr);
                if (s_cg.reason == 0 && s_cg.it >= max_iter) s_cg.reason = tc::kSegMaxIter;
            })) {
            failed = true;
            break;
        }
        if (have_rr && s_cg.reason != 0) { reason = s_cg.reason; break; }
        const float beta = s_cg.beta;
        float acc = 0.f;
        each([&](int j, int a, int s) {
            const float4 z = Vec<false, N>{{}, Z}.get(0, a, LL);
            const float4 pv = axpy4(beta, p.get(j, a, LL), r.get(j, a, LL));
            const float4 gv = axpy4(beta, G.get(j, a, LL), z);
            p.set(j, a, LL, pv);
            G.set(j, a, LL, gv);
            const float sg = t0 + s == Nt - 1 ? c0 : -c0;
            const float4 qv = axpy4(sg, phase4<true>(cis.get(j, a, LL), gv), pv);
            q.set(j, a, LL, qv);
            acc = norm4(qv, acc);
        });
        ++seq;
        post(1, acc);
        // ---- M q: hop e^{i phi} q
        contract(1, [&](int j, int a) {
            return phase4<false>(cis.get(j, a, LL), q.get(j, a, LL));
        });
        ok = receive(1);
        if (!finish(1, ok, true, [&](float qq) { tc::cg_after_q(s_cg, qq); })) {
            failed = true;
            break;
        }
        if (s_cg.reason != 0) { reason = s_cg.reason; break; }
        const float alpha = s_cg.alpha;
        acc = 0.f;
        each([&](int j, int a, int s) {
            const float4 z = Vec<false, N>{{}, Z}.get(0, a, LL);
            const float sg = t0 + s == 0 ? c0 : -c0;
            const float4 ap = axpy4(sg, z, q.get(j, a, LL));
            x.set(j, a, LL, axpy4(alpha, p.get(j, a, LL), x.get(j, a, LL)));
            const float4 rv = axpy4(-alpha, ap, r.get(j, a, LL));
            r.set(j, a, LL, rv);
            acc = norm4(rv, acc);
        });
        ++seq;
        post(0, acc);
        have_rr = true;
    }
    __syncthreads();
    if (threadIdx.x == 0) *wk.seq = seq;
    if (failed) return -1;
    if (reason != tc::kSegNonfinite)
        each([&](int j, int a, int) {
            const float4 d = x.get(j, a, LL), pv = p.get(j, a, LL), gv = G.get(j, a, LL);
            double2 u = x64[g0 + a], w = x64[g0 + a + LL];
            u.x += (double)d.x;
            u.y += (double)d.y;
            w.x += (double)d.z;
            w.y += (double)d.w;
            x64[g0 + a] = u;
            x64[g0 + a + LL] = w;
            Vec<false, 1> pg{{}, c.p_f + g0}, gg{{}, c.g_f + g0};
            pg.set(0, a, LL, pv);
            gg.set(0, a, LL, gv);
        });
    __syncthreads();
    return reason;
}

__device__ inline int run_segment(const ChainView& c, const Team& tm, const Work& wk,
                                  tc::CgScalars& s_cg, bool refresh, int max_iter, double2* x64,
                                  float hop_scale) {
    const Shape sh = shape(c.L, c.Nt, tm.size, blockDim.x);
    if (sh.reg && sh.N == 1)
        return segment<true, 1>(c, tm, wk, sh, s_cg, refresh, max_iter, x64, hop_scale);
    if (sh.reg)
        return segment<true, 2>(c, tm, wk, sh, s_cg, refresh, max_iter, x64, hop_scale);
    return segment<false, kMaxCells>(c, tm, wk, sh, s_cg, refresh, max_iter, x64, hop_scale);
}

}  // namespace ser
}  // namespace hmc
