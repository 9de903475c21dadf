// DOCH steps with the stopping rule of Remark S2 for one CSR instance with short rows:
//   x^(k+1) = T(x^k),  r^(k) = ||x^(k+1) - x^k||_2 / ||x^k||_2 per replica; a replica stops at the
//   first k with r^(k) < eps and keeps x^(k+1).
//
// One launch per step. Its row blocks form x^(k+1) as csr_step_pipe_kernel does (the same sums in the
// same order) and the sums of r^(k) from the values they hold; its first blocks decide r^(k-1) from
// the sums that launch k - 1 left, one warp per replica, so that no launch waits for a reduction.
// A stopped replica is no longer written. The decision of step k - 1 falls while launch k writes
// x^(k+1) over x^(k-1), in the buffer that does not hold x^k: a replica that stops there keeps x^k in
// buffer k mod 2, and later launches leave it alone. until_finish collects the buffers.
//
// Sums: per thread compensated FP32 of split products for FP32 iterates, merged across a block's
// threads with the rounding of every merge kept (relative error below 2^-44 of these positive sums; an
// FP64 operation holds an SM partition for 64 clocks a warp, and widening each warp's eight sums took
// as long as the step), and across blocks; FP64 throughout for FP64 iterates.
//
// Bound by the latency of the gathers, as the step. 100,000 spins of degree 3, R = 8, FP32, 200 steps:
// 5.5 ms with four launches per step (step, norms, decision, copy), 1.5 ms so; 2000 spins of degree 8,
// R = 3: 2.1 -> 0.54 ms.
#include <algorithm>
#include <cmath>

#include "csr_pipe.cuh"
#include "hamsum.cuh"
#include "internal.cuh"

namespace doch {
namespace {

constexpr int kUThreads = 256;
constexpr int kUWarps = kUThreads / 32;
constexpr int kUBatch = 4;  // entries of a row's first batch, loaded one row ahead

// resident blocks per SM that the kernel is compiled for: FP32 sums take 16 registers more than the step
// (four blocks spill: 2.40 -> 3.38 ms for the steps above when measured), FP64 steps gain from a third block (0.95 -> 0.86 ms
// for 12,000 spins, R = 16)
constexpr int kUBlocksPerSm = 3;

// a block's sum as it is left for the next launch, and sums of them
template <typename XT>
struct UntilSum;
template <>
struct UntilSum<float> {
    using Slot = float2;
    DotSum32 v;
    __device__ __forceinline__ void merge(Slot o) { v.merge(o.x, o.y); }
    __device__ __forceinline__ void merge_lane(int o) { merge(from_lane(o)); }
    __device__ __forceinline__ Slot from_lane(int o) const {
        return make_float2(__shfl_xor_sync(0xffffffffu, v.s, o), __shfl_xor_sync(0xffffffffu, v.c, o));
    }
    __device__ __forceinline__ Slot slot() const { return make_float2(v.s, v.c); }
    __device__ __forceinline__ float near() const { return v.s; }
    __device__ __forceinline__ double value() const { return v.value(); }
};
template <>
struct UntilSum<double> {
    using Slot = double;
    double v = 0.0;
    __device__ __forceinline__ void merge(Slot o) { v += o; }
    __device__ __forceinline__ void merge_lane(int o) { merge(from_lane(o)); }
    __device__ __forceinline__ Slot from_lane(int o) const { return __shfl_xor_sync(0xffffffffu, v, o); }
    __device__ __forceinline__ Slot slot() const { return v; }
    __device__ __forceinline__ float near() const { return static_cast<float>(v); }
    __device__ __forceinline__ double value() const { return v; }
};

// r < eps for r = sqrt(d) / sqrt(s), without FP64 where FP32 squares already tell (FP64 operations that
// wait for one another take about 150 clocks each, and every step waits for the slowest block)
template <typename XT>
__device__ __forceinline__ bool below(const UntilSum<XT> &d, const UntilSum<XT> &s, double eps) {
    const float e = static_cast<float>(eps), lim = e * e * s.near();
    if (e > 1e-15f && lim > 1e-30f && lim < 1e30f) {
        if (d.near() > 1.0001f * lim) return false;
        if (d.near() < 0.9999f * lim) return true;
    }
    return sqrt(d.value()) / sqrt(s.value()) < eps;
}

// step k of pair t, whole warp: part[2 t + m][blocks] added in a fixed order
template <typename XT>
__device__ void until_decide(const typename UntilSum<XT>::Slot *__restrict__ part, int blocks, double eps, int k, int t,
                             int *running, int32_t *__restrict__ steps, int *n_running) {
    const int lane = threadIdx.x & 31;
    const typename UntilSum<XT>::Slot *p = part + static_cast<int64_t>(t) * 2 * blocks;
    UntilSum<XT> d, s;
    constexpr int kAhead = 8;  // loads in flight
    for (int b = lane; b < blocks; b += 32 * kAhead) {
        typename UntilSum<XT>::Slot vd[kAhead], vs[kAhead];
#pragma unroll
        for (int e = 0; e < kAhead; ++e)
            if (b + 32 * e < blocks) {
                vd[e] = __ldcg(p + b + 32 * e);
                vs[e] = __ldcg(p + blocks + b + 32 * e);
            }
#pragma unroll
        for (int e = 0; e < kAhead; ++e)
            if (b + 32 * e < blocks) {
                d.merge(vd[e]);
                s.merge(vs[e]);
            }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        d.merge_lane(o);
        s.merge_lane(o);
    }
    if (lane != 0 || !__ldcg(running + t) || !below<XT>(d, s, eps)) return;
    steps[t] = k + 1;
    __stcg(running + t, 0);
    atomicSub(n_running, 1);
}

__device__ __forceinline__ void until_report(UntilProgress *p, int k, int call, bool done) {
    asm volatile("st.volatile.global.v2.u32 [%0], {%1, %2};" ::"l"(p), "r"(k), "r"(call << 1 | (done ? 1 : 0)) : "memory");
}

// ldv_cg that stays where it is written: before the test of the running flags
template <typename T, int V>
__device__ __forceinline__ void ldv_now(const T *p, T (&v)[V]) {
    if constexpr (sizeof(T) * V == 16) {
        uint32_t w[4];
        asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
                     : "l"(p));
#pragma unroll
        for (int k = 0; k < V; ++k) {
            if constexpr (sizeof(T) == 4) v[k] = __uint_as_float(w[k]);
            else v[k] = __hiloint2double(static_cast<int>(w[2 * k + 1]), static_cast<int>(w[2 * k]));
        }
    } else if constexpr (sizeof(T) * V == 8) {
        uint32_t w[2];
        asm volatile("ld.global.cg.v2.u32 {%0, %1}, [%2];" : "=r"(w[0]), "=r"(w[1]) : "l"(p));
        if constexpr (V == 2) {
            v[0] = __uint_as_float(w[0]);
            v[1] = __uint_as_float(w[1]);
        } else {
            v[0] = __hiloint2double(static_cast<int>(w[1]), static_cast<int>(w[0]));
        }
    } else {
        uint32_t w;
        asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(w) : "l"(p));
        v[0] = __uint_as_float(w);
    }
}

// grid: dblocks deciding blocks, then row blocks. A row takes Cp threads: its C = R / V chunks, or C
// rounded up to a power of two (spare lanes idle), so that shuffles add the rows of a warp.
template <typename XT, typename VT, int V>
__global__ void __launch_bounds__(kUThreads, kUBlocksPerSm)
until_kernel(const XT *__restrict__ xi, XT *__restrict__ xo, const int64_t *__restrict__ row_ptr,
             const int32_t *__restrict__ col, const VT *__restrict__ val, const XT *__restrict__ h, int n, int R,
             StepValues<XT> par, int Cp, int dblocks, double eps, int k, typename UntilSum<XT>::Slot *__restrict__ part,
             const typename UntilSum<XT>::Slot *__restrict__ part_before, int *running, int32_t *__restrict__ steps,
             int *n_running, UntilProgress *progress, int call) {
    const int blocks = static_cast<int>(gridDim.x) - dblocks, blk = static_cast<int>(blockIdx.x) - dblocks;
    if (blk < 0) {
        pdl_wait();
        pdl_trigger();
        int t = static_cast<int>(blockIdx.x) * kUWarps + (threadIdx.x >> 5);
        pdl_after(t);
        if (k > 0 && t < R) until_decide<XT>(part_before, blocks, eps, k - 1, t, running, steps, n_running);
        __syncthreads();
        if (blockIdx.x == 0 && threadIdx.x == 0)  // for the host: launch k runs, and whether any replica still does
            until_report(progress, k, call, __ldcg(n_running) == 0);
        return;
    }
    const int C = R / V;
    const int rows_per_block = kUThreads / Cp;
    int ch = threadIdx.x % Cp;
    const int rl = threadIdx.x / Cp;
    const int S = blocks * rows_per_block;
    int i = rl < rows_per_block && ch < C ? blk * rows_per_block + rl : n;
    int e0, e1, f0, f1;  // entry ranges of rows i and i + S
    int32_t js[kUBatch];
    XT ws[kUBatch];
    pipe_row_range(row_ptr, i, n, e0, e1);
    pipe_row_range(row_ptr, i + S, n, f0, f1);
    pipe_first_batch<kUBatch>(col, val, e0, e1, js, ws);
    pdl_wait();  // the couplings above are never written
    pdl_trigger();
    pdl_after(ch);  // x and the flags
    const XT a = par.alpha;
    const StepRoot<XT> root(par);
    // a flag lowered during this launch may or may not be seen: this launch's writes miss x^k either way
    bool run[V], all = true, any = false;
    int flag[V];  // one load: all warps of the grid ask one L2 slice for this line (V loads a warp: 2 us a step)
#pragma unroll
    for (int q = 0; q < V; ++q) flag[q] = 0;
    if (ch < C) {
        if constexpr (V == 4) {
            const int4 w = __ldcg(reinterpret_cast<const int4 *>(running + ch * V));
            flag[0] = w.x;
            flag[1] = w.y;
            flag[2] = w.z;
            flag[3] = w.w;
        } else if constexpr (V == 2) {
            const int2 w = __ldcg(reinterpret_cast<const int2 *>(running + ch * V));
            flag[0] = w.x;
            flag[1] = w.y;
        } else {
            flag[0] = __ldcg(running + ch);
        }
    }
#pragma unroll
    for (int q = 0; q < V; ++q) {
        run[q] = flag[q] != 0;
        all = all && run[q];
        any = any || run[q];
    }
    DotSum32 d32[V], s32[V];
    double d64[V], s64[V];
#pragma unroll
    for (int q = 0; q < V; ++q) d64[q] = s64[q] = 0.0;
    for (; i < n; i += S) {
        const int cnt = e1 - e0 < kUBatch ? e1 - e0 : kUBatch;
        XT xv[kUBatch][V];
#pragma unroll
        for (int t = 0; t < kUBatch; ++t)
            if (t < cnt) ldv_now<XT, V>(xi + static_cast<int64_t>(js[t]) * R + ch * V, xv[t]);
        XT xs[V];
        ldv_now<XT, V>(xi + static_cast<int64_t>(i) * R + ch * V, xs);
        if (!any) break;  // (the loads above do not wait for the flags)
        const XT hi = h ? h[i] : XT(0);
        // the next row's first batch and the range of the row after it
        int32_t js2[kUBatch];
        XT ws2[kUBatch];
        pipe_first_batch<kUBatch>(col, val, f0, f1, js2, ws2);
        int g0, g1;
        pipe_row_range(row_ptr, i + 2 * S, n, g0, g1);
        XT acc[V];
#pragma unroll
        for (int q = 0; q < V; ++q) acc[q] = XT(0);
#pragma unroll
        for (int t = 0; t < kUBatch; ++t)
            if (t < cnt) {
#pragma unroll
                for (int q = 0; q < V; ++q) acc[q] += ws[t] * xv[t][q];
            }
#pragma unroll 4
        for (int e = e0 + kUBatch; e < e1; ++e) {  // entries past the first batch, in entry order
            const int64_t j = __ldg(col + e);
            const XT w = coupling<XT, VT>(__ldg(val + e));
            XT xr[V];
            ldv_now<XT, V>(xi + j * R + ch * V, xr);
#pragma unroll
            for (int q = 0; q < V; ++q) acc[q] += w * xr[q];
        }
        XT out[V];
#pragma unroll
        for (int q = 0; q < V; ++q) {
            out[q] = root(acc[q] + a * xs[q] + hi);
            const XT e = out[q] - xs[q];
            if constexpr (sizeof(XT) == 4) {
                d32[q].add(e, e);
                s32[q].add(xs[q], xs[q]);
            } else {
                d64[q] += e * e;
                s64[q] += xs[q] * xs[q];
            }
        }
        XT *to = xo + static_cast<int64_t>(i) * R + ch * V;
        if (all) {
            stv<XT, V>(to, out);
        } else {
#pragma unroll
            for (int q = 0; q < V; ++q)
                if (run[q]) to[q] = out[q];
        }
        e0 = f0;
        e1 = f1;
        f0 = g0;
        f1 = g1;
#pragma unroll
        for (int t = 0; t < kUBatch; ++t) {
            js[t] = js2[t];
            ws[t] = ws2[t];
        }
    }
    // the block's sums into part[2 (ch V + q) + m][blk]
    __shared__ double red[8 * kUThreads];
    if (!__syncthreads_or(any)) return;  // every replica of the block stopped: no sums
    if (Cp <= 32 && (Cp & (Cp - 1)) == 0) {  // a warp's lanes of one chunk are Cp apart
        // the 2 V sums of a lane by halves: at each level a lane hands one half of its values to the lane
        // `o` away and merges the other half with that lane's, then whole values once one is left (8
        // merges instead of 32 for V = 4, Cp = 2)
        UntilSum<XT> v[2 * V];
#pragma unroll
        for (int q = 0; q < V; ++q) {
            if constexpr (sizeof(XT) == 4) {
                v[2 * q].v = d32[q];
                v[2 * q + 1].v = s32[q];
            } else {
                v[2 * q].v = d64[q];
                v[2 * q + 1].v = s64[q];
            }
        }
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, per = 2 * V * Cp;  // per <= 256
        int base = 0, held = 2 * V;  // this lane holds values base .. base + held - 1
#pragma unroll
        for (int l = 0; l < 5; ++l) {
            const int o = 16 >> l;
            constexpr int kAll = 2 * V;
            const int cnt = kAll >> l > 1 ? kAll >> l : 1;
            if (o >= Cp) {
                if (cnt > 1) {
                    const bool up = (lane & o) != 0;
#pragma unroll
                    for (int j = 0; j < cnt / 2; ++j) {
                        UntilSum<XT> keep = up ? v[cnt / 2 + j] : v[j], send = up ? v[j] : v[cnt / 2 + j];
                        keep.merge(send.from_lane(o));
                        v[j] = keep;
                    }
                    base += up ? cnt / 2 : 0;
                    held = cnt / 2;
                } else {
                    v[0].merge_lane(o);
                }
            }
        }
        typename UntilSum<XT>::Slot *slots = reinterpret_cast<typename UntilSum<XT>::Slot *>(red);  // [warp][chunk][value]
        if (lane % Cp < C) {
#pragma unroll
            for (int j = 0; j < 2 * V; ++j)
                if (j < held) slots[warp * per + (lane % Cp) * 2 * V + base + j] = v[j].slot();
        }
        __syncthreads();
        if (static_cast<int>(threadIdx.x) < 2 * V * C) {
            UntilSum<XT> t;
#pragma unroll
            for (int w = 0; w < kUWarps; ++w) t.merge(slots[w * per + threadIdx.x]);
            part[static_cast<int64_t>(threadIdx.x) * blocks + blk] = t.slot();
        }
        return;
    }
    // any C: a tree over the block's rows
    typename UntilSum<XT>::Slot *slots = reinterpret_cast<typename UntilSum<XT>::Slot *>(red);  // [m][thread]
#pragma unroll
    for (int q = 0; q < V; ++q) {
        UntilSum<XT> d, s;
        if constexpr (sizeof(XT) == 4) {
            d.v = d32[q];
            s.v = s32[q];
        } else {
            d.v = d64[q];
            s.v = s64[q];
        }
        for (int rows = rows_per_block; rows > 1;) {
            const int half = (rows + 1) / 2;
            if (rl >= half && rl < rows) {
                slots[threadIdx.x] = d.slot();
                slots[kUThreads + threadIdx.x] = s.slot();
            }
            __syncthreads();
            if (rl + half < rows) {
                d.merge(slots[threadIdx.x + half * Cp]);
                s.merge(slots[kUThreads + threadIdx.x + half * Cp]);
            }
            __syncthreads();
            rows = half;
        }
        if (rl == 0) {
            typename UntilSum<XT>::Slot *to = part + static_cast<int64_t>((ch * V + q) * 2) * blocks + blk;
            to[0] = d.slot();
            to[blocks] = s.slot();
        }
    }
}

__global__ void until_init_kernel(int pairs, int max_iters, int *running, int32_t *steps, int *n_running) {
    for (int t = threadIdx.x; t < pairs; t += blockDim.x) {
        running[t] = 1;
        steps[t] = max_iters;
    }
    if (threadIdx.x == 0) *n_running = pairs;
}

template <typename XT>
__global__ void __launch_bounds__(kUThreads)
until_last_kernel(const typename UntilSum<XT>::Slot *__restrict__ part, int blocks, double eps, int k, int R, int *running,
                  int32_t *__restrict__ steps, int *n_running) {
    const int t = static_cast<int>(blockIdx.x) * kUWarps + (threadIdx.x >> 5);
    if (t < R) until_decide<XT>(part, blocks, eps, k, t, running, steps, n_running);
}

// x^(steps) of the replicas that ended in the other buffer
template <typename XT>
__global__ void __launch_bounds__(kUThreads)
until_collect(XT *__restrict__ xa, const XT *__restrict__ xb, int64_t count, int R, const int32_t *__restrict__ steps) {
    for (int64_t t = static_cast<int64_t>(blockIdx.x) * kUThreads + threadIdx.x; t < count;
         t += static_cast<int64_t>(gridDim.x) * kUThreads)
        if (steps[t % R] & 1) xa[t] = xb[t];
}

// (the other buffer is an allocation of its own)
int vec_width(const void *x, int xtype, int R) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(x);
    if (xtype == ISING_F64) return R % 2 == 0 && a % 16 == 0 ? 2 : 1;
    return R % 4 == 0 && a % 16 == 0 ? 4 : R % 2 == 0 && a % 8 == 0 ? 2 : 1;
}

// threads per row: the chunks, rounded up to a power of two where at least 3 in 4 lanes stay busy
int row_threads(int C) {
    int p = 1;
    while (p < C) p <<= 1;
    return p <= 32 && 4 * C >= 3 * p ? p : C;
}

int until_blocks(const ising_context *c, int C) {
    const int64_t rows_per_block = kUThreads / row_threads(C);
    const int64_t cap = static_cast<int64_t>(c->num_sms) * kUBlocksPerSm;
    return static_cast<int>(std::max<int64_t>(1, std::min((c->n + rows_per_block - 1) / rows_per_block, cap)));
}

template <typename XT>
typename UntilSum<XT>::Slot *partials_of(const ising_context *c, int R, int k, StopState &s) {
    static_assert(sizeof(typename UntilSum<XT>::Slot) == sizeof(double), "the halves hold either");
    return reinterpret_cast<typename UntilSum<XT>::Slot *>(
        s.partials + (k & 1) * (until_partials_bytes(c, R) / (2 * sizeof(double))));
}

template <typename XT, typename VT, int V>
ising_status_t launch_until(const ising_context *c, const XT *xi, XT *xo, int R, const XT *h, const ParamTabs &p,
                            double eps, int k, StopState &s, cudaStream_t st) {
    const int C = R / V;
    const int blocks = until_blocks(c, C);
    const int dblocks = (R + kUWarps - 1) / kUWarps;
    DOCH_CUDA(launch_chained(until_kernel<XT, VT, V>, dim3(static_cast<unsigned>(dblocks + blocks)), dim3(kUThreads), st,
                             xi, xo, c->row_ptr, c->col, static_cast<const VT *>(c->val), h, static_cast<int>(c->n), R,
                             step_values<XT>(p, 0), row_threads(C), dblocks, eps, k, partials_of<XT>(c, R, k, s),
                             partials_of<XT>(c, R, k + 1, s), s.running, s.steps, s.n_running, s.progress, s.call));
    return ISING_OK;
}

template <typename XT, int V>
ising_status_t until_typed(const ising_context *c, const XT *xi, XT *xo, int R, const XT *h, const ParamTabs &p,
                           double eps, int k, StopState &s, cudaStream_t st) {
    switch (c->jtype) {
        case ISING_I8: return launch_until<XT, int8_t, V>(c, xi, xo, R, h, p, eps, k, s, st);
        case ISING_I32: return launch_until<XT, int32_t, V>(c, xi, xo, R, h, p, eps, k, s, st);
        case ISING_F32: return launch_until<XT, float, V>(c, xi, xo, R, h, p, eps, k, s, st);
        case ISING_F64: return launch_until<XT, double, V>(c, xi, xo, R, h, p, eps, k, s, st);
        default: return fail(ISING_ERR_UNSUPPORTED, "CSR value type not supported on the device");
    }
}

}  // namespace

// the rows that csr_step_pipe_kernel takes, with a block per row chunk at least
bool until_ok(const ising_context *c, const void *x, int xtype, int R) {
    return c->format == ISING_FMT_CSR && c->n_inst == 1 && (xtype == ISING_F32 || xtype == ISING_F64) &&
           R / vec_width(x, xtype, R) <= kUThreads && c->nnz <= static_cast<int64_t>(kPipeAvgDeg) * c->n &&
           c->n < (int64_t(1) << 30) && c->nnz < (int64_t(1) << 30);
}

size_t until_partials_bytes(const ising_context *c, int R) {
    return 2 * sizeof(double) * 2 * static_cast<size_t>(R) * static_cast<size_t>(c->num_sms) * kUBlocksPerSm;
}

ising_status_t until_init(int pairs, int max_iters, StopState &s, cudaStream_t st) {
    until_init_kernel<<<1, 256, 0, st>>>(pairs, max_iters, s.running, s.steps, s.n_running);
    DOCH_CUDA(cudaGetLastError());
    return ISING_OK;
}

ising_status_t until_step(const ising_context *c, const void *cur, void *nxt, int xtype, int R, const ParamTabs &p,
                          double eps, int k, StopState &s, cudaStream_t st) {
    const int V = vec_width(k % 2 == 0 ? cur : nxt, xtype, R);
    if (xtype == ISING_F64) {
        const double *xi = static_cast<const double *>(cur);
        double *xo = static_cast<double *>(nxt);
        return V == 2 ? until_typed<double, 2>(c, xi, xo, R, c->h_f64, p, eps, k, s, st)
                      : until_typed<double, 1>(c, xi, xo, R, c->h_f64, p, eps, k, s, st);
    }
    const float *xi = static_cast<const float *>(cur);
    float *xo = static_cast<float *>(nxt);
    return V == 4   ? until_typed<float, 4>(c, xi, xo, R, c->h_f32, p, eps, k, s, st)
           : V == 2 ? until_typed<float, 2>(c, xi, xo, R, c->h_f32, p, eps, k, s, st)
                    : until_typed<float, 1>(c, xi, xo, R, c->h_f32, p, eps, k, s, st);
}

ising_status_t until_finish(const ising_context *c, void *xa, const void *xb, int xtype, int R, double eps,
                            int launched, StopState &s, cudaStream_t st) {
    const int C = R / vec_width(xa, xtype, R);
    if (launched > 0) {
        const unsigned grid = static_cast<unsigned>((R + kUWarps - 1) / kUWarps);
        if (xtype == ISING_F64)
            until_last_kernel<double><<<grid, kUThreads, 0, st>>>(partials_of<double>(c, R, launched - 1, s), until_blocks(c, C),
                                                                  eps, launched - 1, R, s.running, s.steps, s.n_running);
        else
            until_last_kernel<float><<<grid, kUThreads, 0, st>>>(partials_of<float>(c, R, launched - 1, s), until_blocks(c, C),
                                                                 eps, launched - 1, R, s.running, s.steps, s.n_running);
        DOCH_CUDA(cudaGetLastError());
    }
    const int64_t count = c->n * R;
    const unsigned blocks = static_cast<unsigned>(
        std::max<int64_t>(1, std::min<int64_t>((count + kUThreads - 1) / kUThreads, 16LL * c->num_sms)));
    if (xtype == ISING_F64)
        until_collect<<<blocks, kUThreads, 0, st>>>(static_cast<double *>(xa), static_cast<const double *>(xb), count, R,
                                                   s.steps);
    else
        until_collect<<<blocks, kUThreads, 0, st>>>(static_cast<float *>(xa), static_cast<const float *>(xb), count, R,
                                                   s.steps);
    DOCH_CUDA(cudaGetLastError());
    return ISING_OK;
}

}  // namespace doch
