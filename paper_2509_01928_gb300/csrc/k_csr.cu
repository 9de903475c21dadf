// DOCH step for couplings in CSR form, Eq. FPE with the field inside g:
//   x_out[i][r] = cbrt( ( sum_e val[e] x_in[col[e]][r] + alpha_b x_in[i][r] + h_i ) / beta_b )
// for the instance b that owns row i (batched instances are concatenated).
//
// csr_step: one launch per step. A thread owns one row and a vector chunk of
// V replicas (V = 4/2/1 floats or 2/1 doubles), so the threads of a row read
// consecutive replicas of each neighbour x[j][*] (coalesced) and share the
// row's col/val entries. FP32 steps take the cube root as the prescaled
// power-of-two form of cbrt.cuh (the lattice, batched and dense kernels use the
// same form), FP64 steps two Newton steps (root.cuh): bound by FP64 arithmetic,
// 100,000 spins of degree 8, R = 16, 200 steps with the stopping rule 21.9 -> 14.3 ms
// against a quotient and cbrt.
//
// csr_step_pipe: the same step for short rows (at most kPipeAvgDeg entries per
// row on average, one instance, no monitor). The grid is one resident wave and a
// thread's loads are pipelined across its rows (csr_pipe.cuh); the sums are the
// ones csr_step forms, in the same order. A launch starts, and loads its first
// couplings, while the one before it ends: a gradient of 20,000 spins of degree 3,
// R = 8, FP32, 60 steps (170 short launches) 1.25 -> 0.93 ms, of 100,000 spins,
// R = 64, 100 steps 5.53 -> 4.95 ms.
//
// Instances that fit in shared memory run all their steps in one launch (k_csr_small.cu).
#include <algorithm>

#include "cbrt.cuh"
#include "csr_pipe.cuh"
#include "hamsum.cuh"
#include "internal.cuh"

namespace doch {
namespace {

__device__ __forceinline__ int find_inst(const int64_t *__restrict__ off, int n_inst, int64_t i) {
    int lo = 0, hi = n_inst - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(off + mid) <= i) lo = mid; else hi = mid - 1;
    }
    return lo;
}

constexpr int kCsrBatch = 8;  // entries whose loads are issued together

// H monitor fused into the step (TRACE, one instance): the step already holds
// u = J x^(k) and x^(k), so it also sums the terms of H(x^(k)) (Eq. Hamilton,
// -h^T x for a field): x^4, x^2, x u, h x per replica. FP64 iterates sum in
// FP64; FP32 iterates form the terms in FP32 and sum them per thread with a
// compensated (Kahan) FP32 sum. Each block writes FP64 partials
// hpart[block][R][4], summed over threads in a fixed order.
// A row takes C = R / V <= 256 threads; more replica chunks are taken by further launches, xi and xo moved on (R is the
// rows' stride throughout).
template <typename XT, typename VT, int V, bool TRACE>
__global__ void __launch_bounds__(256)
csr_step_kernel(const XT *__restrict__ xi, XT *__restrict__ xo, const int64_t *__restrict__ row_ptr,
                const int32_t *__restrict__ col, const VT *__restrict__ val, const XT *__restrict__ h,
                const int64_t *__restrict__ inst_off, int n_inst, int64_t n, int R, int C,
                const XT *__restrict__ alpha_tab, int alpha_len, int k,
                const XT *__restrict__ beta_tab, const float *__restrict__ zs_tab,
                const float *__restrict__ xs_tab, double *__restrict__ hpart) {
    const int ak = alpha_len == 1 ? 0 : k;
    // each thread keeps one replica chunk and strides over rows: no division in the loop
    const int rows_per_block = blockDim.x / C;
    const int ch = threadIdx.x % C;
    const int rl = threadIdx.x / C;
    HamSum<XT> hs[TRACE ? V : 1][4];
    // the cube root's constants: one instance's are loaded once per thread -- two loads per row cost the
    // S5 workload 2.5 % -- batched instances look theirs up per row
    const StepRoot<XT> root0(beta_tab, zs_tab, xs_tab, 0);
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * rows_per_block + rl; rl < rows_per_block && i < n;
         i += static_cast<int64_t>(gridDim.x) * rows_per_block) {
        const int b = n_inst > 1 ? find_inst(inst_off, n_inst, i) : 0;
        const XT a = alpha_tab[static_cast<int64_t>(b) * alpha_len + ak];
        const StepRoot<XT> root = n_inst > 1 ? StepRoot<XT>(beta_tab, zs_tab, xs_tab, b) : root0;
        XT acc[V];
#pragma unroll
        for (int q = 0; q < V; ++q) acc[q] = XT(0);
        const int64_t e1 = __ldg(row_ptr + i + 1);
        int64_t e = __ldg(row_ptr + i);
        // entries in batches of kCsrBatch: the index/value loads first, then the gathers, then
        // the products in entry order (the same sums as one entry at a time)
        for (; e + kCsrBatch <= e1; e += kCsrBatch) {
            int32_t js[kCsrBatch];
            XT ws[kCsrBatch];
#pragma unroll
            for (int t = 0; t < kCsrBatch; ++t) {
                js[t] = __ldg(col + e + t);
                ws[t] = coupling<XT, VT>(__ldg(val + e + t));
            }
            XT xv[kCsrBatch][V];
#pragma unroll
            for (int t = 0; t < kCsrBatch; ++t) ldv<XT, V>(xi + static_cast<int64_t>(js[t]) * R + ch * V, xv[t]);
#pragma unroll
            for (int t = 0; t < kCsrBatch; ++t)
#pragma unroll
                for (int q = 0; q < V; ++q) acc[q] += ws[t] * xv[t][q];
        }
        for (; e < e1; ++e) {
            const int64_t j = __ldg(col + e);
            const XT w = coupling<XT, VT>(__ldg(val + e));
            XT xv[V];
            ldv<XT, V>(xi + j * R + ch * V, xv);
#pragma unroll
            for (int q = 0; q < V; ++q) acc[q] += w * xv[q];
        }
        XT xs[V], out[V];
        ldv<XT, V>(xi + i * R + ch * V, xs);
        const XT hi = h ? h[i] : XT(0);
#pragma unroll
        for (int q = 0; q < V; ++q) out[q] = root(acc[q] + a * xs[q] + hi);
        stv<XT, V>(xo + i * R + ch * V, out);
        if constexpr (TRACE) {
#pragma unroll
            for (int q = 0; q < V; ++q) {
                const XT x2 = xs[q] * xs[q];
                hs[q][0].add(x2 * x2);
                hs[q][1].add(x2);
                hs[q][2].add(xs[q] * acc[q]);
                hs[q][3].add(hi * xs[q]);
            }
        }
    }
    if constexpr (TRACE) {
        // per replica: threads of the same chunk ch (rows rl = 0 .. rows_per_block-1) in row order
        __shared__ double red[256][4];
#pragma unroll
        for (int q = 0; q < V; ++q) {
#pragma unroll
            for (int m = 0; m < 4; ++m) red[threadIdx.x][m] = hs[q][m].value();
            __syncthreads();
            if (rl == 0) {
                double t[4] = {0.0, 0.0, 0.0, 0.0};
                for (int r2 = 0; r2 < rows_per_block; ++r2)
#pragma unroll
                    for (int m = 0; m < 4; ++m) t[m] += red[r2 * C + ch][m];
#pragma unroll
                for (int m = 0; m < 4; ++m)
                    hpart[(static_cast<int64_t>(blockIdx.x) * R + ch * V + q) * 4 + m] = t[m];
            }
            __syncthreads();
        }
    }
}

constexpr int kPipeB = 4;  // entries of a row's first batch, loaded one row ahead

// Rows and entry offsets are 32-bit here (n, nnz < 2^30, checked by use_pipe).
template <typename XT>
constexpr int pipe_blocks_per_sm() { return sizeof(XT) == 4 ? kCsrPipeBlocksPerSm : kCsrPipeBlocksPerSm - 1; }

template <typename XT, typename VT, int V>
__global__ void __launch_bounds__(256, pipe_blocks_per_sm<XT>())
csr_step_pipe_kernel(const XT *__restrict__ xi, XT *__restrict__ xo, const int64_t *__restrict__ row_ptr,
                     const int32_t *__restrict__ col, const VT *__restrict__ val, const XT *__restrict__ h,
                     int n, int R, StepValues<XT> par) {
    const int C = R / V;
    const int rows_per_block = blockDim.x / C;
    int ch = threadIdx.x % C;
    const int rl = threadIdx.x / C;
    const int S = static_cast<int>(gridDim.x) * rows_per_block;
    int i = rl < rows_per_block ? static_cast<int>(blockIdx.x) * rows_per_block + rl : n;
    int e0, e1, f0, f1;  // entry ranges of rows i and i + S
    int32_t js[kPipeB];
    XT ws[kPipeB];
    pipe_row_range(row_ptr, i, n, e0, e1);
    pipe_row_range(row_ptr, i + S, n, f0, f1);
    pipe_first_batch<kPipeB>(col, val, e0, e1, js, ws);
    pdl_wait();  // the couplings above are never written
    pdl_trigger();
    pdl_after(ch);
    const XT a = par.alpha;
    const StepRoot<XT> root(par);
    for (; i < n; i += S) {
        const int cnt = e1 - e0 < kPipeB ? static_cast<int>(e1 - e0) : kPipeB;
        XT xv[kPipeB][V];
#pragma unroll
        for (int t = 0; t < kPipeB; ++t)
            if (t < cnt) ldv_cg<XT, V>(xi + static_cast<int64_t>(js[t]) * R + ch * V, xv[t]);
        XT xs[V];
        ldv_cg<XT, V>(xi + static_cast<int64_t>(i) * R + ch * V, xs);
        const XT hi = h ? h[i] : XT(0);
        // the next row's first batch and the range of the row after it
        int32_t js2[kPipeB];
        XT ws2[kPipeB];
        pipe_first_batch<kPipeB>(col, val, f0, f1, js2, ws2);
        int g0, g1;
        pipe_row_range(row_ptr, i + 2 * S, n, g0, g1);
        XT acc[V];
#pragma unroll
        for (int q = 0; q < V; ++q) acc[q] = XT(0);
#pragma unroll
        for (int t = 0; t < kPipeB; ++t)
            if (t < cnt) {
#pragma unroll
                for (int q = 0; q < V; ++q) acc[q] += ws[t] * xv[t][q];
            }
        // entries past the first batch, in entry order
#pragma unroll 4
        for (int e = e0 + kPipeB; e < e1; ++e) {
            const int64_t j = __ldg(col + e);
            const XT w = coupling<XT, VT>(__ldg(val + e));
            XT xr[V];
            ldv_cg<XT, V>(xi + j * R + ch * V, xr);
#pragma unroll
            for (int q = 0; q < V; ++q) acc[q] += w * xr[q];
        }
        XT out[V];
#pragma unroll
        for (int q = 0; q < V; ++q) out[q] = root(acc[q] + a * xs[q] + hi);
        stv<XT, V>(xo + static_cast<int64_t>(i) * R + ch * V, out);
        e0 = f0;
        e1 = f1;
        f0 = g0;
        f1 = g1;
#pragma unroll
        for (int t = 0; t < kPipeB; ++t) {
            js[t] = js2[t];
            ws[t] = ws2[t];
        }
    }
}

int step_blocks(const ising_context *c, int C) {
    const int rows_per_block = C <= 256 ? 256 / C : 1;
    int64_t blocks = (c->n + rows_per_block - 1) / rows_per_block;
    const int64_t cap = static_cast<int64_t>(c->num_sms) * 32;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    return static_cast<int>(blocks);
}

// short rows: the pipelined kernel (one resident wave, 32-bit row and entry offsets) serves one
// instance without the monitor
bool use_pipe(const ising_context *c, int C, bool traced) {
    return !traced && c->n_inst == 1 && C <= 256 && c->nnz <= static_cast<int64_t>(kPipeAvgDeg) * c->n &&
           c->n < (int64_t(1) << 30) && c->nnz < (int64_t(1) << 30);
}

template <typename XT>
int pipe_blocks(const ising_context *c, int C) {
    const int rows_per_block = 256 / C;
    int64_t blocks = (c->n + rows_per_block - 1) / rows_per_block;
    const int64_t cap = static_cast<int64_t>(c->num_sms) * pipe_blocks_per_sm<XT>();
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    return static_cast<int>(blocks);
}

// the update tables of a step: beta (FP64) or the cube root's prescale (FP32, per instance)
template <typename XT>
struct StepTabs {
    const XT *alpha;
    int alpha_len;
    const XT *beta;
    const float *zs;
    const float *xsc;
    StepValues<XT> now;  // one instance: the step's own
};

template <typename XT, typename VT, int V>
cudaError_t launch_step(const ising_context *c, const XT *xi, XT *xo, int R, const XT *h, const StepTabs<XT> &t, int k,
                 double *hpart, cudaStream_t st) {
    const int C = R / V;
    if (use_pipe(c, C, hpart != nullptr)) {
        return launch_chained(csr_step_pipe_kernel<XT, VT, V>, dim3(static_cast<unsigned>(pipe_blocks<XT>(c, C))),
                              dim3(256), st, xi, xo, c->row_ptr, c->col, static_cast<const VT *>(c->val), h,
                              static_cast<int>(c->n), R, t.now);
    }
    if (hpart)  // C <= 256 (dispatch_val)
        csr_step_kernel<XT, VT, V, true><<<static_cast<unsigned>(step_blocks(c, C)), 256, 0, st>>>(
            xi, xo, c->row_ptr, c->col, static_cast<const VT *>(c->val), h, c->inst_off, c->n_inst,
            c->n, R, C, t.alpha, t.alpha_len, k, t.beta, t.zs, t.xsc, hpart);
    else
        for (int c0 = 0; c0 < C; c0 += 256) {
            const int cn = std::min(256, C - c0);
            csr_step_kernel<XT, VT, V, false><<<static_cast<unsigned>(step_blocks(c, cn)), 256, 0, st>>>(
                xi + c0 * V, xo + c0 * V, c->row_ptr, c->col, static_cast<const VT *>(c->val), h, c->inst_off, c->n_inst,
                c->n, R, cn, t.alpha, t.alpha_len, k, t.beta, t.zs, t.xsc, nullptr);
        }
    return cudaGetLastError();
}

template <typename XT, int V>
ising_status_t dispatch_val(const ising_context *c, const XT *xi, XT *xo, int R, const XT *h, const StepTabs<XT> &t,
                            int k, double *hpart, cudaStream_t st) {
    // instances whose iterate fits shared memory take any R (k_csr_small.cu, or single steps where that declines)
    if (R / V > 1024 && static_cast<size_t>(c->max_inst_n) > csr_fused_max_spins(sizeof(XT) == 8 ? ISING_F64 : ISING_F32))
        return fail(ISING_ERR_UNSUPPORTED, "CSR step: R / vector width must be <= 1024");
    if (hpart && R / V > 256) return ISING_ERR_UNSUPPORTED;  // the fused monitor needs one row per 256 threads
    switch (c->jtype) {
        case ISING_I8: DOCH_CUDA((launch_step<XT, int8_t, V>(c, xi, xo, R, h, t, k, hpart, st))); break;
        case ISING_I32: DOCH_CUDA((launch_step<XT, int32_t, V>(c, xi, xo, R, h, t, k, hpart, st))); break;
        case ISING_F32: DOCH_CUDA((launch_step<XT, float, V>(c, xi, xo, R, h, t, k, hpart, st))); break;
        case ISING_F64: DOCH_CUDA((launch_step<XT, double, V>(c, xi, xo, R, h, t, k, hpart, st))); break;
        default: return fail(ISING_ERR_UNSUPPORTED, "CSR value type not supported on the device");
    }
    return ISING_OK;
}

}  // namespace

size_t csr_fused_max_spins(int xtype) {
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return 0;
    return static_cast<size_t>(optin) / (2 * (xtype == ISING_F64 ? 8 : 4));
}

static ising_status_t csr_step_impl(const ising_context *c, const void *xi, void *xo, int xtype, int R,
                                    const ParamTabs &p, int k, double *hpart, int *blocks, cudaStream_t st) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(xi) | reinterpret_cast<uintptr_t>(xo);
    if (xtype == ISING_F32) {
        const float *x_in = static_cast<const float *>(xi);
        float *x_out = static_cast<float *>(xo);
        const StepTabs<float> t{p.alpha_f, p.alpha_len, p.inv_beta_f, p.zscale_f, p.xscale_f, step_values<float>(p, k)};
        if (R % 4 == 0 && a % 16 == 0) {
            *blocks = step_blocks(c, R / 4);
            return dispatch_val<float, 4>(c, x_in, x_out, R, c->h_f32, t, k, hpart, st);
        }
        if (R % 2 == 0 && a % 8 == 0) {
            *blocks = step_blocks(c, R / 2);
            return dispatch_val<float, 2>(c, x_in, x_out, R, c->h_f32, t, k, hpart, st);
        }
        *blocks = step_blocks(c, R);
        return dispatch_val<float, 1>(c, x_in, x_out, R, c->h_f32, t, k, hpart, st);
    }
    if (xtype == ISING_F64) {
        const double *x_in = static_cast<const double *>(xi);
        double *x_out = static_cast<double *>(xo);
        const StepTabs<double> t{p.alpha_d, p.alpha_len, p.beta_d, nullptr, nullptr, step_values<double>(p, k)};
        if (R % 2 == 0 && a % 16 == 0) {
            *blocks = step_blocks(c, R / 2);
            return dispatch_val<double, 2>(c, x_in, x_out, R, c->h_f64, t, k, hpart, st);
        }
        *blocks = step_blocks(c, R);
        return dispatch_val<double, 1>(c, x_in, x_out, R, c->h_f64, t, k, hpart, st);
    }
    return fail(ISING_ERR_UNSUPPORTED, "CSR iterate type must be F32 or F64");
}

ising_status_t csr_step(const ising_context *c, const void *xi, void *xo, int xtype, int R,
                        const ParamTabs &p, int k, cudaStream_t st) {
    int blocks = 0;
    return csr_step_impl(c, xi, xo, xtype, R, p, k, nullptr, &blocks, st);
}

ising_status_t csr_step_traced(ising_context *c, const void *xi, void *xo, int xtype, int R, const ParamTabs &p,
                               int k, double alpha_k, double beta, double *H_out, cudaStream_t st) {
    if (c->n_inst != 1) return ISING_ERR_UNSUPPORTED;
    const size_t max_blocks = static_cast<size_t>(c->num_sms) * 32;  // the cap of step_blocks
    DOCH_CHECK(c->partials.ensure(sizeof(double) * 4 * static_cast<size_t>(R) * max_blocks));
    int blocks = 0;
    const ising_status_t s = csr_step_impl(c, xi, xo, xtype, R, p, k, c->partials.as<double>(), &blocks, st);
    if (s != ISING_OK) return s;
    return ham_fused_finish_launch(c->partials.as<double>(), blocks, R, alpha_k, beta, H_out, st);
}

}  // namespace doch
