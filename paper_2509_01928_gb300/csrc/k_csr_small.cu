// DOCH steps (Eq. FPE) of CSR instances whose iterate fits in shared memory: all steps of a
// run in one launch,
//   x'[i][r] = cbrt( ( sum_e val[e] x[col[e]][r] + alpha_b x[i][r] + h_i ) / beta_b ).
//
// One cluster of K CTAs (K = 16, 8, 4, 2 or 1) per (instance, replica). Every CTA keeps both
// copies of the pair's whole iterate, forms the rows of its share [q c, (q + 1) c), c = ceil(n_b / K),
// and stores each new value into the next copy of all K CTAs (distributed shared memory); a
// cluster barrier (about 400 clocks) ends each step. P threads share a row: each adds every P-th
// entry, a shuffle tree adds the P sums, and then one thread per row takes the cube root, in
// whole warps. The couplings of a CTA's rows are copied to shared memory once per launch, already
// in the iterate's type.
//
// Bound by FP64 arithmetic (2 lanes per clock and SM; an integer -> FP64 conversion costs as much
// as an FP64 FMA): one FMA per entry and replica, the tree and nine operations per cube root. 800
// spins, 38,000 entries, R = 8, FP64: 10.0 us per step with one thread per row, the couplings
// converted at every use and CUDA's cbrt of a quotient, 3.7 us per step now; the arithmetic
// alone takes about 0.9 us on the 128 SMs used.
#include <algorithm>

#include "internal.cuh"
#include "root.cuh"

namespace doch {
namespace {

__device__ __forceinline__ uint32_t cl_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cl_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cl_map(const void *p, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(r)
                 : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(rank));
    return r;
}
__device__ __forceinline__ void cl_store(uint32_t a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void cl_store(uint32_t a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

// Shared memory: cur | nxt (XT [nb] each) | z (XT [rows], P > 1 only), then, as far as there is room
// for at least the shares it fits, val (XT [cap]) | row ranges (int [rows + 1]) | col (uint16 [cap])
template <typename XT, int P>
constexpr int64_t state_bytes(int64_t nb, int64_t rows) {
    return static_cast<int64_t>(sizeof(XT)) * (2 * nb + (P > 1 ? rows : 0)) + 16;
}
template <typename XT>
constexpr int64_t entry_bytes() { return sizeof(XT) + sizeof(uint16_t); }

template <typename XT, typename VT, int P>
__global__ void __launch_bounds__(1024)
csr_small(const XT *x_in, XT *x_out, const int64_t *__restrict__ row_ptr,
          const int32_t *__restrict__ col, const VT *__restrict__ val, const XT *__restrict__ h,
          const int64_t *__restrict__ inst_off, int64_t n, int R, const double *__restrict__ alpha_tab, int alpha_len,
          const double *__restrict__ beta_tab, int k0, int iters, int K, int rows_cap, int cap,
          unsigned char *rec, size_t rec_stride, int rec_every) {
    extern __shared__ __align__(16) unsigned char small_smem[];
    const int q = static_cast<int>(cl_rank());
    const int b = blockIdx.y, r = blockIdx.x / K;
    const int64_t lo = inst_off ? inst_off[b] : 0;
    const int64_t hi = inst_off ? inst_off[b + 1] : n;
    const int nb = static_cast<int>(hi - lo);
    const int chunk = (nb + K - 1) / K;  // <= rows_cap
    const int i0 = min(nb, q * chunk), i1 = min(nb, i0 + chunk), rows = i1 - i0;
    XT *cur = reinterpret_cast<XT *>(small_smem), *nxt = cur + nb;
    XT *z = nxt + nb;
    XT *lv = P > 1 ? z + rows_cap : z;
    int *lr = reinterpret_cast<int *>(lv + cap);
    uint16_t *lc = reinterpret_cast<uint16_t *>(lr + rows_cap + 1);
    for (int i = threadIdx.x; i < nb; i += blockDim.x) cur[i] = x_in[(lo + i) * R + r];
    const int64_t e0 = row_ptr[lo + i0];
    const bool local = row_ptr[lo + i1] - e0 <= cap;  // uniform over the block
    for (int i = threadIdx.x; i <= rows && local; i += blockDim.x) lr[i] = static_cast<int>(row_ptr[lo + i0 + i] - e0);
    if (local) {
        const int cnt = static_cast<int>(row_ptr[lo + i1] - e0);
        for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
            lv[e] = static_cast<XT>(val[e0 + e]);
            lc[e] = static_cast<uint16_t>(col[e0 + e] - lo);
        }
    }
    const auto root = make_root<XT>(beta_tab[b]);
    const double *arow = alpha_tab + static_cast<int64_t>(b) * alpha_len;
    const int sub = threadIdx.x % P;
    const int rl = threadIdx.x / P, rstep = blockDim.x / P;
    const int top = (rows + rstep - 1) / rstep * rstep;  // whole warps take part in the shuffles
    // every CTA of the cluster runs, and has loaded, before the first remote store
    if (K > 1) cl_sync();
    else __syncthreads();
    for (int k = 0; k < iters; ++k) {
        const XT a = static_cast<XT>(arow[alpha_len == 1 ? 0 : k0 + k]);
        const bool keep = rec && (k + 1) % rec_every == 0;
        XT *rp = reinterpret_cast<XT *>(rec + (keep ? static_cast<size_t>((k + 1) / rec_every - 1) : 0) * rec_stride);
        auto update = [&](int i, XT u) {  // row i of the share: the new value into every CTA's next copy
            const int64_t row = lo + i0 + i;
            const XT hv = h ? __ldg(h + row) : XT(0);
            const XT v = root_newton(u + a * cur[i0 + i] + hv, root);
            nxt[i0 + i] = v;
            for (int t = 1; t < K; ++t) {
                const int to = q + t < K ? q + t : q + t - K;
                cl_store(cl_map(nxt + i0 + i, static_cast<uint32_t>(to)), v);
            }
            if (keep) rp[row * R + r] = v;
        };
        for (int i = rl; i < top; i += rstep) {
            XT acc = XT(0);
            if (i < rows) {
                if (local) {
                    const int f1 = lr[i + 1];
#pragma unroll 4
                    for (int e = lr[i] + sub; e < f1; e += P) acc += lv[e] * cur[lc[e]];
                } else {
                    const int64_t f1 = __ldg(row_ptr + lo + i0 + i + 1);
                    for (int64_t e = __ldg(row_ptr + lo + i0 + i) + sub; e < f1; e += P)
                        acc += static_cast<XT>(__ldg(val + e)) * cur[__ldg(col + e) - lo];
                }
            }
#pragma unroll
            for (int o = P / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (P == 1) {
                if (i < rows) update(i, acc);
            } else if (sub == 0 && i < rows) {
                z[i] = acc;
            }
        }
        if (P > 1) {
            __syncthreads();
            for (int i = threadIdx.x; i < rows; i += blockDim.x) update(i, z[i]);
        }
        if (K > 1) cl_sync();  // the new values of every share are in every CTA; the old copy is free
        else __syncthreads();
        XT *t = cur;
        cur = nxt;
        nxt = t;
    }
    if (x_out)
        for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) x_out[(lo + i) * R + r] = cur[i];
}

// the cluster size: the largest K in {16, 8, 4, 2} (16 is a non-portable size) that leaves each CTA
// at least 32 rows and keeps all pairs' clusters within the SMs; 1 when none does
int cluster_k(const ising_context *c, int R, int kmax) {
    for (int K = kmax; K >= 2; K >>= 1)
        if (static_cast<int64_t>(c->n_inst) * R * K <= c->num_sms && c->max_inst_n >= 32LL * K) return K;
    return 1;
}

template <typename XT, typename VT, int P>
ising_status_t launch_k(const ising_context *c, const XT *x_in, XT *x_out, int R, const XT *h, const ParamTabs &p,
                        int k0, int iters, int K, const SmallRecord &rec, int64_t optin, cudaStream_t st) {
    const int64_t chunk = (c->max_inst_n + K - 1) / K;
    const int64_t state = state_bytes<XT, P>(c->max_inst_n, chunk);
    if (state > optin) return ISING_ERR_UNSUPPORTED;
    // room for the couplings of the fullest share, as far as it goes (shares that need more read the CSR arrays)
    const int64_t left = optin - state - static_cast<int64_t>(sizeof(int)) * (chunk + 1);
    const int64_t cap = left <= 0 ? -1 : std::min(left / entry_bytes<XT>(), std::min(c->max_row_nnz * chunk, c->nnz)) / 4 * 4;
    const int smem = static_cast<int>(cap < 0 ? state : optin - left + cap * entry_bytes<XT>());
    auto kern = csr_small<XT, VT, P>;
    DOCH_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    if (K > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        return ISING_ERR_UNSUPPORTED;
    }
    const int threads = static_cast<int>(std::min<int64_t>(1024, (chunk * P + 31) / 32 * 32));
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(K);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(static_cast<unsigned>(R * K), static_cast<unsigned>(c->n_inst));
    cfg.blockDim = dim3(static_cast<unsigned>(threads));
    cfg.dynamicSmemBytes = static_cast<size_t>(smem);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (K > 1) {
        int nclusters = 0;
        if (cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg) != cudaSuccess || nclusters < 1) {
            cudaGetLastError();
            return ISING_ERR_UNSUPPORTED;
        }
    }
    DOCH_CUDA(cudaLaunchKernelEx(&cfg, kern, x_in, x_out, static_cast<const int64_t *>(c->row_ptr),
                                 static_cast<const int32_t *>(c->col), static_cast<const VT *>(c->val), h,
                                 static_cast<const int64_t *>(c->n_inst > 1 ? c->inst_off : nullptr), c->n, R,
                                 p.alpha_d, p.alpha_len, p.beta_d, k0, iters, K, static_cast<int>(chunk),
                                 static_cast<int>(cap), static_cast<unsigned char *>(rec.base), rec.stride,
                                 rec.every));
    return ISING_OK;
}

template <typename XT, typename VT>
ising_status_t launch_small(const ising_context *c, const XT *x_in, XT *x_out, int R, const XT *h, const ParamTabs &p,
                            int k0, int iters, const SmallRecord &rec, cudaStream_t st) {
    int dev = 0, optin = 0;
    DOCH_CUDA(cudaGetDevice(&dev));
    DOCH_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    for (int kmax = 16;; kmax >>= 1) {
        const int K = cluster_k(c, R, kmax);
        const int64_t chunk = (c->max_inst_n + K - 1) / K;
        // threads per row: four or two where a share is small and its rows are long enough to split (more
        // would spend as many FP64 additions on the tree as they take from the rows)
        const bool split = c->nnz >= 8 * c->n;
        const ising_status_t s =
            split && chunk <= 128   ? launch_k<XT, VT, 4>(c, x_in, x_out, R, h, p, k0, iters, K, rec, optin, st)
            : split && chunk <= 512 ? launch_k<XT, VT, 2>(c, x_in, x_out, R, h, p, k0, iters, K, rec, optin, st)
                                    : launch_k<XT, VT, 1>(c, x_in, x_out, R, h, p, k0, iters, K, rec, optin, st);
        if (s != ISING_ERR_UNSUPPORTED || K == 1) return s;
        kmax = K;  // this size is not available: try the next smaller one
    }
}

template <typename XT>
ising_status_t dispatch_small(const ising_context *c, const XT *x_in, XT *x_out, int R, const XT *h,
                              const ParamTabs &p, int k0, int iters, const SmallRecord &rec, cudaStream_t st) {
    switch (c->jtype) {
        case ISING_I8: return launch_small<XT, int8_t>(c, x_in, x_out, R, h, p, k0, iters, rec, st);
        case ISING_I32: return launch_small<XT, int32_t>(c, x_in, x_out, R, h, p, k0, iters, rec, st);
        case ISING_F32: return launch_small<XT, float>(c, x_in, x_out, R, h, p, k0, iters, rec, st);
        case ISING_F64: return launch_small<XT, double>(c, x_in, x_out, R, h, p, k0, iters, rec, st);
        default: return fail(ISING_ERR_UNSUPPORTED, "CSR value type not supported on the device");
    }
}

}  // namespace

ising_status_t csr_small_run(const ising_context *c, const void *x_in, void *x_out, int xtype, int R,
                             const ParamTabs &p, int k0, int iters, const SmallRecord &rec, cudaStream_t st) {
    if (static_cast<size_t>(c->max_inst_n) > csr_fused_max_spins(xtype)) return ISING_ERR_UNSUPPORTED;
    if (xtype == ISING_F64)
        return dispatch_small<double>(c, static_cast<const double *>(x_in), static_cast<double *>(x_out), R, c->h_f64,
                                      p, k0, iters, rec, st);
    if (xtype == ISING_F32)
        return dispatch_small<float>(c, static_cast<const float *>(x_in), static_cast<float *>(x_out), R, c->h_f32, p,
                                     k0, iters, rec, st);
    return ISING_ERR_UNSUPPORTED;
}

ising_status_t csr_fused(const ising_context *c, void *x, int xtype, int R, const ParamTabs &p, int iters,
                         cudaStream_t st) {
    return csr_small_run(c, x, x, xtype, R, p, 0, iters, SmallRecord{}, st);
}

}  // namespace doch
