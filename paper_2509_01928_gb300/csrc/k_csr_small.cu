// DOCH steps (Eq. FPE) of CSR instances whose iterate fits in shared memory: all steps of a
// run in one launch,
//   x'[i][r] = cbrt( ( sum_e val[e] x[col[e]][r] + alpha_b x[i][r] + h_i ) / beta_b ).
//
// One cluster of K <= 16 CTAs per (instance, replica). Every CTA keeps both
// copies of the pair's whole iterate, forms the rows of its share [q c, (q + 1) c), c = ceil(n_b / K),
// and sends each new value to the next copy of all K CTAs (distributed shared memory), each of which
// counts the bytes that arrive (about 650 clocks per step). P threads share a row: each adds every P-th
// entry, a shuffle tree adds the P sums, and then one thread per row takes the cube root, in
// whole warps. The couplings of a CTA's rows are copied to shared memory once per launch, already
// in the iterate's type (FP64 iterates and 8-bit couplings: the integers, or the upper words of the
// FP64 values, whose lower words are zero: 6 instead of 10 bytes an entry).
//
// Bound by the latency of a step's chain: products, tree, cube root, exchange (29 % of the issue slots and 14 %
// of the FP64 pipe active for the instance below, 13 warps per SM, bank conflicts on a random gather), in which
// FP64 operations weigh most (half a lane per clock and SM partition, about 150 clocks from one to the next
// that needs it; an integer -> FP64 conversion costs as much as an FMA). FP64 iterates with 8-bit couplings take their
// products in integers (fixed point, below): eight FP64 operations per cube root and four around it are left.
// 800 spins, 38,000 entries, R = 8, FP64, per step: 10.0 us with one thread per row, the couplings
// converted at every use and CUDA's cbrt of a quotient; 3.4 us with the couplings held in FP64 and four
// threads per row (products 2.3, update 0.8, exchange 0.35); 2.75 us in fixed point with eight. The FP64
// operations alone take about 0.25 us on the 128 SMs used.
#include <algorithm>
#include <type_traits>

#include "hamsum.cuh"
#include "internal.cuh"
#include "mbar.cuh"
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
// a value into a peer's shared memory; its bytes count on the peer's mbarrier when they are there
__device__ __forceinline__ void cl_send(uint32_t a, double v, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(a),
                 "l"(__double_as_longlong(v)), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void cl_send(uint32_t a, float v, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(a),
                 "r"(__float_as_uint(v)), "r"(bar)
                 : "memory");
}

// The exchange of a cluster's shares. Every CTA counts the bytes its peers send for step k on one of
// two mbarriers (k even / odd). A peer sends step k + 1 only after this CTA's step k reached it whole,
// which this CTA sends after it has received step k - 1: so two mbarriers, and two copies of the
// iterate, are enough, and no cluster-wide barrier is needed. This holds among the CTAs that own rows,
// the first `owners` of the cluster. One without rows (a short instance beside a long one, whose size
// sets the cluster's) holds nobody up: it takes no part, and nothing is sent to it. Waits are bounded
// (1 s): on expiry the error word is set and the kernel ends at its closing cluster barrier.
struct Exchange {
    unsigned long long bar[2];
    int abort_flag;
};
constexpr int kStaticSmem = 128;  // at least the kernels' static shared memory

__device__ __forceinline__ void exchange_init(Exchange &x) {  // before the opening cluster barrier
    if (threadIdx.x == 0) {
        mbar_init(&x.bar[0], 1);
        mbar_init(&x.bar[1], 1);
        x.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
}
// step s (from 0): arm for `bytes` from the peers
__device__ __forceinline__ void exchange_expect(Exchange &x, int s, uint32_t bytes) {
    if (threadIdx.x == 0) mbar_expect_tx(&x.bar[s & 1], bytes);
}
template <typename T>
__device__ __forceinline__ void exchange_send(Exchange &x, int s, T *slot, T v, int q, int owners) {
    for (int t = 1; t < owners; ++t) {
        const uint32_t to = static_cast<uint32_t>(q + t < owners ? q + t : q + t - owners);
        cl_send(cl_map(slot, to), v, cl_map(&x.bar[s & 1], to));
    }
}
// all threads: this CTA's own share is written and the peers' have arrived
__device__ __forceinline__ bool exchange_wait(Exchange &x, int s, int owners, int *err) {
    if (owners == 1) {
        __syncthreads();
        return true;
    }
    const bool ok = mbar_wait(&x.bar[s & 1], (s >> 1) & 1, err, &x.abort_flag);
    return !__syncthreads_or(!ok);
}

// a coupling as held in shared memory
template <typename XT, typename VT>
struct Held {
    using type = XT;
    static __device__ __forceinline__ XT pack(VT v) { return static_cast<XT>(v); }
    static __device__ __forceinline__ XT value(XT v) { return v; }
};
template <>
struct Held<double, int8_t> {  // the integer (fixed-point steps), or the FP64 value's upper word
    using type = int;
    static __device__ __forceinline__ int pack(int8_t v) { return v; }
    static __device__ __forceinline__ int upper(int v) { return v ? __double2hiint(static_cast<double>(v)) : 0; }
    static __device__ __forceinline__ double value(int v) { return __hiloint2double(v, 0); }
};

// Fixed-point steps (FP64 iterates, 8-bit couplings). The iterate is held and exchanged in FP64; at the
// start of a step every CTA also forms the integers round(x_j 2^s) of all of it, s from a bound M >= max |x_j|
// such that every row's sum of |J_ij x_j| stays below 2^63. J x is then summed in integers, at integer
// rate, with an error of at most rowabs_i 2^-s / 2 in row i (rowabs_i = sum_j |J_ij|).
// A row takes that sum where it is no less exact than FP64 sums: where sum_j |J_ij x_j| >= rowabs_i 2^52 2^-s, so
// that the error is within 2^-53 of the sum of the terms' magnitudes, one FP64 rounding. Every row tests
// this at every step, from the upper words of its terms (`mag`, in units of 2^(32 - s)), and sums in FP64
// otherwise: rows whose neighbours are small beside the largest component (starts over many orders of
// magnitude, a spin pinned by a strong field, hubs). Where a row sum of |J| reaches kRowLimit most rows
// would fail (rowabs M 2^-63 2^52 against a mean |x_j|), and such instances take FP64 sums throughout.
// Error of the row sums that pass, relative to the terms' magnitudes, rms over all rows (FP64 in four partial
// sums / fixed point): 800 spins of 48 entries 2.4e-17 / 0.9e-17, 1500 of 120 2.1e-17 / 0.5e-17, 1200 of 24
// 2.6e-17 / 1.1e-17; x after 1000 steps of 800 spins, six seeds: within 4.4e-16 to 5.3e-16 of 64-bit torch in both.
// M of the next iterate follows from |x'| <= cbrt(((rowabs + |alpha|) M + max |h|) / beta), rounded up. Runs
// that record iterates keep FP64 sums: the bounds, and so the rounding, would depend on where a run starts.
constexpr int kRowLimit = 256;
__device__ __forceinline__ float next_bound(float m, float rowabs, float alpha, float hmax, float inv_beta) {
    const float z = ((rowabs + fabsf(alpha)) * m + hmax) * inv_beta;
    return ex2_fast(lg2_fast(z) * (1.0f / 3.0f)) * 1.0001f;
}
__device__ __forceinline__ int fixed_shift(float m, float rowabs) {  // rowabs m 2^shift < 2^63 / 1.0001
    return 63 - (ilogbf(rowabs * m * 1.0001f) + 1);
}
// round(v 2^shift), |v 2^shift| < 2^63, by integer shifts (an FP64 conversion costs as much as an FMA)
__device__ __forceinline__ long long to_fixed(double v, int shift) {
    const int hi = __double2hiint(v), e = (hi >> 20) & 0x7ff;
    const unsigned long long m = static_cast<unsigned long long>((hi & 0xfffff) | (e ? 0x100000 : 0)) << 32 |
                                 static_cast<unsigned>(__double2loint(v));
    const int s = (e ? e : 1) + shift - 1075;  // |v| 2^shift = m 2^s
    unsigned long long r = 0;
    if (s >= 0) r = m << s;
    else if (s > -55) r = ((m >> (-s - 1)) + 1) >> 1;
    return hi < 0 ? -static_cast<long long>(r) : static_cast<long long>(r);
}
__device__ __forceinline__ double two_to(int e) { return __hiloint2double((1023 + e) << 20, 0); }

// Shared memory: cur | nxt (XT [nb] each) | z (XT [rows], P > 1 only) | where fixed-point steps may run
// integers (int64 [nb]) | rowabs (int [rows]), then, as far as there is room
// for at least the shares it fits, val (Held [cap]) | row ranges (int [rows + 1]) | col (uint16 [cap])
template <typename XT, int P>
constexpr int64_t state_bytes(int64_t nb, int64_t rows, bool fix) {
    return static_cast<int64_t>(sizeof(XT)) * (2 * nb + (P > 1 ? rows : 0)) + (fix ? 8 * nb + 4 * rows : 0) + 16;
}
template <typename XT, typename VT>
constexpr bool can_fix() { return sizeof(XT) == 8 && sizeof(VT) == 1; }
// Where a launch may take fixed-point steps. The integers of the whole iterate and the rows' tests cost 0.4 to 1 us
// per step (400 to 5000 spins); FP64 sums cost more where more than half of the SMs are busy. us per step, fixed
// point / FP64 sums, by entries a row:
//   R = 8, K = 16, 800 spins: 6 2.9 / 2.0, 9 2.2 / 2.3, 32 2.6 / 2.9, 48 2.7 / 3.4; 1500 spins: 9 2.6 / 3.2, 32 3.3 / 4.3
//   R = 20, K = 7, 800 spins: 6 2.7 / 2.3, 9 2.8 / 3.0, 32 3.7 / 4.4; 5000 spins, R = 8: 9 5.8 / 5.2, 20 6.6 / 6.7, 32 7.7 / 8.2
//   R = 4, K = 16 (64 CTAs), 1200 spins: 32 2.6 / 2.5; 2500 spins: 32 4.5 / 3.8; R = 1, 1200 spins: 72 3.1 / 3.3
//   shares of 34 rows (400 spins, R = 8, K = 12): 16 1.9 / 1.7, 32 2.0 / 1.9
template <typename XT, typename VT>
bool fixed_point(const ising_context *c, int R, const SmallRecord &rec, int K) {
    const int64_t ctas = static_cast<int64_t>(c->n_inst) * R * K, chunk = (c->max_inst_n + K - 1) / K;
    const int64_t entries = 2 * ctas <= c->num_sms || chunk < 48 ? 40 : chunk <= 256 ? 9 : 20;
    return can_fix<XT, VT>() && K > 1 && !rec.base && c->nnz >= entries * c->n;
}

template <typename XT, typename VT>
constexpr int64_t entry_bytes() { return sizeof(typename Held<XT, VT>::type) + sizeof(uint16_t); }

template <typename XT, typename VT, int P>
__global__ void __launch_bounds__(1024)
csr_small(const XT *x_in, XT *x_out, const int64_t *__restrict__ row_ptr,
          const int32_t *__restrict__ col, const VT *__restrict__ val, const XT *__restrict__ h,
          const int64_t *__restrict__ inst_off, int64_t n, int R, const double *__restrict__ alpha_tab, int alpha_len,
          const double *__restrict__ beta_tab, int k0, int iters, int K, int rows_cap, int cap,
          int fix, unsigned char *rec, size_t rec_stride, int rec_every, int *__restrict__ err) {
    extern __shared__ __align__(16) unsigned char small_smem[];
    __shared__ Exchange ex;
    constexpr bool kFix = can_fix<XT, VT>();
    __shared__ int rowabs_of[kFix ? 16 : 1];          // every CTA's largest row sum of |J| (INT_MAX: no fixed point)
    __shared__ unsigned top_word[kFix ? 3 : 1];       // upper words of max |x|, max |h|; the share's rowabs
    const int q = static_cast<int>(cl_rank());
    const int b = blockIdx.y, r = blockIdx.x / K;
    const int64_t lo = inst_off ? inst_off[b] : 0;
    const int64_t hi = inst_off ? inst_off[b + 1] : n;
    const int nb = static_cast<int>(hi - lo);
    const int chunk = (nb + K - 1) / K;  // <= rows_cap
    const int i0 = min(nb, q * chunk), i1 = min(nb, i0 + chunk), rows = i1 - i0;
    const int owners = (nb + chunk - 1) / chunk;  // CTAs with rows: 0 .. owners - 1
    XT *cur = reinterpret_cast<XT *>(small_smem), *nxt = cur + nb;
    XT *z = nxt + nb;
    using Hd = Held<XT, VT>;
    const bool may_fix = kFix && fix;
    long long *fx = reinterpret_cast<long long *>(P > 1 ? z + rows_cap : z);
    int *limit = reinterpret_cast<int *>(fx + nb);  // of a row: rowabs_i, negative while its sum is an FP64 one
    typename Hd::type *lv = may_fix ? reinterpret_cast<typename Hd::type *>(limit + rows_cap)
                                    : reinterpret_cast<typename Hd::type *>(fx);
    int *lr = reinterpret_cast<int *>(lv + cap);
    uint16_t *lc = reinterpret_cast<uint16_t *>(lr + rows_cap + 1);
    if constexpr (kFix) {
        if (threadIdx.x < 3) top_word[threadIdx.x] = 0;
        __syncthreads();
        unsigned tx = 0, th = 0;
        for (int i = threadIdx.x; i < nb; i += blockDim.x) {
            const XT v = x_in[(lo + i) * R + r];
            cur[i] = v;
            tx = max(tx, static_cast<unsigned>(__double2hiint(v)) & 0x7fffffffu);
            if (h) th = max(th, static_cast<unsigned>(__double2hiint(__ldg(h + lo + i))) & 0x7fffffffu);
        }
        atomicMax(&top_word[0], tx);
        atomicMax(&top_word[1], th);
    } else {
        for (int i = threadIdx.x; i < nb; i += blockDim.x) cur[i] = x_in[(lo + i) * R + r];
    }
    const int64_t e0 = row_ptr[lo + i0];
    const bool local = row_ptr[lo + i1] - e0 <= cap;  // uniform over the block
    for (int i = threadIdx.x; i <= rows && local; i += blockDim.x) lr[i] = static_cast<int>(row_ptr[lo + i0 + i] - e0);
    if (local) {
        const int cnt = static_cast<int>(row_ptr[lo + i1] - e0);
        for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
            lv[e] = Hd::pack(val[e0 + e]);
            lc[e] = static_cast<uint16_t>(col[e0 + e] - lo);
        }
    }
    bool fixed = false;
    float bound = 0.f, rowabs = 0.f, hmax = 0.f, inv_beta = 0.f;
    if constexpr (kFix) {
        __syncthreads();
        int sum = 0;
        for (int i = threadIdx.x; i < rows && local; i += blockDim.x) {
            int t = 0;
            for (int e = lr[i]; e < lr[i + 1]; ++e) t += abs(lv[e]);
            if (may_fix) limit[i] = t;
            sum = max(sum, t);
        }
        atomicMax(&top_word[2], static_cast<unsigned>(sum));
        if (K > 1) cl_sync();  // every CTA of the cluster runs
        else __syncthreads();
        if (threadIdx.x < K) {
            const int mine = local ? static_cast<int>(top_word[2]) : 0x7fffffff;
            asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cl_map(&rowabs_of[q], threadIdx.x)), "r"(mine) : "memory");
        }
        if (K > 1) cl_sync();
        else __syncthreads();
        int most = 1;
        for (int t = 0; t < K; ++t) most = max(most, rowabs_of[t]);
        // bounds just above the maxima; FP32 carries them, so their range and the scales' is checked, at
        // the start and at the point that the bounds move towards
        const double mx = __hiloint2double(static_cast<int>(top_word[0] + 1), 0);
        const double mh = top_word[1] ? __hiloint2double(static_cast<int>(top_word[1] + 1), 0) : 0.0;
        bound = __double2float_ru(mx);
        hmax = __double2float_ru(mh);
        rowabs = static_cast<float>(most) * 1.0001f;
        inv_beta = static_cast<float>(1.0 / beta_tab[b]) * 1.0001f;
        bool bad = !(may_fix && top_word[0] < 0x7ff00000u && top_word[1] < 0x7ff00000u && most < kRowLimit &&
                     bound > 1e-12f && bound < 1e10f && hmax < 1e12f && inv_beta > 1e-20f && inv_beta < 1e12f);
        for (int k = threadIdx.x; k < (alpha_len == 1 ? 1 : iters); k += blockDim.x) {
            const float ak = static_cast<float>(alpha_tab[static_cast<int64_t>(b) * alpha_len + (alpha_len == 1 ? 0 : k0 + k)]);
            const float z = (rowabs + fabsf(ak)) * inv_beta;  // without a field the squared bound tends to z
            bad = bad || !(z > 1e-20f && z < 1e12f);
        }
        fixed = !__syncthreads_or(bad);
        if (!fixed && local) {
            const int cnt = lr[rows];
            for (int e = threadIdx.x; e < cnt; e += blockDim.x) lv[e] = Hd::upper(lv[e]);
        }
    }
    const auto root = make_root<XT>(beta_tab[b]);
    const double *arow = alpha_tab + static_cast<int64_t>(b) * alpha_len;
    const int sub = threadIdx.x % P;
    const int rl = threadIdx.x / P, rstep = blockDim.x / P;
    const int top = (rows + rstep - 1) / rstep * rstep;  // whole warps take part in the shuffles
    exchange_init(ex);
    // every CTA of the cluster runs, and has loaded, before the first remote store
    if (K > 1) cl_sync();
    else __syncthreads();
    for (int k = 0; k < iters && rows > 0; ++k) {
        const XT a = static_cast<XT>(arow[alpha_len == 1 ? 0 : k0 + k]);
        if (owners > 1) exchange_expect(ex, k, static_cast<uint32_t>((nb - rows) * sizeof(XT)));
        const bool keep = rec && (k + 1) % rec_every == 0;
        XT *rp = reinterpret_cast<XT *>(rec + (keep ? static_cast<size_t>((k + 1) / rec_every - 1) : 0) * rec_stride);
        double unit = 0.0;
        if constexpr (kFix) {
            if (fixed) {
                const int shift = fixed_shift(bound, rowabs);
                unit = two_to(-shift);
                bound = next_bound(bound, rowabs, static_cast<float>(a), hmax, inv_beta);
                for (int i = threadIdx.x; i < nb; i += blockDim.x) fx[i] = to_fixed(cur[i], shift);
                __syncthreads();
            }
        }
        // row i of the share: the new value into every CTA's next copy; u is J x, as the integer's bits (in_fixed) or FP64
        auto update = [&](int i, XT u, bool in_fixed) {
            const int64_t row = lo + i0 + i;
            const XT hv = h ? __ldg(h + row) : XT(0);
            XT v;
            if (kFix && in_fixed) {
                if constexpr (kFix) {
                    XT w = a * cur[i0 + i];
                    if (h) w += hv;
                    v = root_newton(fma(__ll2double_rn(__double_as_longlong(u)), unit, w), root);
                }
            } else {
                v = root_newton(u + a * cur[i0 + i] + hv, root);
                if (keep) rp[row * R + r] = v;
            }
            nxt[i0 + i] = v;
            exchange_send(ex, k, nxt + i0 + i, v, q, owners);
        };
        for (int i = rl; i < top; i += rstep) {
            XT acc = XT(0);
            bool in_fixed = false;
            if (kFix && fixed) {
                if constexpr (kFix) {
                    long long sum = 0;
                    unsigned mag = 0;  // sum of |J_ij| |upper word of x_j|, above the true magnitudes by at most rowabs_i
                    int f0 = 0, f1 = 0, most = 0;
                    if (i < rows) {
                        f0 = lr[i] + sub;
                        f1 = lr[i + 1];
                        most = limit[i];
#pragma unroll 4
                        for (int e = f0; e < f1; e += P) {
                            const int w = lv[e];
                            const long long x = fx[lc[e]];
                            sum += static_cast<long long>(w) * x;
                            mag += static_cast<unsigned>(abs(w * static_cast<int>(x >> 32)));
                        }
                    }
#pragma unroll
                    for (int o = P / 2; o > 0; o >>= 1) {
                        sum += __shfl_xor_sync(0xffffffffu, sum, o);
                        mag += __shfl_xor_sync(0xffffffffu, mag, o);
                    }
                    in_fixed = most == 0 || (mag >> 20) > static_cast<unsigned>(most);
                    if (__any_sync(0xffffffffu, !in_fixed)) {  // the rows that fail, in FP64
                        if (!in_fixed)
                            for (int e = f0; e < f1; e += P) acc += static_cast<double>(lv[e]) * cur[lc[e]];
#pragma unroll
                        for (int o = P / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                        if (P > 1 && !in_fixed && sub == 0) limit[i] = -most;
                    }
                    if (in_fixed) acc = __longlong_as_double(sum);
                }
            } else if (i < rows) {
                if (local) {
                    const int f1 = lr[i + 1];
#pragma unroll 4
                    for (int e = lr[i] + sub; e < f1; e += P) acc += Hd::value(lv[e]) * cur[lc[e]];
                } else {
                    const int64_t f1 = __ldg(row_ptr + lo + i0 + i + 1);
                    for (int64_t e = __ldg(row_ptr + lo + i0 + i) + sub; e < f1; e += P)
                        acc += static_cast<XT>(__ldg(val + e)) * cur[__ldg(col + e) - lo];
                }
            }
            if (!(kFix && fixed)) {
#pragma unroll
                for (int o = P / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            }
            if (P == 1) {
                if (i < rows) update(i, acc, in_fixed);
            } else if (sub == 0 && i < rows) {
                z[i] = acc;
            }
        }
        if (P > 1) {
            __syncthreads();
            for (int i = threadIdx.x; i < rows; i += blockDim.x) {
                bool in_fixed = kFix && fixed;
                if (in_fixed && limit[i] < 0) {
                    in_fixed = false;
                    limit[i] = -limit[i];
                }
                update(i, z[i], in_fixed);
            }
        }
        if (!exchange_wait(ex, k, owners, err)) break;
        XT *t = cur;
        cur = nxt;
        nxt = t;
    }
    if (x_out)
        for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) x_out[(lo + i) * R + r] = cur[i];
    if (K > 1) cl_sync();  // no CTA leaves while a peer may still send to it
}

// Adjoint steps k0 + len - 1 .. k0 of one instance that fits in shared memory, in one launch: with
// the adjoint state w^k held as csr_small holds its iterate, a cluster per replica and a thread per row,
//   g^k = (J w^k + alpha_k w^k) / beta,   w^(k-1) = g^k / (3 (x^k)^2)  (g^0 itself when k = 0),
// and the partial sums of dL/dalpha_k = sum w^k x^k / beta of every CTA into part[k][CTA]. Within a
// gradient the state has the iterate's type, between segments too (the result does not depend on the
// checkpoint interval): FP64 for FP64 iterates (few rows per CTA, so the latency of the
// chain counts and not the FP64 rate: 7 % of the issue slots, 22 % of the FP64 pipe active, four warps per
// SM, 2000 spins, R = 8, 4 us per step; the factor 1 / (3 x^2) is formed before the wait for the peers' shares); FP32
// with compensated row sums for FP32 ones. The products
// w x (FP64, or FP32 split exactly) stay in shared memory for up to `hold` steps, and are then added in FP64,
// a warp per step: added at every step they were a third of it. x^(k0) is x_first and
// x^(k0 + m) = x_seg + (m - 1) stride, each loaded a step ahead. Every CTA of a cluster owns rows here:
// K <= 16 and n >= 32 K (cluster_max) leave the last share at least 17.
template <typename XT>
struct AdjointRow;
template <>
struct AdjointRow<float> {
    float ib_hi, ib_lo, x;  // 1 / beta as a float and its remainder: its rounding would be the same at every step
    __device__ __forceinline__ explicit AdjointRow(double beta) : x(0.f) {
        const double ib = 1.0 / beta;
        ib_hi = static_cast<float>(ib);
        ib_lo = static_cast<float>(ib - ib_hi);
    }
    __device__ __forceinline__ void set(float x_) { x = x_; }
    template <typename F>
    __device__ __forceinline__ float sum(double alpha, float w, int e0, int e1, F &&term) const {
        const float a_hi = static_cast<float>(alpha), a_lo = static_cast<float>(alpha - a_hi);
        DotSum32 acc;
        acc.add(a_lo * w);
        acc.add(a_hi, w);
#pragma unroll 4
        for (int e = e0; e < e1; ++e) term(e, [&](float v, float wj) { acc.add(v, wj); });
        const float z = acc.s - acc.c;
        return fmaf(z, ib_lo, z * ib_hi);
    }
    using Product = float2;  // rounded product and its error
    static __device__ __forceinline__ float2 product(float a, float b) {
        const float p = __fmul_rn(a, b);
        return make_float2(p, fmaf(a, b, -p));
    }
    static __device__ __forceinline__ double value(float2 p) { return static_cast<double>(p.x) + static_cast<double>(p.y); }
    __device__ __forceinline__ float weigh(float g) const { return x == 0.0f ? 0.0f : g / (3.0f * x * x); }
};
template <>
struct AdjointRow<double> {
    double ib, factor;  // factor = 1 / (3 x^2)
    __device__ __forceinline__ explicit AdjointRow(double beta) : ib(1.0 / beta), factor(0.0) {}
    __device__ __forceinline__ void set(double x) {
        const double d = 3.0 * x * x;
        const float df = static_cast<float>(d);
        if (df > 1e-30f && df < 1e30f) {  // one Newton step from the FP32 reciprocal: within (2^-23)^2 = 1.4e-14
            double r = static_cast<double>(1.0f / df);
            r = fma(r, fma(-d, r, 1.0), r);
            factor = r;
        } else {
            factor = d == 0.0 ? 0.0 : 1.0 / d;
        }
    }
    template <typename F>
    __device__ __forceinline__ double sum(double alpha, double w, int e0, int e1, F &&term) const {
        double acc = alpha * w;
#pragma unroll 4
        for (int e = e0; e < e1; ++e) term(e, [&](double v, double wj) { acc += v * wj; });
        return acc * ib;
    }
    using Product = double;
    static __device__ __forceinline__ double product(double a, double b) { return a * b; }
    static __device__ __forceinline__ double value(double p) { return p; }
    __device__ __forceinline__ double weigh(double g) const { return g * factor; }
};

// bytes before the held products: cur | nxt (XT [n] each) | couplings (XT [cap]) | row ranges (int [rows + 1]) |
// columns (uint16 [cap])
template <typename XT>
constexpr int64_t adjoint_held_at(int64_t n, int64_t rows, int64_t cap) {
    return (static_cast<int64_t>(sizeof(XT)) * (2 * n + cap) + 4 * (rows + 1) + 2 * cap + 15) / 16 * 16;
}

template <typename XT, typename VT>
__global__ void __launch_bounds__(1024)
adjoint_small(const XT *w_in, XT *w_out, const XT *__restrict__ x_first, const unsigned char *__restrict__ x_seg,
              size_t stride, const int64_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
              const VT *__restrict__ val, int n, int R, const double *__restrict__ alpha_tab,
              const double *__restrict__ beta_tab, int k0, int len, int K, int rows_cap, int cap, int hold,
              double *__restrict__ part, unsigned long long *__restrict__ zeros, int *__restrict__ err) {
    extern __shared__ __align__(16) unsigned char small_smem[];
    __shared__ Exchange ex;
    const int q = static_cast<int>(cl_rank());
    const int r = blockIdx.x / K;
    const int i0 = min(n, q * rows_cap), rows = min(n, i0 + rows_cap) - i0;
    XT *cur = reinterpret_cast<XT *>(small_smem), *nxt = cur + n, *lv = nxt + n;
    using Product = typename AdjointRow<XT>::Product;
    Product *held = reinterpret_cast<Product *>(small_smem + adjoint_held_at<XT>(n, rows_cap, cap));
    int *lr = reinterpret_cast<int *>(lv + cap);
    uint16_t *lc = reinterpret_cast<uint16_t *>(lr + rows_cap + 1);
    for (int i = threadIdx.x; i < n; i += blockDim.x) cur[i] = w_in[static_cast<int64_t>(i) * R + r];
    const int64_t e0 = row_ptr[i0];
    const int cnt = static_cast<int>(row_ptr[i0 + rows] - e0);  // <= cap
    for (int i = threadIdx.x; i <= rows; i += blockDim.x) lr[i] = static_cast<int>(row_ptr[i0 + i] - e0);
    for (int e = threadIdx.x; e < cnt; e += blockDim.x) {
        lv[e] = static_cast<XT>(val[e0 + e]);
        lc[e] = static_cast<uint16_t>(col[e0 + e]);
    }
    auto iterate = [&](int m) {
        return m == 0 ? x_first : reinterpret_cast<const XT *>(x_seg + static_cast<size_t>(m - 1) * stride);
    };
    const int64_t at = static_cast<int64_t>(i0 + threadIdx.x) * R + r;  // the thread's row (rows <= blockDim.x)
    const bool has = threadIdx.x < rows;
    const int own = i0 + static_cast<int>(threadIdx.x);
    XT x_own = has ? iterate(len - 1)[at] : XT(0), x_next = has && len > 1 ? iterate(len - 2)[at] : XT(0);
    AdjointRow<XT> row(beta_tab[0]);
    row.set(x_own);
    unsigned nz = 0;
    exchange_init(ex);
    if (K > 1) cl_sync();
    else __syncthreads();
    for (int m = len - 1; m >= 0; --m) {
        const int k = k0 + m;
        const double ad = __ldg(alpha_tab + k);
        const int s = len - 1 - m;
        if (K > 1 && m > 0) exchange_expect(ex, s, static_cast<uint32_t>((n - rows) * sizeof(XT)));
        if (has) {
            const XT wi = cur[own];
            const XT g = row.sum(ad, wi, lr[threadIdx.x], lr[threadIdx.x + 1],
                                 [&](int e, auto &&add) { add(lv[e], cur[lc[e]]); });
            XT out = g;
            if (k > 0) {
                nz += x_own == XT(0);
                out = row.weigh(g);
            }
            if (m == 0) {
                w_out[at] = out;
            } else {
                nxt[own] = out;
                exchange_send(ex, s, nxt + own, out, q, K);
            }
            held[(s % hold) * rows_cap + threadIdx.x] = AdjointRow<XT>::product(wi, x_own);
        }
        x_own = x_next;
        row.set(x_own);
        if (has && m > 1) x_next = iterate(m - 2)[at];
        if (s % hold == hold - 1 || m == 0) {  // the held steps' sums: k + (s % hold) .. k
            __syncthreads();
            for (int t = threadIdx.x / 32; t <= s % hold; t += blockDim.x / 32) {
                double ga = 0.0;
                for (int i = threadIdx.x % 32; i < rows; i += 32) ga += AdjointRow<XT>::value(held[t * rows_cap + i]);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) ga += __shfl_xor_sync(0xffffffffu, ga, o);
                if (threadIdx.x % 32 == 0)
                    part[static_cast<int64_t>(k + s % hold - t) * gridDim.x + blockIdx.x] = ga;
            }
            __syncthreads();
        }
        if (m > 0 && !exchange_wait(ex, s, K, err)) break;
        XT *t = cur;
        cur = nxt;
        nxt = t;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nz += __shfl_xor_sync(0xffffffffu, nz, o);
    if (threadIdx.x % 32 == 0 && nz) atomicAdd(zeros, static_cast<unsigned long long>(nz));
    if (K > 1) cl_sync();  // no CTA leaves while a peer may still send to it
}

// the largest cluster size worth trying: each CTA keeps at least 32 rows and all pairs' clusters have
// an SM per CTA
int cluster_max(const ising_context *c, int R) {
    const int64_t pairs = static_cast<int64_t>(c->n_inst) * R;
    return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>({16, c->num_sms / pairs, c->max_inst_n / 32})));
}

// One instance whose average share of couplings does not fit: here, the couplings read from L2 row by row, or
// single steps? A single step costs about 0.19 us per entry of a row in FP32, 0.26 in FP64 and 0.32 in FP64 with two
// replicas per thread (even R), nearly whatever the number of rows; here it is about 0.95 ns per entry of a
// share while few CTAs read (1.3 with 128 of them). us per step, here / single steps, K = 16:
//   FP64, 3000 spins of 110 entries: R = 1 18.4 / 28.7, R = 4 18.4 / 35.1, R = 8 24.6 / 34.9 (R = 9: 30.0 / 26.7)
//   FP64, 5000 spins of 80: R = 1 24.8 / 22.7, R = 2 25.0 / 30.5, R = 6 25.1 / 28.8, R = 8 33.6 / 28.7
//   FP64, 8000 spins of 50: R = 1 28.4 / 16.5, R = 4 28.4 / 22.0
//   FP32, 5000 spins of 110: R = 1 30.2 / 20.6, R = 4 30.7 / 22.6, R = 8 40.7 / 20.6; 2000 of 110, R = 16, K = 9: 33.3 / 18.5
template <typename XT>
bool from_l2(const ising_context *c, int R, int K) {
    return sizeof(XT) == 8 && static_cast<int64_t>(R) * K <= 128 && c->n * R <= 32768 &&
           (c->n + K - 1) / K <= (R % 2 == 0 ? 320 : 256);
}

template <typename XT, typename VT, int P>
ising_status_t launch_k(const ising_context *c, const XT *x_in, XT *x_out, int R, const XT *h, const ParamTabs &p,
                        int k0, int iters, int K, const SmallRecord &rec, int64_t optin, cudaStream_t st) {
    const int64_t chunk = (c->max_inst_n + K - 1) / K;
    const bool fix = fixed_point<XT, VT>(c, R, rec, K);
    const int64_t state = state_bytes<XT, P>(c->max_inst_n, chunk, fix);
    if (state > optin) return ISING_ERR_UNSUPPORTED;
    // room for the couplings of the fullest share, as far as it goes (shares that need more read the CSR arrays)
    const int64_t left = optin - state - static_cast<int64_t>(sizeof(int)) * (chunk + 1);
    if (c->n_inst == 1 && left / entry_bytes<XT, VT>() < (c->nnz + c->nnz / 16) / K && !from_l2<XT>(c, R, K))
        return ISING_ERR_UNSUPPORTED;
    const int64_t need = std::min(c->max_row_nnz * chunk, c->nnz);
    const int64_t cap = left <= 0 ? -1 : std::min(left / entry_bytes<XT, VT>() / 4 * 4, (need + 3) / 4 * 4);
    const int smem = static_cast<int>(cap < 0 ? state : optin - left + cap * entry_bytes<XT, VT>());
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
        if (cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg) != cudaSuccess || nclusters < R * c->n_inst) {
            cudaGetLastError();
            return ISING_ERR_UNSUPPORTED;
        }
    }
    DOCH_CUDA(cudaLaunchKernelEx(&cfg, kern, x_in, x_out, static_cast<const int64_t *>(c->row_ptr),
                                 static_cast<const int32_t *>(c->col), static_cast<const VT *>(c->val), h,
                                 static_cast<const int64_t *>(c->n_inst > 1 ? c->inst_off : nullptr), c->n, R,
                                 p.alpha_d, p.alpha_len, p.beta_d, k0, iters, K, static_cast<int>(chunk),
                                 static_cast<int>(cap), fix ? 1 : 0, static_cast<unsigned char *>(rec.base), rec.stride,
                                 rec.every, c->err_word));
    return ISING_OK;
}

// room for the couplings of the fullest share of a cluster of K CTAs
int64_t adjoint_cap(const ising_context *c, int K) {
    const int64_t chunk = (c->n + K - 1) / K;
    return (std::min(c->max_row_nnz * chunk, c->nnz) + 3) / 4 * 4;
}

template <typename XT, typename VT>
ising_status_t adjoint_config(const ising_context *c, int R, const AdjointPlan &plan, cudaLaunchConfig_t &cfg,
                              cudaLaunchAttribute *attr) {
    const int n = static_cast<int>(c->n), chunk = (n + plan.K - 1) / plan.K;
    const int64_t smem = adjoint_held_at<XT>(n, chunk, adjoint_cap(c, plan.K)) + plan.hold * 8LL * chunk;
    auto kern = adjoint_small<XT, VT>;
    DOCH_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)));
    if (plan.K > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        return ISING_ERR_UNSUPPORTED;
    }
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(plan.K);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(static_cast<unsigned>(R * plan.K));
    cfg.blockDim = dim3(static_cast<unsigned>(std::min(1024, (chunk + 31) / 32 * 32)));
    cfg.dynamicSmemBytes = static_cast<size_t>(smem);
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return ISING_OK;
}

// The largest cluster whose shares fit and whose copies for all replicas run at once
template <typename XT, typename VT>
ising_status_t adjoint_plan(const ising_context *c, int R, int iters, int64_t optin, AdjointPlan &plan) {
    for (plan.K = cluster_max(c, R); plan.K >= 1; --plan.K) {
        const int n = static_cast<int>(c->n), chunk = (n + plan.K - 1) / plan.K;
        const int64_t left = optin - adjoint_held_at<XT>(n, chunk, adjoint_cap(c, plan.K)), step = 8LL * chunk;
        if (left < step || chunk > 1024) continue;
        plan.hold = static_cast<int>(std::min<int64_t>({iters, 32, left / step}));
        plan.parts = R * plan.K;
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        const ising_status_t s = adjoint_config<XT, VT>(c, R, plan, cfg, attr);
        if (s == ISING_ERR_UNSUPPORTED) continue;
        DOCH_CHECK(s);
        if (plan.K == 1) return ISING_OK;
        int nclusters = 0;
        if (cudaOccupancyMaxActiveClusters(&nclusters, adjoint_small<XT, VT>, &cfg) == cudaSuccess && nclusters >= R)
            return ISING_OK;
        cudaGetLastError();
    }
    return ISING_ERR_UNSUPPORTED;
}

template <typename XT, typename VT>
ising_status_t launch_adjoint(const ising_context *c, const AdjointPlan &plan, const AdjointSegment &s, int R,
                              const ParamTabs &p, cudaStream_t st) {
    const int n = static_cast<int>(c->n), chunk = (n + plan.K - 1) / plan.K;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    DOCH_CHECK((adjoint_config<XT, VT>(c, R, plan, cfg, attr)));
    cfg.stream = st;
    DOCH_CUDA(cudaLaunchKernelEx(&cfg, adjoint_small<XT, VT>, static_cast<const XT *>(s.w_in), static_cast<XT *>(s.w_out),
                                 static_cast<const XT *>(s.x_first), static_cast<const unsigned char *>(s.x_seg), s.stride,
                                 static_cast<const int64_t *>(c->row_ptr), static_cast<const int32_t *>(c->col),
                                 static_cast<const VT *>(c->val), n, R, p.alpha_d, p.beta_d, s.k0, s.len, plan.K, chunk,
                                 static_cast<int>(adjoint_cap(c, plan.K)), plan.hold, s.part, s.zeros, c->err_word));
    return ISING_OK;
}

// f(XT(), VT()) for the types of the iterates and the couplings
template <typename F>
ising_status_t adjoint_types(const ising_context *c, int xtype, F &&f) {
    auto couplings = [&](auto x) -> ising_status_t {
        switch (c->jtype) {
            case ISING_I8: return f(x, int8_t());
            case ISING_I32: return f(x, int32_t());
            case ISING_F32: return f(x, float());
            case ISING_F64: return f(x, double());
            default: return fail(ISING_ERR_UNSUPPORTED, "backward: coupling type");
        }
    };
    return xtype == ISING_F64 ? couplings(double()) : couplings(float());
}

template <typename XT, typename VT>
ising_status_t launch_small(const ising_context *c, const XT *x_in, XT *x_out, int R, const XT *h, const ParamTabs &p,
                            int k0, int iters, const SmallRecord &rec, cudaStream_t st) {
    int dev = 0, optin = 0;
    DOCH_CUDA(cudaGetDevice(&dev));
    DOCH_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    optin -= kStaticSmem;
    // the largest cluster whose copies for all pairs run at once (a cluster lies within one GPU processing
    // cluster, so sizes that fill those badly drop out): 1500 spins at density 0.08, R = 20, FP64: 6 CTAs
    // per pair
    for (int K = cluster_max(c, R);; --K) {
        const int64_t chunk = (c->max_inst_n + K - 1) / K;
        // threads per row: four or two where a share is small and its rows are long enough to split (more
        // would spend as many FP64 additions on the tree as they take from the rows); eight or four where
        // the products are integers (us per step with four / eight / sixteen: 1000 spins at density 0.05, R = 20,
        // shares of 143 rows 4.7 / 4.2 / 4.7; 800 spins at 0.06, R = 8, shares of 50 3.0 / 2.7 / 3.4)
        const bool split = c->nnz >= 8 * c->n;
        auto run = [&](auto p_threads) {
            return launch_k<XT, VT, decltype(p_threads)::value>(c, x_in, x_out, R, h, p, k0, iters, K, rec, optin, st);
        };
        ising_status_t s;
        if (fixed_point<XT, VT>(c, R, rec, K))
            s = split && chunk <= 256   ? run(std::integral_constant<int, 8>())
                : split && chunk <= 512 ? run(std::integral_constant<int, 4>())
                                        : run(std::integral_constant<int, 1>());
        else
            s = split && chunk <= 128   ? run(std::integral_constant<int, 4>())
                : split && chunk <= 512 ? run(std::integral_constant<int, 2>())
                                        : run(std::integral_constant<int, 1>());
        if (s != ISING_ERR_UNSUPPORTED || K == 1) return s;
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

// The adjoint's forward steps and adjoint steps run here for instances of at most 2048 spins with at
// least four CTAs per replica; larger ones take single steps, whose launches overlap and whose adjoint state
// is FP32. Every new value is stored into all CTAs, 13 clocks a warp, so that many rows per CTA lose. Shared
// memory / single steps, ms per gradient of 100 FP64 steps, checkpoints every 10, degree 3: 2000 spins, R = 8 1.45 / 1.49,
// 2500 1.53 / 1.51 (R = 1 1.24 / 1.21, R = 16 1.67 / 1.56), 3000 1.63 / 1.53, 4000 1.80 / 1.53 (R = 16 2.06 / 1.65);
// degree 6: 2500 1.67 / 1.74, 4000 1.82 / 1.75. Relative error of grad_x0: 2e-8 to 1.2e-7 with the FP64 state, 0.7e-6 to
// 3.7e-6 with the FP32 one. FP32, 60 steps: 1000 spins, R = 16 0.76 / 0.87, 2000 spins, R = 8 0.87 / 0.86, 6000
// spins 1.10 / 0.88.
bool backward_small(const ising_context *c, int xtype, int R) {
    return c->n_inst == 1 && c->n <= 2048 && static_cast<size_t>(c->n) <= csr_fused_max_spins(xtype) &&
           cluster_max(c, R) >= 4;
}

int adjoint_small_parts(const ising_context *c, int R) { return R * cluster_max(c, R); }

ising_status_t adjoint_small_plan(const ising_context *c, int xtype, int R, int iters, AdjointPlan &plan) {
    int dev = 0, optin = 0;
    DOCH_CUDA(cudaGetDevice(&dev));
    DOCH_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    optin -= kStaticSmem;
    if (c->n_inst != 1 || c->n > 65536) return ISING_ERR_UNSUPPORTED;
    return adjoint_types(c, xtype, [&](auto x, auto v) {
        return adjoint_plan<decltype(x), decltype(v)>(c, R, iters, optin, plan);
    });
}

ising_status_t adjoint_small_run(const ising_context *c, const AdjointPlan &plan, const AdjointSegment &s, int xtype,
                                 int R, const ParamTabs &p, cudaStream_t st) {
    return adjoint_types(c, xtype, [&](auto x, auto v) {
        return launch_adjoint<decltype(x), decltype(v)>(c, plan, s, R, p, st);
    });
}

ising_status_t csr_fused(const ising_context *c, void *x, int xtype, int R, const ParamTabs &p, int iters,
                         cudaStream_t st) {
    return csr_small_run(c, x, x, xtype, R, p, 0, iters, SmallRecord{}, st);
}

}  // namespace doch
