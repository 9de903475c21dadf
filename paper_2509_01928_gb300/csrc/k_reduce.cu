// Readout reductions: sign rounding (Algorithm 1, return step; sign(0) = +1),
// the Ising energy E = -1/2 s^T J s - h^T s (Eq. IsingModel), the cut value
// cut = 1/4 sum_ij (1 - s_i s_j) W_ij with W = -2J (Supplementary Note 5),
// the Hamiltonian H(x) of Eq. Hamilton (plus -h^T x), and argmin_r E_r.
//
// Every reduction runs over rows x replicas: a thread owns a row and a chunk of V
// consecutive replicas (V = 16 bytes of x, or 1), so the threads of a row share its
// couplings and read whole sectors of each neighbour's replicas. A block sums the
// rows of one chunk of one instance and writes one partial per (replica, chunk),
// its threads added in a fixed tree; a second kernel (one warp per (instance,
// replica)) adds the chunk partials in a fixed order. Integer couplings accumulate
// in int64 (exact); real couplings in FP64 with that fixed order, so results are
// identical run to run.
//
// Energies: per row, D = sum of J_ij over the j whose spin differs from spin i and
// S = sum_j J_ij, so that sum_j J_ij s_i s_j = S - 2 D and sum_j J_ij (1 - s_i s_j)
// = 2 D: one predicated addition per entry and replica (FP64 additions run at 2 lanes
// per clock and SM here, and so do FP32 -> FP64 conversions, which are done on the
// integer pipe). Readout of 128 instances of up to 20,000 spins, R = 16, Gaussian
// couplings: 1.72 ms with one replica per block and a thread per row, 0.74 ms now (FP64
// additions); of the 10^5-spin, 10^7-entry integer matrix, R = 16: 1.15 ms and 0.11 ms
// (gathers from L2); of a lattice of 10^8 sites, R = 1: 0.48 ms and 0.10 ms (HBM).
// E = -acc0/2 - acc2 and cut = -acc1/2 from the sums over all rows of
// acc0 = s_i sum_j J_ij s_j, acc1 = sum_j J_ij (1 - s_i s_j), acc2 = h_i s_i.
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "internal.cuh"

namespace doch {
namespace {

constexpr int kRThreads = 256;

template <typename XT>
__device__ __forceinline__ int spin_of(XT v) {
    if constexpr (sizeof(XT) == 2) return __bfloat162float(v) >= 0.f ? 1 : -1;
    else return v >= XT(0) ? 1 : -1;
}

template <typename XT>
__device__ __forceinline__ double as_double(XT v) {
    if constexpr (sizeof(XT) == 2) return static_cast<double>(__bfloat162float(v));
    else return static_cast<double>(v);
}

template <typename Acc>
__device__ __forceinline__ Acc warp_sum(Acc v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// V consecutive values of x as their own type: one load of up to 16 bytes
template <typename XT, int V>
struct alignas(sizeof(XT) * V) Pack {
    XT v[V];
};
template <typename XT, int V>
__device__ __forceinline__ Pack<XT, V> ldp(const XT *p) {
    return *reinterpret_cast<const Pack<XT, V> *>(p);
}

// FP32 -> FP64 by moving the exponent and mantissa fields (normal numbers; the rest by conversion)
__device__ __forceinline__ double widen(float f) {
    const unsigned u = __float_as_uint(f), e = (u >> 23) & 255u;
    if (e == 0u || e == 255u) return static_cast<double>(f);
    return __hiloint2double(static_cast<int>((u & 0x80000000u) | ((e + 896u) << 20) | ((u & 0x7fffffu) >> 3)),
                            static_cast<int>(u << 29));
}
template <typename Acc, typename VT>
__device__ __forceinline__ Acc weight(VT w) {
    if constexpr (std::is_same<Acc, double>::value && std::is_same<VT, float>::value) return widen(w);
    else if constexpr (std::is_same<Acc, double>::value && sizeof(VT) == 1) return w ? widen(static_cast<float>(w)) : 0.0;
    else return static_cast<Acc>(w);
}

// Fn::kGrid: rows are lattice sites; the functor also gets the (row, column) of site i,
// advanced without divisions.
template <int K, int V, typename Acc, typename Fn>
__global__ void __launch_bounds__(kRThreads)
row_reduce(Fn fn, const int64_t *__restrict__ inst_off, int64_t n, int R, int chunks,
           Acc *__restrict__ partials) {
    const int C = R / V, Cb = C < kRThreads ? C : kRThreads;  // replica chunks: all, of one block
    const int rows = kRThreads / Cb;                          // rows in flight per block
    const int rl = threadIdx.x / Cb;
    const int c = blockIdx.y * Cb + threadIdx.x % Cb;
    const bool active = rl < rows && c < C;
    const int ch = blockIdx.x, b = blockIdx.z;
    const int64_t lo = inst_off ? inst_off[b] : 0;
    const int64_t hi = inst_off ? inst_off[b + 1] : n;
    const int64_t len = hi - lo;
    const int64_t s0 = lo + len * ch / chunks, s1 = lo + len * (ch + 1) / chunks;
    Acc acc[V][K];
#pragma unroll
    for (int q = 0; q < V; ++q)
#pragma unroll
        for (int k = 0; k < K; ++k) acc[q][k] = Acc(0);
    if (active) {
        if constexpr (Fn::kGrid) {
            const int64_t dr = rows / fn.Lc, dc = rows - dr * fn.Lc;
            int64_t rr = (s0 + rl) / fn.Lc, cc = s0 + rl - rr * fn.Lc;
            for (int64_t i = s0 + rl; i < s1; i += rows) {
                fn(i, rr, cc, c * V, acc);
                rr += dr;
                cc += dc;
                if (cc >= fn.Lc) {
                    cc -= fn.Lc;
                    ++rr;
                }
            }
        } else {
            for (int64_t i = s0 + rl; i < s1; i += rows) fn(i, c * V, acc);
        }
    }
    __shared__ Acc red[K * V][kRThreads];
#pragma unroll
    for (int q = 0; q < V; ++q)
#pragma unroll
        for (int k = 0; k < K; ++k) red[q * K + k][threadIdx.x] = acc[q][k];
    __syncthreads();
    int top = 1;
    while (top < rows) top <<= 1;
    for (int h = top >> 1; h > 0; h >>= 1) {  // fixed tree over the block's rows
        if (active && rl < h && rl + h < rows) {
#pragma unroll
            for (int m = 0; m < K * V; ++m) red[m][threadIdx.x] += red[m][threadIdx.x + h * Cb];
        }
        __syncthreads();
    }
    if (active && rl == 0) {
#pragma unroll
        for (int q = 0; q < V; ++q)
#pragma unroll
            for (int k = 0; k < K; ++k)
                partials[((static_cast<int64_t>(b) * R + c * V + q) * chunks + ch) * K + k] =
                    red[q * K + k][threadIdx.x];
    }
}

// ---- energy functors -------------------------------------------------------

constexpr int kEB = 8;  // entries of a row whose loads are issued together

template <typename XT, typename VT, typename Acc, int V>
struct CsrEnergy {
    static constexpr bool kGrid = false;
    const XT *x;
    const int64_t *row_ptr;
    const int32_t *col;
    const VT *val;
    const Acc *h;
    int R;
    __device__ void operator()(int64_t i, int r0, Acc (&acc)[V][3]) const {
        const Pack<XT, V> xi = ldp<XT, V>(x + i * R + r0);
        bool up[V];
        Acc D[V], S = Acc(0);
#pragma unroll
        for (int q = 0; q < V; ++q) {
            up[q] = spin_of(xi.v[q]) > 0;
            D[q] = Acc(0);
        }
        const int64_t e1 = __ldg(row_ptr + i + 1);
        int64_t e = __ldg(row_ptr + i);
        for (; e + kEB <= e1; e += kEB) {
            int32_t js[kEB];
            VT ws[kEB];
#pragma unroll
            for (int t = 0; t < kEB; ++t) {
                js[t] = __ldg(col + e + t);
                ws[t] = __ldg(val + e + t);
            }
            Pack<XT, V> xj[kEB];
#pragma unroll
            for (int t = 0; t < kEB; ++t) xj[t] = ldp<XT, V>(x + static_cast<int64_t>(js[t]) * R + r0);
            if constexpr (sizeof(VT) == 1) {  // eight int8 values add up in 32 bits
                int s8 = 0, d8[V];
#pragma unroll
                for (int q = 0; q < V; ++q) d8[q] = 0;
#pragma unroll
                for (int t = 0; t < kEB; ++t) {
                    s8 += ws[t];
#pragma unroll
                    for (int q = 0; q < V; ++q) d8[q] += (spin_of(xj[t].v[q]) > 0) != up[q] ? static_cast<int>(ws[t]) : 0;
                }
                S += static_cast<Acc>(s8);
#pragma unroll
                for (int q = 0; q < V; ++q) D[q] += static_cast<Acc>(d8[q]);
            } else {
#pragma unroll
                for (int t = 0; t < kEB; ++t) {
                    const Acc w = weight<Acc>(ws[t]);
                    S += w;
#pragma unroll
                    for (int q = 0; q < V; ++q)
                        if ((spin_of(xj[t].v[q]) > 0) != up[q]) D[q] += w;
                }
            }
        }
        for (; e < e1; ++e) {
            const Pack<XT, V> xj = ldp<XT, V>(x + static_cast<int64_t>(__ldg(col + e)) * R + r0);
            const Acc w = weight<Acc>(__ldg(val + e));
            S += w;
#pragma unroll
            for (int q = 0; q < V; ++q)
                if ((spin_of(xj.v[q]) > 0) != up[q]) D[q] += w;
        }
        const Acc hv = h ? h[i] : Acc(0);
#pragma unroll
        for (int q = 0; q < V; ++q) {
            Acc a = S - (D[q] + D[q]), b = D[q] + D[q];
            if constexpr (std::is_same<Acc, double>::value)  // infinite or NaN couplings (unvalidated J)
                if ((__double2hiint(a) & 0x7ff00000) == 0x7ff00000) term_by_term(i, r0 + q, a, b);
            acc[q][0] += a;
            acc[q][1] += b;
            if (h) acc[q][2] += up[q] ? hv : -hv;
        }
    }
    // sum_j J_ij s_i s_j and sum_j J_ij (1 - s_i s_j) of one replica without the S - 2 D form
    __device__ __noinline__ void term_by_term(int64_t i, int r, Acc &a, Acc &b) const {
        const int si = spin_of(x[i * R + r]);
        a = b = Acc(0);
        for (int64_t e = row_ptr[i]; e < row_ptr[i + 1]; ++e) {
            const int ss = si * spin_of(x[static_cast<int64_t>(col[e]) * R + r]);
            a += static_cast<Acc>(val[e]) * static_cast<Acc>(ss);
            b += static_cast<Acc>(val[e]) * static_cast<Acc>(1 - ss);
        }
    }
};

// each lattice edge enters sum_{i,j} twice (J_ab and J_ba)
template <typename XT, int V>
struct TorusEnergy {
    static constexpr bool kGrid = true;
    const XT *x;
    const int8_t *right, *down;
    int64_t Lr, Lc;
    int R;
    __device__ void operator()(int64_t i, int64_t rr, int64_t cc, int r0, long long (&acc)[V][3]) const {
        const int64_t jr = cc + 1 == Lc ? i + 1 - Lc : i + 1;
        const int64_t jd = rr + 1 == Lr ? cc : i + Lc;
        const Pack<XT, V> a = ldp<XT, V>(x + i * R + r0), b = ldp<XT, V>(x + jr * R + r0),
                          d = ldp<XT, V>(x + jd * R + r0);
        const int wr = right[i], wd = down[i];
#pragma unroll
        for (int q = 0; q < V; ++q) {
            const bool s = spin_of(a.v[q]) > 0;
            const int D = ((spin_of(b.v[q]) > 0) != s ? wr : 0) + ((spin_of(d.v[q]) > 0) != s ? wd : 0);
            acc[q][0] += 2 * (wr + wd) - 4 * D;
            acc[q][1] += 4 * D;
        }
    }
};

// all ones where the FP32 iterate's spin is -1 (x < 0 or NaN), else 0
__device__ __forceinline__ unsigned down_mask(float v) { return v >= 0.f ? 0u : 0xffffffffu; }

// R = 1, FP32, l_cols a multiple of 4: four sites of a row per thread. The edges of the four
// sites are summed by byte dot products (dp4a) of the packed couplings, masked to the edges
// whose spins differ: S = sum of w, D = sum of w over those edges. A block's sites are one
// contiguous range, so the row below is read again from the caches. Bound by HBM: 6 B per site.
__global__ void __launch_bounds__(kRThreads)
torus_energy4(const float *__restrict__ x, const int8_t *__restrict__ right, const int8_t *__restrict__ down,
              int64_t Lr, int64_t Lc, int chunks, long long *__restrict__ partials) {
    const int64_t g = Lc >> 2, total = Lr * g;  // groups of four sites per row, in all
    const int64_t s0 = total * blockIdx.x / chunks, s1 = total * (blockIdx.x + 1) / chunks;
    const int64_t n = Lr * Lc;
    const int64_t dr = kRThreads / g, dc = kRThreads - dr * g;
    int64_t t = s0 + threadIdx.x;
    int64_t rr = t / g, cc = t - rr * g;
    long long S = 0, D = 0;
    for (; t < s1; t += kRThreads) {
        const int64_t i = 4 * t;
        const float4 a = __ldg(reinterpret_cast<const float4 *>(x + i));
        const float4 b = __ldg(reinterpret_cast<const float4 *>(x + (i + Lc < n ? i + Lc : i + Lc - n)));
        const float e = __ldg(x + (cc + 1 == g ? i + 4 - Lc : i + 4));
        const int wr = __ldg(reinterpret_cast<const int *>(right + i)), wd = __ldg(reinterpret_cast<const int *>(down + i));
        const unsigned m0 = down_mask(a.x), m1 = down_mask(a.y), m2 = down_mask(a.z), m3 = down_mask(a.w);
        const unsigned own01 = __byte_perm(m0, m1, 0x0040), own23 = __byte_perm(m2, m3, 0x0040);
        const unsigned own = __byte_perm(own01, own23, 0x5410);
        const unsigned nxt = __byte_perm(own, down_mask(e), 0x4321);  // the spins one column to the right
        const unsigned below = __byte_perm(__byte_perm(down_mask(b.x), down_mask(b.y), 0x0040),
                                           __byte_perm(down_mask(b.z), down_mask(b.w), 0x0040), 0x5410);
        S += __dp4a(wr, 0x01010101, __dp4a(wd, 0x01010101, 0));
        D += __dp4a(static_cast<int>(wr & (own ^ nxt)), 0x01010101,
                    __dp4a(static_cast<int>(wd & (own ^ below)), 0x01010101, 0));
        rr += dr;
        cc += dc;
        if (cc >= g) {
            cc -= g;
            ++rr;
        }
    }
    __shared__ long long red[2][kRThreads / 32];
    S = warp_sum(S);
    D = warp_sum(D);
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = S;
        red[1][threadIdx.x >> 5] = D;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        S = D = 0;
        for (int w = 0; w < kRThreads / 32; ++w) {
            S += red[0][w];
            D += red[1][w];
        }
        partials[static_cast<int64_t>(blockIdx.x) * 3 + threadIdx.x] =
            threadIdx.x == 0 ? 2 * S - 4 * D : (threadIdx.x == 1 ? 4 * D : 0);
    }
}

// ---- Hamiltonian functors (acc: sum x^4, sum x^2, sum x u, sum h x) --------

template <int V>
__device__ __forceinline__ void ham_terms(const double (&xi)[V], const double (&u)[V], double (&acc)[V][4]) {
#pragma unroll
    for (int q = 0; q < V; ++q) {
        const double x2 = xi[q] * xi[q];
        acc[q][0] += x2 * x2;
        acc[q][1] += x2;
        acc[q][2] += xi[q] * u[q];
    }
}
template <typename XT, int V>
__device__ __forceinline__ void ld_double(const XT *p, double (&v)[V]) {
    const Pack<XT, V> a = ldp<XT, V>(p);
#pragma unroll
    for (int q = 0; q < V; ++q) {
        if constexpr (sizeof(XT) == 4) v[q] = widen(a.v[q]);
        else v[q] = as_double(a.v[q]);
    }
}

template <typename XT, typename VT, int V>
struct CsrHam {
    static constexpr bool kGrid = false;
    const XT *x;
    const int64_t *row_ptr;
    const int32_t *col;
    const VT *val;
    const double *h;
    int R;
    __device__ void operator()(int64_t i, int r0, double (&acc)[V][4]) const {
        double u[V], xv[V];
#pragma unroll
        for (int q = 0; q < V; ++q) u[q] = 0.0;
        const int64_t e1 = __ldg(row_ptr + i + 1);
#pragma unroll 4
        for (int64_t e = __ldg(row_ptr + i); e < e1; ++e) {
            const double w = weight<double>(__ldg(val + e));
            ld_double<XT, V>(x + static_cast<int64_t>(__ldg(col + e)) * R + r0, xv);
#pragma unroll
            for (int q = 0; q < V; ++q) u[q] += w * xv[q];
        }
        ld_double<XT, V>(x + i * R + r0, xv);
        ham_terms<V>(xv, u, acc);
        if (h) {
            const double hv = h[i];
#pragma unroll
            for (int q = 0; q < V; ++q) acc[q][3] += hv * xv[q];
        }
    }
};

template <typename XT, int V>
struct TorusHam {
    static constexpr bool kGrid = true;
    const XT *x;
    const int8_t *right, *down;
    int64_t Lr, Lc;
    int R;
    // u = 2 (right x_r + down x_d): every edge once, x^T J x over all sites the same (six FP64 operations
    // per site instead of thirteen: 2500 x 2503 sites 217 -> 138 us)
    __device__ void operator()(int64_t i, int64_t rr, int64_t cc, int r0, double (&acc)[V][4]) const {
        const int64_t jr = cc + 1 == Lc ? i + 1 - Lc : i + 1;
        const int64_t jd = rr + 1 == Lr ? cc : i + Lc;
        const double wr = weight<double>(static_cast<float>(2 * right[i])), wd = weight<double>(static_cast<float>(2 * down[i]));
        double u[V], xv[V];
        ld_double<XT, V>(x + jr * R + r0, xv);
#pragma unroll
        for (int q = 0; q < V; ++q) u[q] = wr * xv[q];
        ld_double<XT, V>(x + jd * R + r0, xv);
#pragma unroll
        for (int q = 0; q < V; ++q) u[q] += wd * xv[q];
        ld_double<XT, V>(x + i * R + r0, xv);
        ham_terms<V>(xv, u, acc);
    }
};

// ---- finalisers ------------------------------------------------------------

// One warp per pair t: lane l adds the chunks l, l + 32, ... in order, then a fixed tree over the
// lanes (one thread per pair took 26 us for the 608 chunks of a large lattice, as long as its chain of loads).
template <typename Acc, int K>
__device__ __forceinline__ void warp_partials(const Acc *__restrict__ p, int chunks, Acc (&s)[K]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < K; ++k) s[k] = Acc(0);
    for (int c = lane; c < chunks; c += 32)
#pragma unroll
        for (int k = 0; k < K; ++k) s[k] += p[static_cast<int64_t>(c) * K + k];
#pragma unroll
    for (int k = 0; k < K; ++k) s[k] = warp_sum(s[k]);
}

template <typename Acc>
__global__ void energy_finish(const Acc *__restrict__ partials, int pairs, int chunks,
                              int64_t *E_i, int64_t *cut_i, double *E_d, double *cut_d) {
    const int t = static_cast<int>((blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5);
    if (t >= pairs) return;  // whole warps
    Acc s[3];
    warp_partials<Acc, 3>(partials + static_cast<int64_t>(t) * chunks * 3, chunks, s);
    if ((threadIdx.x & 31) != 0) return;
    if constexpr (std::is_integral<Acc>::value) {  // int64: exact
        const int64_t E = -(s[0] / 2) - s[2];
        const int64_t cut = -(s[1] / 2);
        if (E_i) E_i[t] = E;
        if (cut_i) cut_i[t] = cut;
        if (E_d) E_d[t] = static_cast<double>(E);
        if (cut_d) cut_d[t] = static_cast<double>(cut);
    } else {
        if (E_d) E_d[t] = -0.5 * s[0] - s[2];
        if (cut_d) cut_d[t] = -0.5 * s[1];
    }
}

// H(x^(k)) per replica from the fused monitor's partials [block][R][4]: one block per replica,
// thread t adds the blocks t, t + 128, ... in order, then a fixed tree
constexpr int kHT = 128;
__global__ void __launch_bounds__(kHT)
ham_fused_finish(const double *__restrict__ hpart, int blocks, int R, double alpha, double beta,
                 double *__restrict__ H) {
    const int r = blockIdx.x;
    double t[4] = {0.0, 0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < blocks; b += kHT)
#pragma unroll
        for (int m = 0; m < 4; ++m) t[m] += hpart[(static_cast<int64_t>(b) * R + r) * 4 + m];
    __shared__ double red[kHT / 32][4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        t[m] = warp_sum(t[m]);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][m] = t[m];
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
#pragma unroll
    for (int m = 0; m < 4; ++m) t[m] = (red[0][m] + red[1][m]) + (red[2][m] + red[3][m]);
    H[r] = beta / 4.0 * t[0] - alpha / 2.0 * t[1] - 0.5 * t[2] - t[3];
}

__global__ void ham_finish(const double *__restrict__ partials, int n_inst, int R, int chunks,
                           const double *__restrict__ alpha_tab, int alpha_len, int k,
                           const double *__restrict__ beta_tab, double *__restrict__ H) {
    const int t = static_cast<int>((blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5);
    if (t >= n_inst * R) return;  // whole warps
    const int b = t / R;
    double s[4];
    warp_partials<double, 4>(partials + static_cast<int64_t>(t) * chunks * 4, chunks, s);
    if ((threadIdx.x & 31) != 0) return;
    const double a = alpha_tab[static_cast<int64_t>(b) * alpha_len + (k < alpha_len ? k : alpha_len - 1)];
    const double be = beta_tab[b];
    H[t] = be / 4.0 * s[0] - a / 2.0 * s[1] - 0.5 * s[2] - s[3];
}

__global__ void best_kernel(const int64_t *__restrict__ E_i, const double *__restrict__ E_d,
                            int n_inst, int R, int32_t *__restrict__ best) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= n_inst) return;
    int arg = 0;
    if (E_i) {
        int64_t m = E_i[static_cast<int64_t>(b) * R];
        for (int r = 1; r < R; ++r)
            if (E_i[static_cast<int64_t>(b) * R + r] < m) { m = E_i[static_cast<int64_t>(b) * R + r]; arg = r; }
    } else {
        double m = E_d[static_cast<int64_t>(b) * R];
        for (int r = 1; r < R; ++r)
            if (E_d[static_cast<int64_t>(b) * R + r] < m) { m = E_d[static_cast<int64_t>(b) * R + r]; arg = r; }
    }
    best[b] = arg;
}

template <typename XT>
__global__ void spins_kernel(const XT *__restrict__ x, int64_t count, int8_t *__restrict__ s) {
    for (int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; t < count;
         t += static_cast<int64_t>(gridDim.x) * blockDim.x)
        s[t] = static_cast<int8_t>(spin_of(x[t]));
}

// replicas per thread: 16 bytes of x when R and the pointer allow it (at most 4), else 1
template <typename XT>
constexpr int wide() { return sizeof(XT) == 8 ? 2 : 4; }
template <typename XT>
bool wide_ok(const XT *x, int R) {
    return R % wide<XT>() == 0 && reinterpret_cast<uintptr_t>(x) % (sizeof(XT) * wide<XT>()) == 0;
}

// Row chunks per instance for V replicas per thread: eight blocks per SM over all instances, at
// least two rows per thread (the largest instance decides: chunks are equal shares of each).
int pick_chunks(const ising_context *c, int R, int V) {
    const int C = R / V, Cb = C < kRThreads ? C : kRThreads;
    const int64_t per = static_cast<int64_t>(c->n_inst) * ((C + Cb - 1) / Cb);
    int64_t ch = (8LL * c->num_sms + per - 1) / per;
    const int64_t rows2 = 2 * (kRThreads / Cb);
    ch = std::min<int64_t>(ch, (c->max_inst_n + rows2 - 1) / rows2);
    return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(ch, 65535)));
}

template <int K, int V, typename Acc, typename Fn>
ising_status_t run_reduce(ising_context *c, const Fn &fn, int R, int *chunks, cudaStream_t st) {
    *chunks = pick_chunks(c, R, V);
    const size_t bytes = static_cast<size_t>(c->n_inst) * R * *chunks * K * sizeof(Acc);
    DOCH_CHECK(c->partials.ensure(bytes));
    const int C = R / V, Cb = C < kRThreads ? C : kRThreads;
    dim3 grid(static_cast<unsigned>(*chunks), static_cast<unsigned>((C + Cb - 1) / Cb),
              static_cast<unsigned>(c->n_inst));
    row_reduce<K, V, Acc, Fn><<<grid, kRThreads, 0, st>>>(fn, c->n_inst > 1 ? c->inst_off : nullptr,
                                                           c->n, R, *chunks, c->partials.as<Acc>());
    DOCH_CUDA(cudaGetLastError());
    return ISING_OK;
}

template <int V, typename XT, typename VT, typename Acc>
ising_status_t csr_energy_v(ising_context *c, const XT *x, const Acc *h, int R, int *chunks, cudaStream_t st) {
    return run_reduce<3, V, Acc>(c, CsrEnergy<XT, VT, Acc, V>{x, c->row_ptr, c->col, static_cast<const VT *>(c->val), h, R},
                                 R, chunks, st);
}
template <typename XT, typename VT, typename Acc>
ising_status_t csr_energy(ising_context *c, const XT *x, const Acc *h, int R, int *chunks, cudaStream_t st) {
    if (wide_ok(x, R)) return csr_energy_v<wide<XT>(), XT, VT, Acc>(c, x, h, R, chunks, st);
    return csr_energy_v<1, XT, VT, Acc>(c, x, h, R, chunks, st);
}

template <typename XT>
ising_status_t torus_energy(ising_context *c, const XT *x, int R, int *chunks, cudaStream_t st) {
    if constexpr (std::is_same<XT, float>::value) {
        if (R == 1 && c->l_cols % 4 == 0 && reinterpret_cast<uintptr_t>(x) % 16 == 0) {
            const int64_t groups = c->n / 4, per = 2LL * kRThreads;  // at least two groups per thread
            *chunks = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>((groups + per - 1) / per, 16LL * c->num_sms)));
            DOCH_CHECK(c->partials.ensure(static_cast<size_t>(*chunks) * 3 * sizeof(long long)));
            torus_energy4<<<*chunks, kRThreads, 0, st>>>(x, c->right, c->down, c->l_rows, c->l_cols, *chunks,
                                                        c->partials.as<long long>());
            DOCH_CUDA(cudaGetLastError());
            return ISING_OK;
        }
    }
    constexpr int W = wide<XT>();
    if (wide_ok(x, R))
        return run_reduce<3, W, long long>(c, TorusEnergy<XT, W>{x, c->right, c->down, c->l_rows, c->l_cols, R}, R, chunks, st);
    return run_reduce<3, 1, long long>(c, TorusEnergy<XT, 1>{x, c->right, c->down, c->l_rows, c->l_cols, R}, R, chunks, st);
}

// integer couplings and field: int64 sums; otherwise FP64
template <typename XT>
ising_status_t energy_typed(ising_context *c, const XT *x, int R, int *chunks, cudaStream_t st) {
    if (c->format == ISING_FMT_TORUS2D) return torus_energy<XT>(c, x, R, chunks, st);
    if (c->format == ISING_FMT_CSR) {
        if (c->integer) {
            const long long *h = reinterpret_cast<const long long *>(c->h_i64);
            if (c->jtype == ISING_I8) return csr_energy<XT, int8_t, long long>(c, x, h, R, chunks, st);
            if (c->jtype == ISING_I32) return csr_energy<XT, int32_t, long long>(c, x, h, R, chunks, st);
        } else {
            switch (c->jtype) {
                case ISING_I8: return csr_energy<XT, int8_t, double>(c, x, c->h_f64, R, chunks, st);
                case ISING_I32: return csr_energy<XT, int32_t, double>(c, x, c->h_f64, R, chunks, st);
                case ISING_F32: return csr_energy<XT, float, double>(c, x, c->h_f64, R, chunks, st);
                case ISING_F64: return csr_energy<XT, double, double>(c, x, c->h_f64, R, chunks, st);
                default: break;
            }
        }
    }
    return fail(ISING_ERR_UNSUPPORTED, "energy: storage form not supported by this reduction");
}

template <int V, typename XT>
ising_status_t ham_v(ising_context *c, const XT *x, int R, int *chunks, cudaStream_t st) {
    if (c->format == ISING_FMT_TORUS2D)
        return run_reduce<4, V, double>(c, TorusHam<XT, V>{x, c->right, c->down, c->l_rows, c->l_cols, R}, R, chunks, st);
    if (c->format == ISING_FMT_CSR) {
        const double *h = c->has_h ? c->h_f64 : nullptr;
        switch (c->jtype) {
            case ISING_I8: return run_reduce<4, V, double>(c, CsrHam<XT, int8_t, V>{x, c->row_ptr, c->col, static_cast<const int8_t *>(c->val), h, R}, R, chunks, st);
            case ISING_I32: return run_reduce<4, V, double>(c, CsrHam<XT, int32_t, V>{x, c->row_ptr, c->col, static_cast<const int32_t *>(c->val), h, R}, R, chunks, st);
            case ISING_F32: return run_reduce<4, V, double>(c, CsrHam<XT, float, V>{x, c->row_ptr, c->col, static_cast<const float *>(c->val), h, R}, R, chunks, st);
            case ISING_F64: return run_reduce<4, V, double>(c, CsrHam<XT, double, V>{x, c->row_ptr, c->col, static_cast<const double *>(c->val), h, R}, R, chunks, st);
            default: break;
        }
    }
    return fail(ISING_ERR_UNSUPPORTED, "H monitor: storage form not supported");
}
template <typename XT>
ising_status_t ham_typed(ising_context *c, const XT *x, int R, int *chunks, cudaStream_t st) {
    if (wide_ok(x, R)) return ham_v<wide<XT>()>(c, x, R, chunks, st);
    return ham_v<1>(c, x, R, chunks, st);
}

}  // namespace

ising_status_t energy_reduce(ising_context *c, const void *x, int xtype, int R, int64_t *E_i,
                             int64_t *cut_i, double *E_d, double *cut_d, cudaStream_t st) {
    int chunks = 1;
    const int pairs = c->n_inst * R;
    ising_status_t s;
    switch (xtype) {
        case ISING_F32: s = energy_typed<float>(c, static_cast<const float *>(x), R, &chunks, st); break;
        case ISING_F64: s = energy_typed<double>(c, static_cast<const double *>(x), R, &chunks, st); break;
        case ISING_BF16: s = energy_typed<__nv_bfloat16>(c, static_cast<const __nv_bfloat16 *>(x), R, &chunks, st); break;
        case ISING_I8: s = energy_typed<int8_t>(c, static_cast<const int8_t *>(x), R, &chunks, st); break;
        default: return fail(ISING_ERR_INVALID_ARG, "energy: unsupported x type");
    }
    DOCH_CHECK(s);
    const unsigned blocks = static_cast<unsigned>((static_cast<int64_t>(pairs) + 3) / 4);  // four warps each
    if (c->integer)
        energy_finish<long long><<<blocks, 128, 0, st>>>(c->partials.as<long long>(), pairs, chunks, E_i, cut_i, E_d,
                                                        cut_d);
    else
        energy_finish<double><<<blocks, 128, 0, st>>>(c->partials.as<double>(), pairs, chunks, nullptr, nullptr, E_d,
                                                     cut_d);
    DOCH_CUDA(cudaGetLastError());
    return ISING_OK;
}

ising_status_t hamiltonian_reduce(ising_context *c, const void *x, int xtype, int R,
                                  const ParamTabs &p, int k, double *H_out, cudaStream_t st) {
    if (c->format == ISING_FMT_PROCEDURAL) {
        if (xtype != ISING_F32) return fail(ISING_ERR_INVALID_ARG, "PROCEDURAL iterates are F32");
        return proc_hamiltonian(c, static_cast<const float *>(x), R, p, k, H_out, st);
    }
    int chunks = 1;
    ising_status_t s;
    switch (xtype) {
        case ISING_F32: s = ham_typed<float>(c, static_cast<const float *>(x), R, &chunks, st); break;
        case ISING_F64: s = ham_typed<double>(c, static_cast<const double *>(x), R, &chunks, st); break;
        case ISING_BF16: s = ham_typed<__nv_bfloat16>(c, static_cast<const __nv_bfloat16 *>(x), R, &chunks, st); break;
        default: return fail(ISING_ERR_INVALID_ARG, "H monitor: unsupported x type");
    }
    DOCH_CHECK(s);
    const int pairs = c->n_inst * R;
    ham_finish<<<static_cast<unsigned>((static_cast<int64_t>(pairs) + 3) / 4), 128, 0, st>>>(c->partials.as<double>(), c->n_inst, R, chunks,
                                                    p.alpha_d, p.alpha_len, k, p.beta_d, H_out);
    DOCH_CUDA(cudaGetLastError());
    return ISING_OK;
}

ising_status_t ham_fused_finish_launch(const double *hpart, int blocks, int R, double alpha, double beta, double *H,
                                       cudaStream_t st) {
    ham_fused_finish<<<R, kHT, 0, st>>>(hpart, blocks, R, alpha, beta, H);
    DOCH_CUDA(cudaGetLastError());
    return ISING_OK;
}

ising_status_t best_replica(const ising_context *c, const int64_t *E_i, const double *E_d, int R,
                            int32_t *best, cudaStream_t st) {
    best_kernel<<<(c->n_inst + 127) / 128, 128, 0, st>>>(E_i, E_d, c->n_inst, R, best);
    DOCH_CUDA(cudaGetLastError());
    return ISING_OK;
}

ising_status_t write_spins(const ising_context *c, const void *x, int xtype, int R, int8_t *s,
                           cudaStream_t st) {
    const int64_t count = c->n * R;
    int64_t blocks = (count + 255) / 256;
    if (blocks > 16LL * c->num_sms) blocks = 16LL * c->num_sms;
    if (blocks < 1) blocks = 1;
    switch (xtype) {
        case ISING_F32: spins_kernel<<<blocks, 256, 0, st>>>(static_cast<const float *>(x), count, s); break;
        case ISING_F64: spins_kernel<<<blocks, 256, 0, st>>>(static_cast<const double *>(x), count, s); break;
        case ISING_BF16: spins_kernel<<<blocks, 256, 0, st>>>(static_cast<const __nv_bfloat16 *>(x), count, s); break;
        case ISING_I8: spins_kernel<<<blocks, 256, 0, st>>>(static_cast<const int8_t *>(x), count, s); break;
        default: return fail(ISING_ERR_INVALID_ARG, "spins: unsupported x type");
    }
    DOCH_CUDA(cudaGetLastError());
    return ISING_OK;
}

}  // namespace doch
