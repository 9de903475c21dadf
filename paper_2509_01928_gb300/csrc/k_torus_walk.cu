// DOCH steps (Eq. FPE) on a periodic lattice for any number of replicas, any width and
// alignment, FP32 and FP64: x' = cbrt((sum_j J_ij x_j + alpha x_i) / beta).
//
// One pass does TS steps (TS = 3, 2 or 1; FP64 takes 1). A block owns a window of
// columns and one group of G chunks of V replicas (V values = up to 16 bytes; thread =
// one site column, one chunk) and walks down a strip of rows. x rows arrive D rows ahead by
// cp.async in a shared-memory ring; a thread keeps its own column's rows in registers and
// takes the left and right neighbours from the ring. Level l of the pass (step k + l) lags
// level l - 1 by one row: in iteration i level 1 forms row r, level 2 row r - 1 from the
// level-1 rows r - 2 .. r, level 3 row r - 2, so x is read and written once per TS steps.
// Each level's row is also stored to shared memory and read by its neighbours in the next
// iteration: one barrier per row. A pass of TS steps needs a halo of TS columns on each
// side of the window and of TS rows; the halo is recomputed (256 / G columns per window,
// 2 TS of them halo). All sums and updates are the same for every TS and V, so the
// results do not depend on how the steps are grouped.
//
// Couplings: one word per site, (right, left, down, up) as bytes offset by 128, built once
// per handle, 4 bytes per site kept beside the couplings (the four edges of a site in one 4-byte load
// instead of two rows and a neighbour of two int8 arrays).
//
// FP32, three steps: 71 % of the issue slots active at 33 lane slots per value and step (halo included),
// XU, FMA and ALU pipes at 31 to 38 %; the rest are waits of the 16 warps per SM that registers (up to 96)
// and the ring (47 KB) leave, with a barrier per row. 1000 x 1000 lattice, R = 16: 106 us per step with one
// thread per value and divisions for its site, 20.5 us now. FP64: its arithmetic.
//
// FP32 roots: the walk takes them without a test of their range and walks a strip once more, tests
// included, where one of its roots left it (zeros do: twice the time for blocks that hold a zero replica).
#include <algorithm>
#include <cmath>

#include "internal.cuh"
#include "root.cuh"

namespace doch {
namespace {

constexpr int kWT = 256;  // threads per block
constexpr int kWD = 6;    // ring rows

template <typename T, int V>
struct alignas(sizeof(T) * V) Vec {
    T v[V];
};

template <int BYTES>
__device__ __forceinline__ void copy_async(void *dst, const void *src) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void commit_async() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void wait_async() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// byte k of an edge word as a coupling: the byte in the low mantissa of 2^23, less 2^23 + 128
__device__ __forceinline__ void unpack(uint32_t w, float (&f)[4]) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
        f[k] = __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7540u | static_cast<unsigned>(k))) - 8388736.0f;
}
__device__ __forceinline__ void unpack(uint32_t w, double (&f)[4]) {
    float g[4];
    unpack(w, g);
#pragma unroll
    for (int k = 0; k < 4; ++k) f[k] = g[k] == 0.f ? 0.0 : widen_normal(g[k]);
}

// one row of a thread's V values: the four neighbours in the order right, left, down, up. NEAR (FP32): the
// roots without the test of their range, which `far` collects (root.cuh).
template <typename T, int V, bool NEAR, typename P>
__device__ __forceinline__ Vec<T, V> row_new(const Vec<T, V> &m, const Vec<T, V> &l, const Vec<T, V> &r,
                                             const Vec<T, V> &u, const Vec<T, V> &d, const T (&w)[4], T alpha,
                                             const P &p, float &far) {
    Vec<T, V> o;
#pragma unroll
    for (int q = 0; q < V; ++q) {
        T z = w[0] * r.v[q];
        z = fma(w[1], l.v[q], z);
        z = fma(w[2], d.v[q], z);
        z = fma(w[3], u.v[q], z);
        z = fma(alpha, m.v[q], z);
        if constexpr (NEAR) o.v[q] = root_near(z, p, far);
        else o.v[q] = root_newton(z, p);
    }
    return o;
}

template <typename T, int TS>
struct Alphas {
    T a[TS];
};

template <typename T, int V, int TS>
struct WalkSmem {
    Vec<T, V> x[kWD][kWT];
    uint32_t e[kWD][kWT];
    Vec<T, V> y[TS > 1 ? TS - 1 : 1][2][TS > 1 ? kWT : 1];
};

// one block's strip of rows; returns the largest |log2| of its roots (NEAR)
template <typename T, int V, int TS, bool NEAR>
__device__ __forceinline__ float walk_strip(WalkSmem<T, V, TS> &sm, const T *xc, T *oc, const uint32_t *ec, int64_t Lr,
                                            int64_t Lc, int64_t W, int64_t r0, int rows, int s, int g, int tl, int left,
                                            int right, bool writes, const Alphas<T, TS> &alpha,
                                            const typename RootOf<T>::type &root) {
    float far = 0.f;
    // ring row k holds lattice row r0 - TS + k (wrapped); rows 0 .. nk - 1 are needed
    const int nk = rows + 2 * TS;
    int64_t rk = (r0 - TS) % Lr;  // lattice row of the next ring row to stage
    if (rk < 0) rk += Lr;
    auto stage = [&](int k, int slot) {
        if (k < nk) {
            copy_async<sizeof(T) * V>(&sm.x[slot][tl], xc + rk * W);
            if (g == 0) copy_async<4>(&sm.e[slot][s], ec + rk * Lc);
            rk = rk + 1 == Lr ? 0 : rk + 1;
        }
        commit_async();
    };
#pragma unroll
    for (int k = 0; k < kWD; ++k) stage(k, k);
    wait_async<kWD - 3>();  // rows 0, 1, 2 have landed
    __syncthreads();
    Vec<T, V> xu = sm.x[0][tl], xm = sm.x[1][tl];
    Vec<T, V> ya[TS], yb[TS];
    T w[TS][4];  // couplings of the rows of levels 1 .. TS
#pragma unroll
    for (int l = 0; l < TS; ++l) {
#pragma unroll
        for (int q = 0; q < V; ++q) ya[l].v[q] = yb[l].v[q] = T(0);
#pragma unroll
        for (int q = 0; q < 4; ++q) w[l][q] = T(0);
    }
    T *op = oc + r0 * W;
    const int iters = rows + 2 * (TS - 1);
    int s0 = 0;  // ring slot of row i
    for (int i = 0; i < iters; ++i) {
        const int s1 = s0 + 1 == kWD ? 0 : s0 + 1, s2 = s1 + 1 == kWD ? 0 : s1 + 1;
        stage(i + kWD, s0);  // row i was last read before the barrier
#pragma unroll
        for (int l = TS - 1; l > 0; --l)
#pragma unroll
            for (int q = 0; q < 4; ++q) w[l][q] = w[l - 1][q];
        unpack(sm.e[s1][s], w[0]);
        const Vec<T, V> xd = sm.x[s2][tl];
        Vec<T, V> y = row_new<T, V, NEAR>(xm, sm.x[s1][left], sm.x[s1][right], xu, xd, w[0], alpha.a[0], root, far);
        xu = xm;
        xm = xd;
#pragma unroll
        for (int l = 1; l < TS; ++l) {
            if (i < 2 * (l - 1)) break;  // level l has no row yet (uniform)
            sm.y[l - 1][i & 1][tl] = y;
            Vec<T, V> yn = y;
            if (i >= 2 * l)
                yn = row_new<T, V, NEAR>(yb[l], sm.y[l - 1][(i & 1) ^ 1][left], sm.y[l - 1][(i & 1) ^ 1][right], ya[l], y,
                                         w[l], alpha.a[l], root, far);
            ya[l] = yb[l];
            yb[l] = y;
            y = yn;
        }
        if (i >= 2 * (TS - 1)) {
            if (writes) *reinterpret_cast<Vec<T, V> *>(op) = y;
            op += W;
        }
        wait_async<kWD - 3>();  // row i + 3 has landed
        __syncthreads();
        s0 = s1;
    }
    wait_async<0>();
    return far;
}

// the strip again, each root with its test: out of line, so that the strip before it keeps its registers
template <int V, int TS>
__device__ __noinline__ void walk_again(WalkSmem<float, V, TS> *sm, const float *xc, float *oc, const uint32_t *ec,
                                        int64_t Lr, int64_t Lc, int64_t W, int64_t r0, int rows, int s, int g, int tl,
                                        int left, int right, bool writes, Alphas<float, TS> alpha, RootF32 root) {
    walk_strip<float, V, TS, false>(*sm, xc, oc, ec, Lr, Lc, W, r0, rows, s, g, tl, left, right, writes, alpha, root);
}

template <typename T, int V, int TS>
__global__ void __launch_bounds__(kWT, sizeof(T) == 8 ? 3 : 2)
torus_walk(const T *__restrict__ xi, T *__restrict__ xo, const uint32_t *__restrict__ edge, int64_t Lr, int64_t Lc, int R,
           int G, int groups, int nwin, int wout, int strips, Alphas<T, TS> alpha,
           typename RootOf<T>::type root) {
    extern __shared__ __align__(16) unsigned char walk_smem[];
    WalkSmem<T, V, TS> &sm = *reinterpret_cast<WalkSmem<T, V, TS> *>(walk_smem);
    const int t = threadIdx.x;
    const int grp = blockIdx.x % groups, rest = blockIdx.x / groups;
    const int win = rest % nwin, strip = rest / nwin;
    const int64_t r0 = Lr * strip / strips;
    const int rows = static_cast<int>(Lr * (strip + 1) / strips - r0);  // (launch_walk)
    const int sites = blockDim.x / G;          // columns of the window, halo included
    const int s = min(t / G, sites - 1);       // threads past the last whole site repeat it
    const int g = t % G;
    const int tl = s * G + g;                  // this thread's slot (repeated ones write the same values)
    const int left = s > 0 ? tl - G : tl, right = s + 1 < sites ? tl + G : tl;
    const int64_t off = static_cast<int64_t>(win) * wout + s - TS;  // column, not wrapped
    int64_t col = off % Lc;
    if (col < 0) col += Lc;
    const bool writes = s >= TS && s < TS + wout && off < Lc && t / G < sites;
    const int64_t W = Lc * R;
    const int64_t at = col * R + (static_cast<int64_t>(grp) * G + g) * V;
    if constexpr (sizeof(T) == 4) {
        const float far = walk_strip<T, V, TS, true>(sm, xi + at, xo + at, edge + col, Lr, Lc, W, r0, rows, s, g, tl, left,
                                                     right, writes, alpha, root);
        if (__syncthreads_or(!(far < kNear)))
            walk_again<V, TS>(&sm, xi + at, xo + at, edge + col, Lr, Lc, W, r0, rows, s, g, tl, left, right, writes, alpha,
                              root);
    } else {
        walk_strip<T, V, TS, false>(sm, xi + at, xo + at, edge + col, Lr, Lc, W, r0, rows, s, g, tl, left, right, writes,
                                    alpha, root);
    }
}

__global__ void edge_words(const int8_t *__restrict__ right, const int8_t *__restrict__ down, int64_t Lr, int64_t Lc,
                           uint32_t *__restrict__ e) {
    const int64_t n = Lr * Lc;
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t c = i % Lc;
        const uint32_t r = static_cast<uint8_t>(right[i]), l = static_cast<uint8_t>(right[c == 0 ? i + Lc - 1 : i - 1]);
        const uint32_t d = static_cast<uint8_t>(down[i]), u = static_cast<uint8_t>(down[i < Lc ? i + n - Lc : i - Lc]);
        e[i] = (r | l << 8 | d << 16 | u << 24) ^ 0x80808080u;
    }
}

// chunks per thread group: the smallest divisor of C that makes a site's piece at least one 32-byte
// sector, else the largest divisor up to 20 (wider groups would leave too few columns per window)
int group_of(int C, size_t bytes) {
    int best = 1;
    for (int d = 1; d <= 20 && d <= C; ++d) {
        if (C % d) continue;
        best = d;
        if (d * bytes >= 32) break;
    }
    return best;
}

template <typename T, int V, int TS>
ising_status_t launch_walk(const ising_context *c, const T *xi, T *xo, int R, const Alphas<T, TS> &a,
                           const typename RootOf<T>::type &root, cudaStream_t st) {
    const int64_t Lr = c->l_rows, Lc = c->l_cols;
    const int C = R / V, G = group_of(C, sizeof(T) * V), groups = C / G;
    // the window: up to 256 / G columns, no wider than the lattice with its halo
    const int64_t most = std::min<int64_t>(kWT / G, Lc + 2 * TS);
    const int64_t nwin = (Lc + most - 2 * TS - 1) / (most - 2 * TS);
    const int wout = static_cast<int>((Lc + nwin - 1) / nwin);
    const int threads = std::min(kWT, ((wout + 2 * TS) * G + 31) / 32 * 32);
    auto kern = torus_walk<T, V, TS>;
    const int smem = static_cast<int>(sizeof(WalkSmem<T, V, TS>));
    static int occ_of[kWT / 32 + 1] = {};  // blocks per SM by warps per block
    int &occ = occ_of[threads / 32];
    if (!occ) {
        DOCH_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        int o = 0;
        DOCH_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, threads, smem));
        occ = std::max(1, o);
    }
    // one resident wave of blocks: the strips take what the windows and groups leave
    const int64_t slots = static_cast<int64_t>(c->num_sms) * occ;
    const int64_t strips = std::max<int64_t>(1, std::min<int64_t>(Lr, slots / (nwin * groups)));
    const int64_t blocks = strips * nwin * groups;
    // (sides of 2^31 and more fit the memory; a block's rows stay below 2^31: strips fill the slots unless the
    // windows and groups do, and then 2^31 rows of them do not fit)
    if (blocks > INT32_MAX || Lr / strips > INT32_MAX - 16) return fail(ISING_ERR_UNSUPPORTED, "lattice too large");
    kern<<<static_cast<unsigned>(blocks), threads, smem, st>>>(xi, xo, c->edge.as<uint32_t>(), Lr, Lc, R, G, groups,
                                                               static_cast<int>(nwin), wout,
                                                               static_cast<int>(strips), a, root);
    DOCH_CUDA(cudaGetLastError());
    return ISING_OK;
}

template <typename T, int V>
ising_status_t walk_v(const ising_context *c, const T *xi, T *xo, int R, const double *alpha, int ts,
                      const typename RootOf<T>::type &root, cudaStream_t st) {
    if constexpr (sizeof(T) == 4) {
        if (ts == 3)
            return launch_walk<T, V, 3>(c, xi, xo, R,
                                        {{static_cast<T>(alpha[0]), static_cast<T>(alpha[1]), static_cast<T>(alpha[2])}},
                                        root, st);
        if (ts == 2)
            return launch_walk<T, V, 2>(c, xi, xo, R, {{static_cast<T>(alpha[0]), static_cast<T>(alpha[1])}}, root, st);
    }
    return launch_walk<T, V, 1>(c, xi, xo, R, {{static_cast<T>(alpha[0])}}, root, st);
}

// the edge words, built once per handle; the host waits, so that a later call may use any stream
ising_status_t ensure_edges(ising_context *c, cudaStream_t st) {
    if (c->edge.ptr) return ISING_OK;
    DevBuf b;
    DOCH_CHECK(b.ensure(sizeof(uint32_t) * static_cast<size_t>(c->n)));
    const int64_t blocks = std::min<int64_t>((c->n + 255) / 256, 16LL * c->num_sms);
    edge_words<<<static_cast<unsigned>(blocks), 256, 0, st>>>(c->right, c->down, c->l_rows, c->l_cols, b.as<uint32_t>());
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        b.release();
        return cuda_fail(e, "lattice edge words");
    }
    c->edge = b;
    return ISING_OK;
}

}  // namespace

ising_status_t torus_walk_f32(ising_context *c, const float *x_in, float *x_out, int R, const double *alpha, int ts,
                              double inv_beta, cudaStream_t st) {
    DOCH_CHECK(ensure_edges(c, st));
    const uintptr_t a = reinterpret_cast<uintptr_t>(x_in) | reinterpret_cast<uintptr_t>(x_out);
    const RootF32 root = root_f32(inv_beta);
    if (R % 4 == 0 && a % 16 == 0) return walk_v<float, 4>(c, x_in, x_out, R, alpha, ts, root, st);
    if (R % 2 == 0 && a % 8 == 0) return walk_v<float, 2>(c, x_in, x_out, R, alpha, ts, root, st);
    return walk_v<float, 1>(c, x_in, x_out, R, alpha, ts, root, st);
}

ising_status_t torus_step_f64(ising_context *c, const double *x_in, double *x_out, int R, double alpha, double beta,
                              cudaStream_t st) {
    DOCH_CHECK(ensure_edges(c, st));
    const uintptr_t a = reinterpret_cast<uintptr_t>(x_in) | reinterpret_cast<uintptr_t>(x_out);
    const RootF64 root = root_f64(beta);
    if (R % 2 == 0 && a % 16 == 0) return walk_v<double, 2>(c, x_in, x_out, R, &alpha, 1, root, st);
    return walk_v<double, 1>(c, x_in, x_out, R, &alpha, 1, root, st);
}

}  // namespace doch
