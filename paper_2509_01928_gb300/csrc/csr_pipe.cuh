// Loads of the CSR row pipeline. A thread that owns rows i, i + S, i + 2S, ...
// keeps the next row's first batch of column / value entries and the entry range
// of the row after it in flight while the current row's neighbours are gathered,
// so a row waits for one round of memory latency instead of three
// (row_ptr -> col -> gather).
//
// Also here: the vector loads and stores and the update of the CSR step kernels.
#pragma once

#include <cstdint>

#include "cbrt.cuh"
#include "internal.cuh"
#include "root.cuh"

namespace doch {

// a coupling in the arithmetic's type; 8-bit couplings reach FP64 through FP32 and a move of its fields
// (root.cuh), an FP64 conversion costs as much as an FMA
template <typename AT, typename VT>
__device__ __forceinline__ AT coupling(VT v) { return static_cast<AT>(v); }
template <>
__device__ __forceinline__ double coupling<double, int8_t>(int8_t v) {
    return v ? widen_normal(static_cast<float>(v)) : 0.0;
}

// entry range [e0, e1) of row i (empty past the last row), in the kernel's index type IT
// (32-bit where the rows and entries allow it: fewer registers, more resident warps)
template <typename IT>
__device__ __forceinline__ void pipe_row_range(const int64_t *__restrict__ row_ptr, IT i, IT n, IT &e0, IT &e1) {
    if (i < n) {
        e0 = static_cast<IT>(__ldg(row_ptr + i));
        e1 = static_cast<IT>(__ldg(row_ptr + i + 1));
    } else {
        e0 = e1 = 0;
    }
}

// the first B entries of [e0, e1): columns and values as AT (0 past the end)
template <int B, typename AT, typename VT, typename IT>
__device__ __forceinline__ void pipe_first_batch(const int32_t *__restrict__ col, const VT *__restrict__ val,
                                                 IT e0, IT e1, int32_t (&js)[B], AT (&ws)[B]) {
    const int m = e1 - e0 < B ? static_cast<int>(e1 - e0) : B;
    const int32_t *c = col + e0;
    const VT *v = val + e0;
#pragma unroll
    for (int t = 0; t < B; ++t) {
        js[t] = t < m ? __ldg(c + t) : 0;
        ws[t] = t < m ? coupling<AT, VT>(__ldg(v + t)) : AT(0);
    }
}

// The update of the step kernels, x = cbrt(z / beta) for z = (J x + alpha x + h)_i: FP32 through the
// prescaled power-of-two cube root (cbrt.cuh; zs = 2^(3k) / beta, xsc = 2^-k per instance), FP64
// through two Newton steps (root.cuh: 11 FP64 operations, against about 50 for z / beta and cbrt).
template <typename T>
struct StepRoot;
template <>
struct StepRoot<float> {
    float zs, xsc;
    __device__ __forceinline__ explicit StepRoot(const StepValues<float> &v) : zs(v.zs), xsc(v.xsc) {}
    __device__ __forceinline__ StepRoot(const float *, const float *zs_tab, const float *xs_tab, int b)
        : zs(__ldg(zs_tab + b)), xsc(__ldg(xs_tab + b)) {}
    __device__ __forceinline__ float operator()(float z) const { return cbrt_pow2(z * zs) * xsc; }
};
template <>
struct StepRoot<double> {
    RootF64 p;
    __device__ __forceinline__ explicit StepRoot(const StepValues<double> &v) : p(make_root<double>(v.beta)) {}
    __device__ __forceinline__ StepRoot(const double *beta_tab, const float *, const float *, int b)
        : p(make_root<double>(__ldg(beta_tab + b))) {}
    __device__ __forceinline__ double operator()(double z) const { return root_newton(z, p); }
};

template <typename T, int V> struct VecOf;
template <> struct VecOf<float, 1> { using type = float; };
template <> struct VecOf<float, 2> { using type = float2; };
template <> struct VecOf<float, 4> { using type = float4; };
template <> struct VecOf<double, 1> { using type = double; };
template <> struct VecOf<double, 2> { using type = double2; };

template <typename T, int V>
__device__ __forceinline__ void ldv(const T *p, T (&v)[V]) {
    using VT = typename VecOf<T, V>::type;
    const VT w = __ldg(reinterpret_cast<const VT *>(p));
    const T *q = reinterpret_cast<const T *>(&w);
#pragma unroll
    for (int k = 0; k < V; ++k) v[k] = q[k];
}

// the same past L1: values that the kernel before this one wrote while this one was starting
template <typename T, int V>
__device__ __forceinline__ void ldv_cg(const T *p, T (&v)[V]) {
    using VT = typename VecOf<T, V>::type;
    const VT w = __ldcg(reinterpret_cast<const VT *>(p));
    const T *q = reinterpret_cast<const T *>(&w);
#pragma unroll
    for (int k = 0; k < V; ++k) v[k] = q[k];
}

template <typename T, int V>
__device__ __forceinline__ void stv(T *p, const T (&v)[V]) {
    using VT = typename VecOf<T, V>::type;
    VT w;
    T *q = reinterpret_cast<T *>(&w);
#pragma unroll
    for (int k = 0; k < V; ++k) q[k] = v[k];
    *reinterpret_cast<VT *>(p) = w;
}

}  // namespace doch
