// 16-byte vector helpers of the flat Krylov passes (kernels_aux.cu) and the Gram-Schmidt
// column kernel (kernels_mgs.cu).  Both take their products, updates and dot products from
// here, so that the two forms of a pass compute the same values bit for bit.
#pragma once

#include "ewave_internal.cuh"

namespace ewv {

template <typename T>
__device__ __forceinline__ T* vptr(const ProblemDev* P, int k) {
    return k == 0 ? (T*)P->state : (T*)P->work + (long long)(k - 1) * P->vec_stride;
}

template <typename T>
struct Vec16;
template <>
struct Vec16<float> {
    using type = float4;
    static constexpr int N = 4;
};
template <>
struct Vec16<double> {
    using type = double2;
    static constexpr int N = 2;
};

__device__ __forceinline__ float dot16(const float4& a, const float4& b) {
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, a.x * b.x)));
}
__device__ __forceinline__ double dot16d(const double2& a, const double2& b) {
    return fma(a.y, b.y, a.x * b.x);
}
__device__ __forceinline__ float4 axpy16(const float4& w, float c, const float4& q) {
    return make_float4(fmaf(-c, q.x, w.x), fmaf(-c, q.y, w.y), fmaf(-c, q.z, w.z), fmaf(-c, q.w, w.w));
}
__device__ __forceinline__ double2 axpy16(const double2& w, double c, const double2& q) {
    return make_double2(fma(-c, q.x, w.x), fma(-c, q.y, w.y));
}
__device__ __forceinline__ void fma16(float4& acc, float c, const float4& q) {
    acc.x = fmaf(c, q.x, acc.x);
    acc.y = fmaf(c, q.y, acc.y);
    acc.z = fmaf(c, q.z, acc.z);
    acc.w = fmaf(c, q.w, acc.w);
}
__device__ __forceinline__ void fma16(double2& acc, double c, const double2& q) {
    acc.x = fma(c, q.x, acc.x);
    acc.y = fma(c, q.y, acc.y);
}
// hi + lo += x, the rounding of hi + x kept in lo (Knuth's TwoSum)
__device__ __forceinline__ void two_sum_add(float& hi, float& lo, float x) {
    const float s = hi + x;
    const float b = s - hi;
    lo += (hi - (s - b)) + (x - b);
    hi = s;
}

// Sum of dot products of 16-byte vectors.  FP64 vectors: an FP64 sum.  FP32 vectors: the products
// of four elements are added in FP32 (dot16), those sums accumulated as an unevaluated pair of
// FP32 numbers (48 bits) that is widened to FP64 once: an FP64 conversion and addition for every
// 16 bytes would occupy the FP64 pipe (16 cycles each) longer than memory takes to deliver them.
// Nothing is lost by it: over 200,000 elements a total is within 2e-17 |a| |b| of an FP64
// accumulation of the same four-element sums, which are off by 1e-10 |a| |b| themselves.
template <typename V>
struct DotSum;
template <>
struct DotSum<double2> {
    double s = 0.0;
    __device__ __forceinline__ void add(const double2& a, const double2& b) { s += dot16d(a, b); }
    // sum over the warp, valid on lane 0
    __device__ __forceinline__ double warp_total() const {
        double v = s;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        return v;
    }
};
template <>
struct DotSum<float4> {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(const float4& a, const float4& b) { two_sum_add(hi, lo, dot16(a, b)); }
    __device__ __forceinline__ double warp_total() const {
        float h = hi, l = lo;
        for (int o = 16; o > 0; o >>= 1) {
            const float oh = __shfl_down_sync(0xffffffffu, h, o), ol = __shfl_down_sync(0xffffffffu, l, o);
            two_sum_add(h, l, oh);
            l += ol;
        }
        return (double)h + (double)l;
    }
};

// An infinity or NaN (by the exponent's bits: a comparison of FP64 values would occupy the FP64 pipe).
__device__ __forceinline__ bool out_of_range(double v) { return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000; }

// sum <a[q], b[q]> over the vectors q < n that the warp's lanes visit (q = lane's thread number, + NTHREADS,
// ...), accumulated in FP64 by one thread.
template <typename V>
__device__ __forceinline__ double warp_dot_in_fp64(const V* a, const V* b, int n, int warp) {
    double s = 0.0;
    if constexpr (sizeof(a->x) == 4)
        for (int q0 = 32 * warp; q0 < n; q0 += NTHREADS)
            for (int q = q0; q < q0 + 32 && q < n; ++q) s += (double)dot16(a[q], b[q]);
    return s;
}

// Block-wide total (fixed order), valid on thread 0; red: one double per warp.  Called by all threads.
// again(warp): the warp's sum from memory in FP64 (warp_dot_in_fp64), for FP32 pairs that left their
// range: a pair holds a warp's sum up to 3.4e38, a 256th of what the sums of four products that make
// it up may reach.
template <typename V, class F>
__device__ __forceinline__ double block_total(const DotSum<V>& d, double* red, F&& again) {
    const int tid = threadIdx.y * blockDim.x + threadIdx.x;
    double w = d.warp_total();
    if ((tid & 31) == 0) {
        if constexpr (sizeof(V) / sizeof(decltype(V::x)) == 4)
            if (out_of_range(w)) w = again(tid >> 5);
        red[tid >> 5] = w;
    }
    __syncthreads();
    double s = 0.0;
    if (tid == 0)
        for (int i = 0; i < NTHREADS / 32; ++i) s += red[i];
    __syncthreads();
    return s;
}

}  // namespace ewv
