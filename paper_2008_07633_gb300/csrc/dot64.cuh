// FP64 dot products of FP32 or BF16 rows in the sequential order of the affinity's definition.
//
// The definition is s <- s + x_k y_k in FP64 with increasing k, the product and the sum rounded
// separately. The product of two widened FP32 numbers is exact in FP64 (24 + 24 bits of significand, no
// overflow or underflow), so the sum's rounding is the only one and one fused multiply-add gives
// the same bits. FP64 arithmetic and the FP32 -> FP64 conversion instruction both run at about
// 2 lanes per clock and SM here, so the conversions cost as much as the arithmetic: normal numbers
// are widened by integer moves instead (rebias the exponent, shift the significand; exact), and
// only vectors that hold a zero, subnormal, infinity or NaN take the conversion. What bounds the
// kernels is then the K fused multiply-adds of a row pair. On the 128^3 grid and its coarse graph
// (K = 32) distances and row norms together went from 2,990 to about 910 us.
#pragma once
#include "vec.cuh"

// Stored block entry widened to FP64 (exact for FP32 and BF16).
__device__ __forceinline__ double widen(float x) { return (double)x; }
__device__ __forceinline__ double widen(__nv_bfloat16 x) { return (double)__bfloat162float(x); }

// A normal FP32 number (exponent field not 0 or 255) as FP64, by integer moves.
__device__ __forceinline__ bool is_normal32(float x) {
    return ((__float_as_uint(x) & 0x7fffffffu) - 0x00800000u) < 0x7f000000u;
}
__device__ __forceinline__ double widen_normal(float x) {
    const uint32_t b = __float_as_uint(x);
    const uint32_t hi = (((b & 0x7fffffffu) >> 3) + 0x38000000u) | (b & 0x80000000u);
    return __hiloint2double((int)hi, (int)(b << 29));
}

template <int E>
__device__ __forceinline__ void widen_vec(const float (&x)[E], double (&d)[E]) {
    bool plain = true;
#pragma unroll
    for (int e = 0; e < E; ++e) plain = plain && is_normal32(x[e]);
    if (plain) {
#pragma unroll
        for (int e = 0; e < E; ++e) d[e] = widen_normal(x[e]);
    } else {
#pragma unroll
        for (int e = 0; e < E; ++e) d[e] = (double)x[e];
    }
}

// sum_k a_k b_k, increasing k. VEC: both rows 16-byte aligned and K a multiple of the vector.
template <typename T, bool VEC>
__device__ __forceinline__ double dot_seq(const T* __restrict__ a, const T* __restrict__ b, int K) {
    double s = 0.0;
    if constexpr (VEC) {
        constexpr int E = Vec<T>::E;
#pragma unroll 2
        for (int k = 0; k < K; k += E) {
            float x[E], y[E];
            double xd[E], yd[E];
            Vec<T>::load(a + k, x);
            Vec<T>::load(b + k, y);
            widen_vec<E>(x, xd);
            widen_vec<E>(y, yd);
#pragma unroll
            for (int e = 0; e < E; ++e) s = __fma_rn(xd[e], yd[e], s);
        }
    } else {
        for (int k = 0; k < K; ++k) s = __fma_rn(widen(a[k]), widen(b[k]), s);
    }
    return s;
}

// sum_k a_k^2, increasing k.
template <typename T, bool VEC>
__device__ __forceinline__ double norm2_seq(const T* __restrict__ a, int K) {
    double s = 0.0;
    if constexpr (VEC) {
        constexpr int E = Vec<T>::E;
#pragma unroll 4
        for (int k = 0; k < K; k += E) {
            float x[E];
            double xd[E];
            Vec<T>::load(a + k, x);
            widen_vec<E>(x, xd);
#pragma unroll
            for (int e = 0; e < E; ++e) s = __fma_rn(xd[e], xd[e], s);
        }
    } else {
        for (int k = 0; k < K; ++k) {
            const double x = widen(a[k]);
            s = __fma_rn(x, x, s);
        }
    }
    return s;
}

// delta = 1 - dot^2 / (|p|^2 |q|^2), each operation rounded; a zero row gives 1.
__device__ __forceinline__ double affinity_delta(double dot, double np, double nq) {
    const double den = __dmul_rn(np, nq);
    return den > 0.0 ? __dsub_rn(1.0, __ddiv_rn(__dmul_rn(dot, dot), den)) : 1.0;
}

// Whether rows of K entries of T at X can be read by 16-byte vectors.
template <typename T>
static inline bool rows_vectorised(const T* X, int K) {
    return ((uintptr_t)X & 15) == 0 && K % Vec<T>::E == 0;
}
