// Arithmetic of one cell with stored face coefficients.
#pragma once

namespace afg {

// n / s, with is = 1/s
template <typename T>
__device__ __forceinline__ T var_quot(T n, T s, T is) {
    const T q = n * is;
    return fma(fma(-q, s, n), is, q);
}

// sum_s c_s u_s for the neighbours x[0..2D-1] of one cell, in side order
template <int D, typename T>
__device__ __forceinline__ T var_dot(const T (&c)[2 * D], const T (&x)[2 * D]) {
    T a = T(0);
#pragma unroll
    for (int s = 0; s < 2 * D; ++s) a += c[s] * x[s];
    return a;
}

}  // namespace afg
