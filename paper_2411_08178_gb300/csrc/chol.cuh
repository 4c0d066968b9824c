// One-CTA in-place Cholesky (the factor) and symmetric solve (the Newton prox).
#pragma once
#include "internal.cuh"

namespace nys {

// in-place lower Cholesky of an n x n row-major matrix by one CTA; returns
// false (uniformly) if a pivot is not positive.  `flag` is shared memory.
__device__ __forceinline__ bool block_cholesky(double* A, int n, int* flag) {
    if (threadIdx.x == 0) *flag = 0;
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        if (threadIdx.x == 0) {
            const double d = A[(size_t)k * n + k];
            if (!(d > 0.0) || !isfinite(d)) *flag = 1;
            else A[(size_t)k * n + k] = sqrt(d);
        }
        __syncthreads();
        if (*flag) return false;
        const double dk = A[(size_t)k * n + k];
        for (int i = k + 1 + threadIdx.x; i < n; i += blockDim.x) A[(size_t)i * n + k] /= dk;
        __syncthreads();
        const int m = n - k - 1;
        for (int t = threadIdx.x; t < m * m; t += blockDim.x) {
            const int i = k + 1 + t / m, j = k + 1 + t % m;
            if (j <= i) A[(size_t)i * n + j] -= A[(size_t)i * n + k] * A[(size_t)j * n + k];
        }
        __syncthreads();
    }
    for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
        const int i = t / n, j = t % n;
        if (j > i) A[t] = 0.0;
    }
    __syncthreads();
    return true;
}

// x = A^{-1} b for the symmetric positive definite n x n A in the lower triangle
// of rows 0 .. n - 1 of M (shared memory, row pitch ld > n) and b in row n: L D
// L^T elimination with the right-hand side as the last row, one barrier per
// column, then the back substitution by one warp.  M is overwritten, inv (n
// doubles, shared) holds 1 / D, x may be shared or global.  Returns false
// (uniformly) if a pivot is not positive.  n <= 128.
__device__ __forceinline__ bool block_ldl_solve(double* M, int ld, int n, double* inv, double* x) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (threadIdx.x == 0) inv[0] = 1.0 / M[0];
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        const double ik = inv[k];        // written before the last barrier, the same for every thread
        if (!(ik > 0.0) || !isfinite(ik)) return false;
        for (int i = k + 1 + warp; i <= n; i += nw) {
            const double f = M[(size_t)i * ld + k] * ik;
            for (int j = k + 1 + lane; j <= min(i, n - 1); j += 32) {
                const double v = M[(size_t)i * ld + j] - f * M[(size_t)j * ld + k];
                M[(size_t)i * ld + j] = v;
                if (i == k + 1 && j == k + 1) inv[k + 1] = 1.0 / v;   // the next pivot
            }
        }
        __syncthreads();
    }
    if (warp == 0) {
        // x_k = inv_k (y_k - sum_{i > k} M(i, k) x_i), y the eliminated last row
        double y[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) y[c] = lane + 32 * c < n ? M[(size_t)n * ld + lane + 32 * c] : 0.0;
        for (int k = n - 1; k >= 0; --k) {
            double yk = 0.0;
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if ((k >> 5) == c) yk = __shfl_sync(0xffffffffu, y[c], k & 31);
            const double xk = yk * inv[k];
            if (lane == 0) x[k] = xk;
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (lane + 32 * c < k) y[c] -= M[(size_t)k * ld + lane + 32 * c] * xk;
        }
    }
    __syncthreads();
    return true;
}

}  // namespace nys
