// The dense factor of the composite transform (paper Sec. 3.3): Q1 = (I - A)(I + A)^{-1}, A skew-symmetric, from its strict
// upper triangle, and the gradient of the parameters from the gradient of Q1.
//
// (I - A) and (I + A)^{-1} commute, so Q1 solves (I + A) Q1 = I - A: Gauss-Jordan with partial pivoting on the augmented
// matrix [I + A | I - A], one CTA, float64 in shared memory (I + A has all singular values >= 1).  With M = (I + A)^{-1},
// I + Q1 = 2 M and dQ1 = -(I + Q1) dA M, so dL/dA = -(I + Q1)^T (dL/dQ1) M^T = -2 M^T (dL/dQ1) M^T and the parameter (i < j)
// receives dL/dA[i][j] - dL/dA[j][i].
//
// A column step is a chain (find the pivot, divide, update), so its latency is what counts.  Two copies of the matrix take
// turns: every thread reads the old one (the row exchange is only a matter of where a row is read) and writes the new one,
// one block barrier per column; every warp finds the pivot by itself.  Four barriers and a serial pivot search per column
// took 96 us for n1 = 40.
#include <cuda_runtime.h>

#include "bfq_fast.h"

namespace bfq {
namespace cay {

constexpr int kThreads = 256;

// Q1 of the parameters, row-major with row stride 2 n1 and the returned offset, in one of the two buffers [n1][2 n1] of `aug`
__device__ __forceinline__ const double* solve(const float* __restrict__ params, int n1, double* aug) {
    const int t = threadIdx.x, lane = t & 31, w = 2 * n1;
    double* cur = aug;
    double* nxt = aug + n1 * w;
    for (int e = t; e < n1 * n1; e += kThreads) {
        const int i = e / n1, j = e % n1;
        double a = 0.0;
        if (i < j) a = static_cast<double>(params[i * n1 - i * (i + 1) / 2 + (j - i - 1)]);
        if (i > j) a = -static_cast<double>(params[j * n1 - j * (j + 1) / 2 + (i - j - 1)]);
        const double id = (i == j) ? 1.0 : 0.0;
        cur[i * w + j] = id + a;
        cur[i * w + n1 + j] = id - a;
    }
    __syncthreads();
    const int tx = t & 31, ty = t >> 5;  // a warp updates consecutive columns of a row
    for (int col = 0; col < n1; ++col) {
        // the largest entry of the column from row `col` down, the first of equals (n1 <= 64: two rows per lane)
        double best = -1.0;
        int at = col;
        for (int r = col + lane; r < n1; r += 32) {
            const double v = fabs(cur[r * w + col]);
            if (v > best) best = v, at = r;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double v = __shfl_xor_sync(0xFFFFFFFFu, best, o);
            const int r = __shfl_xor_sync(0xFFFFFFFFu, at, o);
            if (v > best || (v == best && r < at)) best = v, at = r;
        }
        const double inv = 1.0 / cur[at * w + col];
        const double* pivot = cur + at * w;
        for (int j = col + 1 + tx; j < w; j += 32) {  // columns up to `col` are columns of the identity: not read again
            const double pj = pivot[j] * inv;
            for (int r = ty; r < n1; r += kThreads / 32) {
                const double* src = cur + (r == at ? col : r) * w;  // row `col` has changed places with the pivot row
                nxt[r * w + j] = r == col ? pj : src[j] - src[col] * pj;
            }
        }
        __syncthreads();
        double* tmp = cur;
        cur = nxt, nxt = tmp;
    }
    return cur + n1;
}

__global__ void __launch_bounds__(kThreads) k_cayley(const float* __restrict__ params, int n1, float* __restrict__ q1) {
    extern __shared__ double aug[];  // [2][n1][2 n1]
    const double* q = solve(params, n1, aug);
    for (int e = threadIdx.x; e < n1 * n1; e += kThreads) q1[e] = static_cast<float>(q[(e / n1) * 2 * n1 + e % n1]);
}

__global__ void __launch_bounds__(kThreads) k_cayley_backward(const float* __restrict__ params, int n1, const float* __restrict__ dq1,
                                                              float* __restrict__ dparams) {
    extern __shared__ double aug[];  // [2][n1][2 n1], then two n1 x n1 matrices
    const double* q = solve(params, n1, aug);
    const int t = threadIdx.x, w = 2 * n1, nn = n1 * n1;
    double* m2 = aug + 4 * nn;   // 2 M = I + Q1, transposed: m2[j][i] = 2 M[i][j]
    double* g = m2 + nn;         // dL/dQ1, then (2 M)^T (dL/dQ1)
    for (int e = t; e < nn; e += kThreads) {
        const int i = e / n1, j = e % n1;
        m2[j * n1 + i] = q[i * w + j] + (i == j ? 1.0 : 0.0);
        g[e] = static_cast<double>(dq1[e]);
    }
    __syncthreads();
    double* left = aug;  // the solve is done with its buffers
    for (int e = t; e < nn; e += kThreads) {  // left = (2 M)^T dQ1
        const int i = e / n1, j = e % n1;
        double s = 0.0;
        for (int k = 0; k < n1; ++k) s = fma(m2[i * n1 + k], g[k * n1 + j], s);
        left[e] = s;
    }
    __syncthreads();
    for (int e = t; e < nn; e += kThreads) {  // g = dL/dA = -left M^T
        const int i = e / n1, j = e % n1;
        double s = 0.0;
        for (int k = 0; k < n1; ++k) s = fma(left[i * n1 + k], m2[k * n1 + j], s);
        g[e] = -0.5 * s;
    }
    __syncthreads();
    for (int e = t; e < nn; e += kThreads) {
        const int i = e / n1, j = e % n1;
        if (i < j) dparams[i * n1 - i * (i + 1) / 2 + (j - i - 1)] = static_cast<float>(g[i * n1 + j] - g[j * n1 + i]);
    }
}

}  // namespace cay

template <class K>
static cudaError_t allow_smem(K kern, size_t smem) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
}

cudaError_t cayley_launch(const float* params, int n1, float* q1, cudaStream_t st) {
    const size_t smem = sizeof(double) * 4 * n1 * n1;
    cudaError_t e = allow_smem(cay::k_cayley, smem);
    if (e != cudaSuccess) return e;
    cay::k_cayley<<<1, cay::kThreads, smem, st>>>(params, n1, q1);
    return cudaGetLastError();
}

cudaError_t cayley_backward_launch(const float* params, int n1, const float* dq1, float* dparams, cudaStream_t st) {
    const size_t smem = sizeof(double) * 6 * n1 * n1;
    cudaError_t e = allow_smem(cay::k_cayley_backward, smem);
    if (e != cudaSuccess) return e;
    cay::k_cayley_backward<<<1, cay::kThreads, smem, st>>>(params, n1, dq1, dparams);
    return cudaGetLastError();
}

}  // namespace bfq
