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
// one block barrier per column; every warp finds the pivot by itself; a row is 2 n1 + 1 doubles, so that the lanes that read
// down a column fall into different banks, and a thread's loads are all issued before its stores.  Four barriers and a serial
// pivot search per column took 96 us for n1 = 40; now 35 us, and the gradient 24 us (76 with a solve of its own).
#include "../../include/bfq.h"

#include <cuda_runtime.h>

#include "bfq_fast.h"

namespace bfq {
namespace cay {

constexpr int kThreads = 256;

constexpr int kMaxRows = 64 / (kThreads / 32);  // rows of a warp
__host__ __device__ constexpr int pitch(int n1) { return 2 * n1 + 1; }

// Q1 of the parameters, row-major with row stride pitch(n1), in one of the two buffers [n1][pitch] of `aug`
__device__ __forceinline__ const double* solve(const float* __restrict__ params, int n1, double* aug) {
    const int t = threadIdx.x, lane = t & 31, w = pitch(n1), cols = 2 * n1;
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
        // the largest entry of the column from row `col` down, compared in fp32 to 17 bits (as good a pivot as the largest), the
        // row in the low bits so that one integer reduction gives both; n1 <= 64: two rows per lane
        uint32_t key = 0u;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = lane + 32 * h;
            if (r >= col && r < n1) key = max(key, (__float_as_uint(fabsf(static_cast<float>(cur[r * w + col]))) & ~63u) | (63u - r));
        }
        const int at = 63 - static_cast<int>(__reduce_max_sync(0xFFFFFFFFu, key) & 63u);
        const double inv = 1.0 / cur[at * w + col];
        const double* pivot = cur + at * w;
        const double* src[kMaxRows];  // row `col` has changed places with the pivot row
        double f[kMaxRows];
#pragma unroll
        for (int a = 0; a < kMaxRows; ++a) {
            const int r = ty + a * (kThreads / 32);  // the same for the whole warp
            src[a] = cur + (r == at ? col : r) * w;
            f[a] = r < n1 ? src[a][col] : 0.0;
        }
        for (int j = col + 1 + tx; j < cols; j += 32) {  // columns up to `col` are columns of the identity: not read again
            const double pj = pivot[j] * inv;
            double v[kMaxRows];
#pragma unroll
            for (int a = 0; a < kMaxRows; ++a) v[a] = ty + a * (kThreads / 32) < n1 ? src[a][j] : 0.0;
#pragma unroll
            for (int a = 0; a < kMaxRows; ++a) {
                const int r = ty + a * (kThreads / 32);
                if (r < n1) nxt[r * w + j] = r == col ? pj : v[a] - f[a] * pj;
            }
        }
        __syncthreads();
        double* tmp = cur;
        cur = nxt, nxt = tmp;
    }
    return cur + n1;
}

__global__ void __launch_bounds__(kThreads) k_cayley(const float* __restrict__ params, int n1, float* __restrict__ q1) {
    extern __shared__ double aug[];  // [2][n1][pitch]
    const double* q = solve(params, n1, aug);
    for (int e = threadIdx.x; e < n1 * n1; e += kThreads) q1[e] = static_cast<float>(q[(e / n1) * pitch(n1) + e % n1]);
}

// out = scale a b + add I (n1 x n1, row stride n1, all threads): four rows x two columns per thread, so that eight chains
// overlap and a value that is read serves several of them
__device__ __forceinline__ void product(double* out, const double* a, const double* b, int n1, double scale, double add) {
    const int cols = (n1 + 1) / 2, items = ((n1 + 3) / 4) * cols;
    for (int it = threadIdx.x; it < items; it += kThreads) {
        const int i0 = 4 * (it / cols), j0 = 2 * (it % cols), j1 = min(j0 + 1, n1 - 1);
        double s[4][2];
        const double* row[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) s[r][0] = s[r][1] = 0.0, row[r] = a + min(i0 + r, n1 - 1) * n1;
#pragma unroll 4
        for (int k = 0; k < n1; ++k) {
            const double x = b[k * n1 + j0], y = b[k * n1 + j1];
#pragma unroll
            for (int r = 0; r < 4; ++r) s[r][0] = fma(row[r][k], x, s[r][0]), s[r][1] = fma(row[r][k], y, s[r][1]);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 2; ++c)
                if (i0 + r < n1 && j0 + c < n1) out[(i0 + r) * n1 + j0 + c] = scale * s[r][c] + (i0 + r == j0 + c ? add : 0.0);
    }
}

// M = (I + A)^{-1} in float64 from the Q1 the caller has: (I + Q1) / 2 is M to fp32 rounding, and each Newton step
// M (2 I - (I + A) M) squares the error (residual of the first guess up to |A| 2^-24; two steps).  If Q1 is not the transform of
// these parameters (the first residual is not small) the solve is done after all.  Six small products instead of a solve.
__global__ void __launch_bounds__(kThreads) k_cayley_backward(const float* __restrict__ params, int n1, const float* __restrict__ q1,
                                                              const float* __restrict__ dq1, float* __restrict__ dparams) {
    extern __shared__ double aug[];  // [2][n1][pitch] of the solve = four n1 x n1 matrices and more, then two
    const int t = threadIdx.x, nn = n1 * n1;
    double *ia = aug, *m = ia + nn, *r = m + nn, *next = r + nn;  // I + A, M, 2 I - (I + A) M, the next M
    double* g = aug + 2 * n1 * pitch(n1);
    double* left = g + nn;
    __shared__ int far;
    if (t == 0) far = 0;
    for (int e = t; e < nn; e += kThreads) {
        const int i = e / n1, j = e % n1;
        double a = 0.0;
        if (i < j) a = static_cast<double>(params[i * n1 - i * (i + 1) / 2 + (j - i - 1)]);
        if (i > j) a = -static_cast<double>(params[j * n1 - j * (j + 1) / 2 + (i - j - 1)]);
        const double id = i == j ? 1.0 : 0.0;
        ia[e] = id + a;
        m[e] = 0.5 * (id + static_cast<double>(q1[e]));
        g[e] = static_cast<double>(dq1[e]);
    }
    __syncthreads();
    for (int step = 0; step < 2; ++step) {
        product(r, ia, m, n1, -1.0, 2.0);
        __syncthreads();
        if (step == 0) {
            for (int e = t; e < nn; e += kThreads)
                if (!(fabs(r[e] - (e / n1 == e % n1 ? 1.0 : 0.0)) < 1e-4)) far = 1;
            __syncthreads();
            if (far != 0) break;
        }
        product(next, m, r, n1, 1.0, 0.0);
        __syncthreads();
        double* tmp = m;
        m = next, next = tmp;
    }
    if (far != 0) {  // uniform
        const double* q = solve(params, n1, aug);
        // 2 M = I + Q1, kept in `left` while the solve's buffers turn back into matrices
        for (int e = t; e < nn; e += kThreads) left[e] = 0.5 * (q[(e / n1) * pitch(n1) + e % n1] + (e / n1 == e % n1 ? 1.0 : 0.0));
        __syncthreads();
        m = aug;
        for (int e = t; e < nn; e += kThreads) m[e] = left[e];
        __syncthreads();
        r = aug + nn;
    }
    // dL/dA = -2 M^T dQ1 M^T; M^T in r
    for (int e = t; e < nn; e += kThreads) r[(e % n1) * n1 + e / n1] = m[e];
    __syncthreads();
    product(left, r, g, n1, 1.0, 0.0);
    __syncthreads();
    product(g, left, r, n1, -2.0, 0.0);
    __syncthreads();
    for (int e = t; e < nn; e += kThreads) {
        const int i = e / n1, j = e % n1;
        if (i < j) dparams[i * n1 - i * (i + 1) / 2 + (j - i - 1)] = static_cast<float>(g[i * n1 + j] - g[j * n1 + i]);
    }
}

}  // namespace cay

// shared memory for n1 rows, and the limit of every n1: set once per device (a limit per call would be pulled away by another
// thread's call with a smaller n1)
static constexpr size_t cayley_smem(int n1) { return sizeof(double) * 2 * n1 * cay::pitch(n1); }
static constexpr size_t cayley_backward_smem(int n1) { return cayley_smem(n1) + sizeof(double) * 2 * n1 * n1; }
static cudaError_t allow_smem(int device) {
    static bool allowed[kMaxDevices] = {false};
    if (allowed[device]) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(cay::k_cayley, cudaFuncAttributeMaxDynamicSharedMemorySize, int(cayley_smem(BFQ_MAX_N1)));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(cay::k_cayley_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, int(cayley_backward_smem(BFQ_MAX_N1)));
    allowed[device] = e == cudaSuccess;
    return e;
}

cudaError_t cayley_launch(const bfq_plan* plan, const float* params, int n1, float* q1, cudaStream_t st) {
    cudaError_t e = allow_smem(plan->device);
    if (e != cudaSuccess) return e;
    cay::k_cayley<<<1, cay::kThreads, cayley_smem(n1), st>>>(params, n1, q1);
    return cudaGetLastError();
}

cudaError_t cayley_backward_launch(const bfq_plan* plan, const float* params, int n1, const float* q1, const float* dq1, float* dparams, cudaStream_t st) {
    cudaError_t e = allow_smem(plan->device);
    if (e != cudaSuccess) return e;
    cay::k_cayley_backward<<<1, cay::kThreads, cayley_backward_smem(n1), st>>>(params, n1, q1, dq1, dparams);
    return cudaGetLastError();
}

}  // namespace bfq
