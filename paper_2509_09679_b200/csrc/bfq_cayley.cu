// The dense factor of the composite transform (paper Sec. 3.3): Q1 = (I - A)(I + A)^{-1}, A skew-symmetric, from its strict
// upper triangle, and the gradient of the parameters from the gradient of Q1.
//
// With M = (I + A)^{-1}: Q1 = 2 M - I, and dQ1 = -(I + Q1) dA M = -2 M dA M, so dL/dA = -2 M^T (dL/dQ1) M^T and the parameter
// (i < j) receives dL/dA[i][j] - dL/dA[j][i].
//
// The inverse, one CTA, float64.  The symmetric part of I + A is I, and so is at least that of every Schur complement: pivots are
// 1 and more wherever one eliminates, without a search, and entries grow by at most 1 + |A|^2 in all.  So the matrix is inverted
// in place in registers (a 16 x 16 grid of threads, up to 4 x 4 entries each, cyclic), and a column step is one chain: the owners
// of the pivot's row and column write them to shared memory, a barrier, every thread takes the reciprocal for itself and updates its
// entries.  Parameters above 32, where that growth would show in fp32 results, take Gauss-Jordan with partial pivoting on
// [I + A | I - A] (`solve`).  What bounds it is that chain.  n1 = 40: the
// pivoted solve and its gradient took 35 and 24 us, these two 14.0 and 14.8; a learning step of 2048 tokens of 40 x 128 went from 243
// to 196 us with them and the backward on matrix instructions.
//
// The gradient: M to float64 from the Q1 the caller has, and two products, on 8 x 8 x 4 float64 matrix instructions: a product on
// the plain pipe took 4 us, most of it operands from shared memory.
#include "../../include/bfq.h"

#include <cuda_runtime.h>

#include "bfq_fast.h"
#include "bfq_n4096.cuh"

namespace bfq {
namespace cay {
using namespace ptx;

constexpr int kThreads = 256;

constexpr int kMaxRows = 64 / (kThreads / 32);  // rows of a warp
__host__ __device__ constexpr int pitch(int n1) { return 2 * n1 + 1; }

// Q1 of the parameters, row-major with row stride pitch(n1), in one of the two buffers [n1][pitch] of `aug`
__device__ __forceinline__ const double* solve(const float* params, int n1, double* aug) {
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

// 1 / p for 1 <= p < 2^100: the fp32 reciprocal and two Newton steps
__device__ __forceinline__ double reciprocal(double p) {
    double r = static_cast<double>(__frcp_rn(static_cast<float>(p)));
    r = fma(r, fma(-p, r, 1.0), r);
    return fma(r, fma(-p, r, 1.0), r);
}

// T = ceil(n1 / 16): entries (ty + 16 a, tx + 16 b) of thread (tx, ty); rows and columns from n1 on are never pivots
template <int T>
__device__ __forceinline__ void invert(double (&m)[T][T], int n1, double (&line)[2][2][64]) {
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    auto publish = [&](int k) {  // row k and column k
        double(&to)[2][64] = line[k & 1];
#pragma unroll
        for (int a = 0; a < T; ++a)
            if (ty + 16 * a == k) {
#pragma unroll
                for (int b = 0; b < T; ++b) to[0][tx + 16 * b] = m[a][b];
            }
#pragma unroll
        for (int b = 0; b < T; ++b)
            if (tx + 16 * b == k) {
#pragma unroll
                for (int a = 0; a < T; ++a) to[1][ty + 16 * a] = m[a][b];
            }
        __syncthreads();
    };
    for (int k = 0; k < n1; ++k) {
        publish(k);
        const double(&at)[2][64] = line[k & 1];
        double row[T], col[T];
#pragma unroll
        for (int a = 0; a < T; ++a) row[a] = at[0][tx + 16 * a], col[a] = at[1][ty + 16 * a];
        const double inv = reciprocal(at[0][k]);
#pragma unroll
        for (int b = 0; b < T; ++b) row[b] *= inv;
#pragma unroll
        for (int a = 0; a < T; ++a)
#pragma unroll
            for (int b = 0; b < T; ++b) {
                const bool in_row = ty + 16 * a == k, in_col = tx + 16 * b == k;
                const double other = fma(-col[a], row[b], m[a][b]);
                m[a][b] = in_row ? (in_col ? inv : row[b]) : (in_col ? -col[a] * inv : other);
            }
    }
}

__device__ __forceinline__ float parameter(const float* params, int n1, int i, int j) {  // A[i][j]
    if (i == j) return 0.f;
    const int lo = min(i, j), hi = max(i, j);
    const float v = params[lo * n1 - lo * (lo + 1) / 2 + (hi - lo - 1)];
    return i < j ? v : -v;
}

template <int T>
__global__ void __launch_bounds__(kThreads) k_cayley(const float* params, int n1, float* __restrict__ q1) {
    extern __shared__ double aug[];  // [2][n1][pitch], for `solve`
    __shared__ double line[2][2][64];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    grid_dep_launch();
    grid_dep_wait();
    double m[T][T];
    bool large = false;
#pragma unroll
    for (int a = 0; a < T; ++a)
#pragma unroll
        for (int b = 0; b < T; ++b) {
            const int i = ty + 16 * a, j = tx + 16 * b;
            const float v = i < n1 && j < n1 ? parameter(params, n1, i, j) : 0.f;
            large |= !(fabsf(v) <= 32.f);
            m[a][b] = static_cast<double>(v) + (i == j ? 1.0 : 0.0);
        }
    if (__syncthreads_or(large)) {
        const double* q = solve(params, n1, aug);
        for (int e = threadIdx.x; e < n1 * n1; e += kThreads) q1[e] = static_cast<float>(q[(e / n1) * pitch(n1) + e % n1]);
        return;
    }
    invert<T>(m, n1, line);
#pragma unroll
    for (int a = 0; a < T; ++a)
#pragma unroll
        for (int b = 0; b < T; ++b) {
            const int i = ty + 16 * a, j = tx + 16 * b;
            if (i < n1 && j < n1) q1[i * n1 + j] = static_cast<float>(2.0 * m[a][b] - (i == j ? 1.0 : 0.0));
        }
}

// matrices of the gradient: np = n1 rounded up to 8 rows of np + 4 numbers, zero from n1 on (the pitch spreads the eight rows of a
// fragment over the banks)
__host__ __device__ constexpr int padded(int n1) { return (n1 + 7) & ~7; }
__host__ __device__ constexpr int row_of(int n1) { return padded(n1) + 4; }

__device__ __forceinline__ void mma_884(double (&c)[2], double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};" : "+d"(c[0]), "+d"(c[1]) : "d"(a), "d"(b));
}

// out = scale op(a) op(b) + add I: a warp takes 8 x 8 blocks, all its blocks' chains side by side.  AT / BT: the operand is stored
// transposed.  Ends in a barrier.
template <bool AT, bool BT>
__device__ __forceinline__ void product(double* out, const double* a, const double* b, int n1, double scale, double add) {
    constexpr int kWarps = kThreads / 32, kMost = 64 / kWarps;  // blocks of a warp at most
    const int nb = padded(n1) / 8, blocks = nb * nb, w = row_of(n1), warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
    const int mine = (blocks - warp + kWarps - 1) / kWarps;
    double acc[kMost][2];
    const double *pa[kMost], *pb[kMost];
#pragma unroll
    for (int i = 0; i < kMost; ++i) {
        const int blk = min(warp + i * kWarps, blocks - 1), bi = 8 * (blk / nb), bj = 8 * (blk % nb);
        acc[i][0] = acc[i][1] = 0.0;
        pa[i] = AT ? a + q * w + bi + g : a + (bi + g) * w + q;
        pb[i] = BT ? b + (bj + g) * w + q : b + q * w + bj + g;
    }
    for (int k = 0; k < 2 * nb; ++k) {
#pragma unroll
        for (int i = 0; i < kMost; ++i)
            if (i < mine) mma_884(acc[i], pa[i][AT ? 4 * k * w : 4 * k], pb[i][BT ? 4 * k : 4 * k * w]);
    }
#pragma unroll
    for (int i = 0; i < kMost; ++i) {
        if (i >= mine) continue;
        const int blk = warp + i * kWarps, r = 8 * (blk / nb) + g, c = 8 * (blk % nb) + 2 * q;
        out[r * w + c] = scale * acc[i][0] + (r == c ? add : 0.0);
        out[r * w + c + 1] = scale * acc[i][1] + (r == c + 1 ? add : 0.0);
    }
    __syncthreads();
}

// M = (I + A)^{-1} in float64 from the Q1 the caller has: (I + Q1) / 2 is M to fp32 rounding (residual up to |A| 2^-24), and a
// Newton step M (2 I - (I + A) M) squares the residual; a second one follows where the first residual's square is not far below
// fp32 rounding.  If Q1 is not the transform of these parameters (the first residual is not small) the solve is done after all.
__global__ void __launch_bounds__(kThreads) k_cayley_backward(const float* params, int n1, const float* q1,
                                                              const float* dq1, float* __restrict__ dparams) {
    extern __shared__ double aug[];  // [2][n1][pitch] of the solve, or I + A, M, 2 I - (I + A) M, the next M; then dQ1
    const int t = threadIdx.x, np = padded(n1), w = row_of(n1), size = np * w;
    double *ia = aug, *m = ia + size, *r = m + size, *next = r + size, *g = next + size;
    grid_dep_launch();
    grid_dep_wait();
    for (int e = t; e < np * np; e += kThreads) {
        const int i = e / np, j = e % np, at = i * w + j;
        const bool in = i < n1 && j < n1;
        const double id = i == j ? 1.0 : 0.0;
        ia[at] = in ? id + static_cast<double>(parameter(params, n1, i, j)) : 0.0;
        m[at] = in ? 0.5 * (id + static_cast<double>(q1[i * n1 + j])) : 0.0;
        g[at] = in ? static_cast<double>(dq1[i * n1 + j]) : 0.0;
    }
    __syncthreads();
    // whether an entry of I - (I + A) M is not below a limit (NaN is not); rows and columns from n1 on hold 2 I there
    auto above = [&](double limit) {
        bool far = false;
        for (int e = t; e < n1 * n1; e += kThreads) {
            const int i = e / n1, j = e % n1;
            far |= !(fabs(r[i * w + j] - (i == j ? 1.0 : 0.0)) < limit);
        }
        return __syncthreads_or(far) != 0;
    };
    product<false, false>(r, ia, m, n1, -1.0, 2.0);
    if (!above(1e-4)) {
        const bool twice = above(1e-6);  // else the residual's square, at most 64^2 1e-12, leaves M better than 4e-9
        product<false, false>(next, m, r, n1, 1.0, 0.0);
        double* done = next;
        if (twice) {
            product<false, false>(r, ia, next, n1, -1.0, 2.0);
            product<false, false>(m, next, r, n1, 1.0, 0.0);
            done = m;
        }
        m = done;
    } else {
        const double* q = solve(params, n1, aug);  // dQ1 lies behind its two buffers
        __syncthreads();
        double keep[64 * 64 / kThreads];
#pragma unroll
        for (int e = 0; e < 64 * 64 / kThreads; ++e) {  // 2 M = I + Q1, while the solve's buffers turn back into matrices
            const int at = t + e * kThreads, i = at / np, j = at % np;
            keep[e] = at < np * np && i < n1 && j < n1 ? 0.5 * (q[i * pitch(n1) + j] + (i == j ? 1.0 : 0.0)) : 0.0;
        }
        __syncthreads();
        m = aug;
#pragma unroll
        for (int e = 0; e < 64 * 64 / kThreads; ++e) {
            const int at = t + e * kThreads;
            if (at < np * np) m[(at / np) * w + at % np] = keep[e];
        }
        __syncthreads();
    }
    // dL/dA = -2 M^T dQ1 M^T
    double *left = m == ia ? r : ia, *both = r == left ? next : r;
    product<true, false>(left, m, g, n1, 1.0, 0.0);
    product<false, true>(both, left, m, n1, -2.0, 0.0);
    for (int e = t; e < n1 * n1; e += kThreads) {
        const int i = e / n1, j = e % n1;
        if (i < j) dparams[i * n1 - i * (i + 1) / 2 + (j - i - 1)] = static_cast<float>(both[i * w + j] - both[j * w + i]);
    }
}

}  // namespace cay

// shared memory for n1 rows, and the limit of every n1: set once per device (a limit per call would be pulled away by another
// thread's call with a smaller n1)
static constexpr size_t cayley_smem(int n1) { return sizeof(double) * 2 * n1 * cay::pitch(n1); }
static constexpr size_t cayley_backward_smem(int n1) { return sizeof(double) * 5 * cay::padded(n1) * cay::row_of(n1); }
static_assert(4 * cay::padded(64) * cay::row_of(64) >= 2 * 64 * cay::pitch(64) && cayley_backward_smem(64) <= 227 * 1024, "room for the solve, and in a CTA");
template <class F>
static cudaError_t for_tile(int n1, F&& f) {
    if (n1 <= 16) return f(cay::k_cayley<1>);
    if (n1 <= 32) return f(cay::k_cayley<2>);
    if (n1 <= 48) return f(cay::k_cayley<3>);
    return f(cay::k_cayley<4>);
}
static cudaError_t allow_smem(int device) {
    static bool allowed[kMaxDevices] = {false};
    if (allowed[device]) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(cay::k_cayley_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, int(cayley_backward_smem(BFQ_MAX_N1)));
    for (int n1 = 16; n1 <= 64; n1 += 16)
        if (e == cudaSuccess)
            e = for_tile(n1, [](auto kern) { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(cayley_smem(BFQ_MAX_N1))); });
    allowed[device] = e == cudaSuccess;
    return e;
}

cudaError_t cayley_launch(const bfq_plan* plan, const float* params, int n1, float* q1, cudaStream_t st) {
    cudaError_t e = allow_smem(plan->device);
    if (e != cudaSuccess) return e;
    return for_tile(n1, [&](auto kern) { return launch_overlapped(kern, dim3(1), dim3(cay::kThreads), cayley_smem(n1), st, params, n1, q1); });
}

cudaError_t cayley_backward_launch(const bfq_plan* plan, const float* params, int n1, const float* q1, const float* dq1, float* dparams, cudaStream_t st) {
    cudaError_t e = allow_smem(plan->device);
    if (e != cudaSuccess) return e;
    return launch_overlapped(cay::k_cayley_backward, dim3(1), dim3(cay::kThreads), cayley_backward_smem(n1), st, params, n1, q1, dq1, dparams);
}

}  // namespace bfq
