// Backward of the composite transform (paper Sec. 3.3) in one pass over the tokens.  With a token row as an n1 x n2 matrix X,
// Y = Q1 (X Q2^T) and G = dL/dY:
//     X' = X Q2^T,  G' = Q1^T G,  dL/dX = G' Q2,  dL/dQ1 = sum G X'^T,  dL/dtheta of Q2 = the butterfly's own, on (X', G').
//
// A CTA keeps one token's X, G and G' in shared memory in fp32 (rows of n2 + 4 floats) and everything else in registers:
//   * X' in place: passes of three stages; a thread holds eight elements of a run whose three local index bits are the
//     pass's stage bits, and the same eight positions of every run it takes, so it also owns their angles;
//   * G' = Q1^T G: eight output runs x four positions per thread;
//   * dL/dQ1 += G X'^T: up to 4 x 4 entries per thread, kept over all tokens of the CTA (n1 <= 8: four slices of the
//     positions, so that all threads have work);
//   * X' and G' walked down together, d-theta in registers over all tokens, dL/dX straight from the last pass to memory.
// Multiply-adds are packed two by two (a scalar one with three register operands issues at half rate, profiled in
// bfq_fma_rates.cu): X' and G' of an element share a rotation, so do two runs on the way up; two positions, or two output runs,
// in the dense products.
// The sums of a thread, of the threads that share an angle, of the slices and of the CTAs are each added in a fixed order.
//
// All fp32 on the CUDA cores: at 40 x 128 a token takes 410 k multiply-adds for the two dense products and 110 k for the
// walks, and 20 KB of memory traffic in bf16, so the arithmetic bounds it (2048 tokens: 29 us at one multiply-add per lane and
// cycle).  Composed from a dense product on permuted copies, the butterfly backward on 40 rows per token, a forward in fp32
// and another dense product it took about 1000 us for 2048 tokens, and G' went through bf16 in between; this kernel
// takes 145 us (191 us with scalar multiply-adds).
#include "../../include/bfq.h"

#include <cuda_runtime.h>

#include "bfq_fast.h"
#include "bfq_comp_walk.cuh"
#include "bfq_generic.cuh"

namespace bfq {
namespace cbw {

constexpr int kBackwardSmem = 227 * 1024;  // dynamic shared memory of a CTA at most

struct Params {
    const float2* tw;
    const float* q1;
    int n1;
    const void* x;
    int xt;
    const void* g;
    int gt;
    int64_t ld;
    void* dx;  // type of x; may be null
    float* partial;  // [gridDim.x][L * n2 / 2 + n1 * n1]
    int64_t rows;
};

// v: (x', g') of each element
template <int L, int P, int K>
__device__ __forceinline__ void walk_down(u64 (&v)[8], const float2 (&cs)[3][4], float (&acc)[3][4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        constexpr int bit = Pair<L, P, K>::kBit;
        const int lo = Pair<L, P, K>::lo(q), hi = lo | (1 << bit);
        const u64 c = pack2(cs[K][q].x, cs[K][q].x), s = pack2(cs[K][q].y, cs[K][q].y), ns = pack2(-cs[K][q].y, -cs[K][q].y);
        const u64 a = v[lo], b = v[hi];
        float xa, ga, xb, gb;
        unpack2(a, xa, ga), unpack2(b, xb, gb);
        acc[K][q] = fmaf(gb, xa, fmaf(-ga, xb, acc[K][q]));  // on the stage's outputs
        v[lo] = fma2(s, b, mul2(c, a));
        v[hi] = fma2(ns, a, mul2(c, b));
    }
    if constexpr (K > 0) walk_down<L, P, K - 1>(v, cs, acc);
}

template <int L, int P>
__device__ __forceinline__ void passes_down(float* X, float* W, const Params& p, int64_t row, int u, int r0, float (&acc)[4][3][4]) {
    using G = Geo<L>;
    float2 cs[3][4];
    load_angles<L, P>(p.tw, u, cs);
    for (int r = r0; r < p.n1; r += G::kRuns) {
        float v[8], w[8];
        load8<L, P>(X + r * G::kPitch, u, v);
        load8<L, P>(W + r * G::kPitch, u, w);
        u64 vw[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) vw[e] = pack2(v[e], w[e]);
        walk_down<L, P, Pass<L, P>::kNs - 1>(vw, cs, acc[P]);
#pragma unroll
        for (int e = 0; e < 8; ++e) unpack2(vw[e], v[e], w[e]);
        if constexpr (P > 0) {
            store8<L, P>(X + r * G::kPitch, u, v);
            store8<L, P>(W + r * G::kPitch, u, w);
        } else if (p.dx != nullptr) {  // eight consecutive elements of dL/dX
            const int64_t off = row * p.ld + r * G::kN2 + 8 * u;
            if (p.xt == kF32) {
                float4* dst = reinterpret_cast<float4*>(static_cast<float*>(p.dx) + off);
                dst[0] = make_float4(w[0], w[1], w[2], w[3]), dst[1] = make_float4(w[4], w[5], w[6], w[7]);
            } else {
                *reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(p.dx) + off) =
                    make_uint4(pack_bf16x2(w[0], w[1]), pack_bf16x2(w[2], w[3]), pack_bf16x2(w[4], w[5]), pack_bf16x2(w[6], w[7]));
            }
        }
    }
    if constexpr (P > 0) {
        __syncthreads();
        passes_down<L, P - 1>(X, W, p, row, u, r0, acc);
    }
}

// this thread's d-theta sums into sh [kAngles], added to what is there
template <int L, int P, int K = 0>
__device__ __forceinline__ void add_angles(float* sh, int u, const float (&acc)[4][3][4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) sh[Pair<L, P, K>::angle(u, q)] += acc[P][K][q];
    if constexpr (K + 1 < Pass<L, P>::kNs) {
        add_angles<L, P, K + 1>(sh, u, acc);
    } else if constexpr (P + 1 < Geo<L>::kPasses) {
        add_angles<L, P + 1>(sh, u, acc);
    }
}

// TILES x TILES entries of dL/dQ1 per thread
template <int L, int TILES>
__global__ void __launch_bounds__(kThreads, 2) k_composite_backward(const Params p) {
    using Ge = Geo<L>;
    extern __shared__ __align__(16) float sm[];
    const int n1 = p.n1, n1p = (n1 + 7) & ~7, t = threadIdx.x;
    float* X = sm;
    float* G = X + n1 * Ge::kPitch;
    float* W = G + n1 * Ge::kPitch;
    float* q1s = W + n1 * Ge::kPitch;  // [n1][n1p], columns from n1 on zero
    for (int e = t; e < n1 * n1p; e += kThreads) {
        const int i = e / n1p, k = e % n1p;
        q1s[e] = k < n1 ? p.q1[i * n1 + k] : 0.f;
    }
    const int u = t % Ge::kU, r0 = t / Ge::kU;
    // dL/dQ1: thread (ti, tk) of a dim x dim grid has entries (ti + a dim, tk + b dim); a slice of the grid takes every
    // slices-th chunk of positions
    const int dim = n1 <= 8 ? 8 : 16, slices = kThreads / (dim * dim);
    const int slice = t / (dim * dim), tk = t % dim, ti = (t / dim) % dim;
    float acc[4][3][4];
    u64 dq[TILES][TILES];  // sums over even and over odd positions
#pragma unroll
    for (int a = 0; a < TILES; ++a)
#pragma unroll
        for (int b = 0; b < TILES; ++b) dq[a][b] = 0ull;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[a][b][c] = 0.f;

    for (int64_t row = blockIdx.x; row < p.rows; row += gridDim.x) {
        __syncthreads();  // the buffers' readers of the token before are done
        load_token<L>(p.x, p.xt, row, p.ld, n1, X);
        load_token<L>(p.g, p.gt, row, p.ld, n1, G);
        __syncthreads();
        passes_up<L, 0>(X, p.tw, n1, u, r0);
        across_runs<L>(q1s, G, W, n1, n1p);  // G' = Q1^T G
        // dL/dQ1 += G X'^T
        {
            const float *gr[TILES], *xr[TILES];
#pragma unroll
            for (int a = 0; a < TILES; ++a) {  // entries past n1 take the last run and are never written
                gr[a] = G + min(ti + a * dim, n1 - 1) * Ge::kPitch;
                xr[a] = X + min(tk + a * dim, n1 - 1) * Ge::kPitch;
            }
#pragma unroll 2
            for (int c = slice; c < Ge::kN2 / 4; c += slices) {
                const int at = place(4 * c);
                ulonglong2 xv[TILES];
#pragma unroll
                for (int b = 0; b < TILES; ++b)
                    xv[b] = *reinterpret_cast<const ulonglong2*>(xr[b] + at);
#pragma unroll
                for (int a = 0; a < TILES; ++a) {
                    const ulonglong2 gv = *reinterpret_cast<const ulonglong2*>(gr[a] + at);
#pragma unroll
                    for (int b = 0; b < TILES; ++b) {
                        dq[a][b] = fma2(gv.y, xv[b].y, fma2(gv.x, xv[b].x, dq[a][b]));
                    }
                }
            }
        }
        __syncthreads();
        passes_down<L, Ge::kPasses - 1>(X, W, p, row, u, r0, acc);
    }

    // ---- the CTA's sums, in the order of the run lanes and of the slices, to its slot ----
    __syncthreads();
    float* out = p.partial + static_cast<int64_t>(blockIdx.x) * (Ge::kAngles + n1 * n1);
    for (int e = t; e < Ge::kAngles; e += kThreads) sm[e] = 0.f;
    __syncthreads();
    for (int r = 0; r < Ge::kRuns; ++r) {
        if (r0 == r) add_angles<L, 0>(sm, u, acc);
        __syncthreads();
    }
    for (int e = t; e < Ge::kAngles; e += kThreads) out[e] = sm[e];
    __syncthreads();
    float total[TILES][TILES];
#pragma unroll
    for (int a = 0; a < TILES; ++a)
#pragma unroll
        for (int b = 0; b < TILES; ++b) {
            float even, odd;
            unpack2(dq[a][b], even, odd);
            total[a][b] = even + odd;
        }
    if (slices > 1) {  // n1 <= 8: one entry per thread
        sm[t] = total[0][0];
        __syncthreads();
        if (slice == 0) {
            for (int s = 1; s < slices; ++s) total[0][0] += sm[t + s * dim * dim];
        }
    }
    if (slice == 0) {
#pragma unroll
        for (int a = 0; a < TILES; ++a)
#pragma unroll
            for (int b = 0; b < TILES; ++b)
                if (ti + a * dim < n1 && tk + b * dim < n1) out[Ge::kAngles + (ti + a * dim) * n1 + tk + b * dim] = total[a][b];
    }
}

// dtheta [angles], dq1 [count - angles]: the slots' entries added in a fixed order (a block = 32 slot lanes x 32 entries)
__global__ void __launch_bounds__(1024) k_reduce_composite(const float* __restrict__ partial, int slots, int count, int angles,
                                                           float* __restrict__ dtheta, float* __restrict__ dq1) {
    __shared__ float sh[32][33];
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5, k = blockIdx.x * 32 + x;
    float acc = 0.f;
    if (k < count) {
#pragma unroll 4
        for (int s = y; s < slots; s += 32) acc += partial[static_cast<int64_t>(s) * count + k];
    }
    sh[y][x] = acc;
    __syncthreads();
    if (y == 0 && k < count) {
        float a = sh[0][x];
#pragma unroll
        for (int i = 1; i < 32; ++i) a += sh[i][x];
        (k < angles ? dtheta : dq1 - angles)[k] = a;
    }
}

template <int L, int TILES>
static cudaError_t launch(const bfq_plan* plan, Params p, float* dtheta, float* dq1, cudaStream_t st) {
    using G = Geo<L>;
    const int n1p = (p.n1 + 7) & ~7;
    size_t floats = size_t(3) * p.n1 * G::kPitch + size_t(p.n1) * n1p;
    if (floats < size_t(G::kAngles)) floats = G::kAngles;  // the sums at the end
    if (floats < size_t(kThreads)) floats = kThreads;
    const size_t smem = floats * sizeof(float);
    auto kern = k_composite_backward<L, TILES>;
    // as for the forward kernel: the limit of every n1, and CTAs per SM for each
    static int8_t per_sm[kMaxDevices][BFQ_MAX_N1 + 1] = {{0}};
    int8_t& occ = per_sm[plan->device][p.n1];
    cudaError_t e = cudaSuccess;
    if (occ == 0) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kBackwardSmem);
        if (e != cudaSuccess) return e;
        int o = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, kThreads, smem);
        if (e != cudaSuccess) return e;
        occ = static_cast<int8_t>(o > 0 ? o : 1);
    }
    const int count = G::kAngles + p.n1 * p.n1;
    int64_t grid = int64_t(plan->sm_count) * occ;
    if (grid > p.rows) grid = p.rows;
    if (grid * count > int64_t(plan->partial_floats)) grid = int64_t(plan->partial_floats) / count;
    if (grid < 1) return cudaErrorInvalidValue;
    kern<<<int(grid), kThreads, smem, st>>>(p);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_reduce_composite<<<(count + 31) / 32, 1024, 0, st>>>(p.partial, int(grid), count, G::kAngles, dtheta, dq1);
    return cudaGetLastError();
}

template <int L>
static cudaError_t launch(const bfq_plan* plan, const Params& p, float* dtheta, float* dq1, cudaStream_t st) {
    if (p.n1 <= 16) return launch<L, 1>(plan, p, dtheta, dq1, st);
    if (p.n1 <= 32) return launch<L, 2>(plan, p, dtheta, dq1, st);
    if (p.n1 <= 48) return launch<L, 3>(plan, p, dtheta, dq1, st);
    return launch<L, 4>(plan, p, dtheta, dq1, st);
}

}  // namespace cbw

// n1 runs of plan->n elements fit a CTA three times, and the walk is built for this n
bool composite_backward_available(const bfq_plan* plan, int n1) {
    if (plan->n < 128 || plan->n > 1024) return false;
    const size_t n1p = (n1 + 7) & ~7;
    return (size_t(3) * n1 * (plan->n + 4) + size_t(n1) * n1p) * sizeof(float) <= cbw::kBackwardSmem;
}

cudaError_t composite_backward_launch(bfq_plan* plan, const float* q1, int n1, const void* x, int xt, const void* g, int gt, int64_t rows,
                                      int64_t ld, void* dx, float* dtheta, float* dq1, cudaStream_t st) {
    cbw::Params p{};
    p.tw = plan->tw, p.q1 = q1, p.n1 = n1, p.x = x, p.xt = xt, p.g = g, p.gt = gt, p.ld = ld, p.dx = dx, p.partial = plan->partial, p.rows = rows;
    switch (plan->log_n) {
        case 7: return cbw::launch<7>(plan, p, dtheta, dq1, st);
        case 8: return cbw::launch<8>(plan, p, dtheta, dq1, st);
        case 9: return cbw::launch<9>(plan, p, dtheta, dq1, st);
        case 10: return cbw::launch<10>(plan, p, dtheta, dq1, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace bfq
