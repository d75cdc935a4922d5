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
#include <cuda_runtime.h>

#include "bfq_fast.h"
#include "bfq_generic.cuh"
#include "bfq_ptx.cuh"

namespace bfq {
namespace cbw {
using namespace ptx;

constexpr int kThreads = 256;

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

// A run's floats in shared memory: 16-byte chunk c sits at chunk c ^ (bits 4, 5 of c, shifted to 1, 2), so that the eight
// consecutive floats that lanes read at strides of 64 (second pass) fall into different banks.
__device__ __forceinline__ int place(int i) {
    const int c = i >> 2;
    return ((c ^ (((c >> 4) & 3) << 1)) << 2) | (i & 3);
}

// pass P of the butterfly on n2 = 2^L points: stages B0 .. B0 + NS - 1, local bits = F lowest index bits (filler), then those
template <int L, int P>
struct Pass {
    static constexpr int kB0 = 3 * P, kNs = L - kB0 >= 3 ? 3 : L - kB0, kF = 3 - kNs, kMid = kB0 - kF;
    __device__ __forceinline__ static int idx(int u, int e) {
        return (e & ((1 << kF) - 1)) | ((u & ((1 << kMid) - 1)) << kF) | ((e >> kF) << kB0) | ((u >> kMid) << (kB0 + kNs));
    }
    // consecutive elements a thread holds
    static constexpr int kRun = P == 0 ? 8 : (1 << kF);
};

template <int L, int P>
__device__ __forceinline__ void load8(const float* run, int u, float (&v)[8]) {
    using PS = Pass<L, P>;
    if constexpr (PS::kRun >= 4) {
#pragma unroll
        for (int e = 0; e < 8; e += 4) {
            const float4 f = *reinterpret_cast<const float4*>(run + place(PS::idx(u, e)));
            v[e] = f.x, v[e + 1] = f.y, v[e + 2] = f.z, v[e + 3] = f.w;
        }
    } else if constexpr (PS::kRun == 2) {
#pragma unroll
        for (int e = 0; e < 8; e += 2) {
            const float2 f = *reinterpret_cast<const float2*>(run + place(PS::idx(u, e)));
            v[e] = f.x, v[e + 1] = f.y;
        }
    } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = run[place(PS::idx(u, e))];
    }
}
template <int L, int P>
__device__ __forceinline__ void store8(float* run, int u, const float (&v)[8]) {
    using PS = Pass<L, P>;
    if constexpr (PS::kRun >= 4) {
#pragma unroll
        for (int e = 0; e < 8; e += 4) *reinterpret_cast<float4*>(run + place(PS::idx(u, e))) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
    } else if constexpr (PS::kRun == 2) {
#pragma unroll
        for (int e = 0; e < 8; e += 2) *reinterpret_cast<float2*>(run + place(PS::idx(u, e))) = make_float2(v[e], v[e + 1]);
    } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) run[place(PS::idx(u, e))] = v[e];
    }
}

// pair q of local stage K: its elements, and its angle's index within the stage
template <int L, int P, int K>
struct Pair {
    static constexpr int kBit = Pass<L, P>::kF + K, kStage = Pass<L, P>::kB0 + K;
    __device__ __forceinline__ static constexpr int lo(int q) { return ((q >> kBit) << (kBit + 1)) | (q & ((1 << kBit) - 1)); }
    __device__ __forceinline__ static int angle(int u, int q) {
        const int i = Pass<L, P>::idx(u, lo(q));
        return (kStage << (L - 1)) + (((i >> (kStage + 1)) << kStage) | (i & ((1 << kStage) - 1)));
    }
};

template <int L, int P, int K = 0>
__device__ __forceinline__ void load_angles(const float2* __restrict__ tw, int u, float2 (&cs)[3][4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) cs[K][q] = __ldg(tw + Pair<L, P, K>::angle(u, q));
    if constexpr (K + 1 < Pass<L, P>::kNs) load_angles<L, P, K + 1>(tw, u, cs);
}

// two runs at once
template <int L, int P, int K = 0>
__device__ __forceinline__ void rotate(u64 (&v)[8], const float2 (&cs)[3][4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        constexpr int bit = Pair<L, P, K>::kBit;
        const int lo = Pair<L, P, K>::lo(q), hi = lo | (1 << bit);
        const u64 c = pack2(cs[K][q].x, cs[K][q].x), s = pack2(cs[K][q].y, cs[K][q].y), ns = pack2(-cs[K][q].y, -cs[K][q].y);
        const u64 a = v[lo], b = v[hi];
        v[lo] = fma2(ns, b, mul2(c, a));
        v[hi] = fma2(s, a, mul2(c, b));
    }
    if constexpr (K + 1 < Pass<L, P>::kNs) rotate<L, P, K + 1>(v, cs);
}

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

template <int L>
struct Geo {
    static constexpr int kN2 = 1 << L, kPasses = (L + 2) / 3, kU = kN2 / 8, kRuns = kThreads / kU;  // runs side by side
    static constexpr int kPitch = kN2 + 4;
    static constexpr int kAngles = L * kN2 / 2;
};

template <int L, int P>
__device__ __forceinline__ void passes_up(float* X, const Params& p, int u, int r0) {
    using G = Geo<L>;
    float2 cs[3][4];
    load_angles<L, P>(p.tw, u, cs);
    for (int r = r0; r < p.n1; r += 2 * G::kRuns) {
        const bool two = r + G::kRuns < p.n1;
        float* second = X + (two ? r + G::kRuns : r) * G::kPitch;
        float v[8], w[8];
        load8<L, P>(X + r * G::kPitch, u, v);
        load8<L, P>(second, u, w);
        u64 vw[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) vw[e] = pack2(v[e], w[e]);
        rotate<L, P>(vw, cs);
#pragma unroll
        for (int e = 0; e < 8; ++e) unpack2(vw[e], v[e], w[e]);
        store8<L, P>(X + r * G::kPitch, u, v);
        if (two) store8<L, P>(second, u, w);
    }
    __syncthreads();
    if constexpr (P + 1 < G::kPasses) passes_up<L, P + 1>(X, p, u, r0);
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

template <int L>
__device__ __forceinline__ void load_token(const void* base, int type, int64_t row, int64_t ld, int n1, float* to) {
    using G = Geo<L>;
    const int t = threadIdx.x;
    if (type == kF32) {
        const float4* src = reinterpret_cast<const float4*>(static_cast<const float*>(base) + row * ld);
        for (int c = t; c < n1 * (G::kN2 / 4); c += kThreads) {
            const int r = c / (G::kN2 / 4), i = 4 * (c % (G::kN2 / 4));
            *reinterpret_cast<float4*>(to + r * G::kPitch + place(i)) = __ldg(src + c);
        }
    } else {
        const uint4* src = reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(base) + row * ld);
        for (int c = t; c < n1 * (G::kN2 / 8); c += kThreads) {
            const int r = c / (G::kN2 / 8), i = 8 * (c % (G::kN2 / 8));
            const uint4 w = __ldg(src + c);
            auto lo = [](uint32_t b) { return __uint_as_float(b << 16); };
            auto hi = [](uint32_t b) { return __uint_as_float(b & 0xFFFF0000u); };
            *reinterpret_cast<float4*>(to + r * G::kPitch + place(i)) = make_float4(lo(w.x), hi(w.x), lo(w.y), hi(w.y));
            *reinterpret_cast<float4*>(to + r * G::kPitch + place(i + 4)) = make_float4(lo(w.z), hi(w.z), lo(w.w), hi(w.w));
        }
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
        passes_up<L, 0>(X, p, u, r0);
        // G' = Q1^T G
        for (int item = t; item < (n1p / 8) * (Ge::kN2 / 4); item += kThreads) {
            const int j = place(4 * (item % (Ge::kN2 / 4))), k0 = 8 * (item / (Ge::kN2 / 4));
            u64 s[4][4];  // output runs k0 + 2a, k0 + 2a + 1 at position b
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) s[a][b] = 0ull;
#pragma unroll 4
            for (int i = 0; i < n1; ++i) {
                const float4 gv = *reinterpret_cast<const float4*>(G + i * Ge::kPitch + j);
                const ulonglong2 qa = *reinterpret_cast<const ulonglong2*>(q1s + i * n1p + k0), qb = *reinterpret_cast<const ulonglong2*>(q1s + i * n1p + k0 + 4);
                const u64 qs[4] = {qa.x, qa.y, qb.x, qb.y};
                const u64 gs[4] = {pack2(gv.x, gv.x), pack2(gv.y, gv.y), pack2(gv.z, gv.z), pack2(gv.w, gv.w)};
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int b = 0; b < 4; ++b) s[a][b] = fma2(qs[a], gs[b], s[a][b]);
            }
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                float lo[4], hi[4];
#pragma unroll
                for (int b = 0; b < 4; ++b) unpack2(s[a][b], lo[b], hi[b]);
                if (k0 + 2 * a < n1) *reinterpret_cast<float4*>(W + (k0 + 2 * a) * Ge::kPitch + j) = make_float4(lo[0], lo[1], lo[2], lo[3]);
                if (k0 + 2 * a + 1 < n1) *reinterpret_cast<float4*>(W + (k0 + 2 * a + 1) * Ge::kPitch + j) = make_float4(hi[0], hi[1], hi[2], hi[3]);
            }
        }
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
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    int occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kThreads, smem);
    if (e != cudaSuccess) return e;
    const int count = G::kAngles + p.n1 * p.n1;
    int64_t grid = int64_t(plan->sm_count) * (occ > 0 ? occ : 1);
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
    return (size_t(3) * n1 * (plan->n + 4) + size_t(n1) * n1p) * sizeof(float) <= 227 * 1024;
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
