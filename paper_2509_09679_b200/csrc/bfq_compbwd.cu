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
// takes 143 us (191 us with scalar multiply-adds) where G is fp32; bf16 G: k_composite_backward_mma, 112 us.
#include "../../include/bfq.h"

#include <cuda_bf16.h>
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

// ---- bf16 gradients: the two dense products on the tensor cores ----------------------------------------------------
// G in bf16 is an exact operand.  The other one, Q1 or X', goes in as three bf16 terms, 24 significant bits, so the products are those of
// fp32 numbers and their sums are fp32 (m16n8k16; the small terms first or apart).  G stays in shared memory as bf16 rows, read as
// matrices of 8 x 8 either way; Q1's terms are there as fragments; X' is split as it is read.
// An infinity has no such terms (infinity less itself, or times a term that is zero, is NaN): products that are not finite are formed
// again in fp32, so that infinities stay infinities.
// (a, b) = t[0] + t[1] + t[2], largest first: eight significant bits each, cut off, so that the sum is exact
__device__ __forceinline__ void three_terms(float a, float b, uint32_t (&t)[3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        t[i] = __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
        a -= __uint_as_float(__float_as_uint(a) & 0xFFFF0000u), b -= __uint_as_float(__float_as_uint(b) & 0xFFFF0000u);
    }
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint4& a, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint4 matrices(uint32_t at) {
    uint4 v;
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(at) : "memory");
    return v;
}
__device__ __forceinline__ uint4 matrices_transposed(uint32_t at) {
    uint4 v;
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(at) : "memory");
    return v;
}

__device__ __forceinline__ bool finite(float v) { return fabsf(v) <= 3.402823466e38f; }
__device__ __forceinline__ float bf16_at(const uint16_t* p) { return __uint_as_float(static_cast<uint32_t>(*p) << 16); }

constexpr int kWarps = kThreads / 32;
// MT blocks of 16 runs.  dL/dQ1 is cut into tiles of 16 x 8, a warp has up to kTiles of them; with fewer tiles than warps, slices of the
// positions go to different warps
template <int L, int MT>
struct Mma {
    static constexpr int kTiles = MT <= 2 ? 1 : MT, kRow = (1 << L) + 8;  // bf16 of a row of G: 16 bytes off a multiple of 128
    static constexpr int kFragments = 3 * MT * MT * 32;                   // uint4 of Q1
    static size_t smem(int n1) { return size_t(16) * kFragments + size_t(2) * 16 * MT * kRow + sizeof(float) * 2 * n1 * Geo<L>::kPitch; }
};

template <int L, int MT>
__global__ void __launch_bounds__(kThreads, 2) k_composite_backward_mma(const Params p) {
    using Ge = Geo<L>;
    using M = Mma<L, MT>;
    extern __shared__ __align__(16) uint4 sm4[];
    const int n1 = p.n1, t = threadIdx.x, warp = t >> 5, lane = t & 31, g8 = lane >> 2, q = lane & 3;
    uint4* const frag = sm4;  // [term][block of k][block of rows][lane]: element [row][k] = Q1[k][row]
    uint16_t* const Gb = reinterpret_cast<uint16_t*>(sm4 + M::kFragments);
    float* const X = reinterpret_cast<float*>(Gb + 16 * MT * M::kRow);
    float* const W = X + n1 * Ge::kPitch;
    for (int e = t; e < MT * MT * 32; e += kThreads) {
        const int l = e & 31, mt = (e >> 5) % MT, kt = (e >> 5) / MT;
        uint32_t w[4][3];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int row = 16 * mt + (l >> 2) + 8 * (r & 1), k = 16 * kt + 2 * (l & 3) + 8 * (r >> 1);
            auto at = [&](int i) { return i < n1 && row < n1 ? p.q1[i * n1 + row] : 0.f; };
            three_terms(at(k), at(k + 1), w[r]);
            if (isinf(at(k))) w[r][1] &= 0xFFFF0000u, w[r][2] &= 0xFFFF0000u;
            if (isinf(at(k + 1))) w[r][1] &= 0xFFFFu, w[r][2] &= 0xFFFFu;
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) frag[i * MT * MT * 32 + e] = make_uint4(w[0][i], w[1][i], w[2][i], w[3][i]);
    }
    for (int e = n1 * M::kRow + t; e < 16 * MT * M::kRow; e += kThreads) Gb[e] = 0;  // runs that do not exist
    const uint32_t gbase = smem_u32(Gb);
    const int u = t % Ge::kU, r0 = t / Ge::kU;
    const int nt = (n1 + 7) / 8, tiles = MT * nt;
    const int slices = tiles >= kWarps ? 1 : kWarps / tiles, slice = tiles >= kWarps ? 0 : warp / tiles;
    const int first_tile = tiles >= kWarps ? warp : (slice < slices ? warp % tiles : tiles);
    float acc[4][3][4], dq[M::kTiles][4];
#pragma unroll
    for (int i = 0; i < 48; ++i) acc[i / 12][i / 4 % 3][i & 3] = 0.f;
#pragma unroll
    for (int i = 0; i < 4 * M::kTiles; ++i) dq[i >> 2][i & 3] = 0.f;

    for (int64_t row = blockIdx.x; row < p.rows; row += gridDim.x) {
        __syncthreads();  // the buffers' readers of the token before are done
        load_token<L>(p.x, p.xt, row, p.ld, n1, X);
        {
            const uint4* src = reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(p.g) + row * p.ld);
            for (int c = t; c < n1 * (Ge::kN2 / 8); c += kThreads)
                *reinterpret_cast<uint4*>(Gb + (c / (Ge::kN2 / 8)) * M::kRow + 8 * (c % (Ge::kN2 / 8))) = __ldg(src + c);
        }
        __syncthreads();
        // G' = Q1^T G: a warp takes 16 positions at a time
        for (int j0 = 16 * warp; j0 < Ge::kN2; j0 += 16 * kWarps) {
            uint4 b[MT];
            float s[MT][2][4];
            float least[2][4];  // MT = 1: the sums of the small terms, apart
#pragma unroll
            for (int kt = 0; kt < MT; ++kt) b[kt] = matrices_transposed(gbase + 2u * ((16 * kt + (lane & 15)) * M::kRow + j0 + 8 * (lane >> 4)));
#pragma unroll
            for (int i = 0; i < 8 * MT; ++i) s[i >> 3][(i >> 2) & 1][i & 3] = 0.f;
#pragma unroll
            for (int term = 2; term >= 0; --term) {
                if constexpr (MT == 1) {  // an MMA cuts its sum off: with a few runs that shows (dx, n1 = 2: 1.15e-7, so 1.05e-7)
                    if (term == 0) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) least[i >> 2][i & 3] = s[0][i >> 2][i & 3], s[0][i >> 2][i & 3] = 0.f;
                    }
                }
#pragma unroll
                for (int kt = 0; kt < MT; ++kt)
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt) {
                        const uint4 a = frag[((term * MT + kt) * MT + mt) * 32 + lane];
                        mma_bf16(s[mt][0], a, b[kt].x, b[kt].y);
                        mma_bf16(s[mt][1], a, b[kt].z, b[kt].w);
                    }
            }
            if constexpr (MT == 1) {
#pragma unroll
                for (int i = 0; i < 8; ++i) s[0][i >> 2][i & 3] += least[i >> 2][i & 3];
            }
            if (!finite(s[0][0][0]) || !finite(s[0][0][1]) || !finite(s[0][1][0]) || !finite(s[0][1][1])) {
                // an element of G that is not finite shows in every run at its position
#pragma unroll
                for (int i = 0; i < 8 * MT; ++i) {
                    const int r = 16 * (i >> 3) + g8 + 4 * (i & 2), j = j0 + 2 * (i & 4) + 2 * q + (i & 1);
                    float v = 0.f;
                    for (int k = 0; k < n1 && r < n1; ++k) v = fmaf(p.q1[k * n1 + r], bf16_at(Gb + k * M::kRow + j), v);
                    s[i >> 3][(i >> 2) & 1][i & 3] = v;
                }
            }
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const int r = 16 * mt + g8 + 8 * c;
                        if (r < n1) *reinterpret_cast<float2*>(W + r * Ge::kPitch + place(j0 + 8 * h + 2 * q)) = make_float2(s[mt][h][2 * c], s[mt][h][2 * c + 1]);
                    }
        }
        passes_up<L, 0>(X, p.tw, n1, u, r0);  // ends in a barrier
        // dL/dQ1 += G X'^T
#pragma unroll
        for (int i = 0; i < M::kTiles; ++i) {
            const int tile = first_tile + i * kWarps;
            if (tile >= tiles) continue;
            const int mt = tile % MT, run = min(8 * (tile / MT) + g8, n1 - 1);
            const uint32_t arow = gbase + 2u * ((16 * mt + (lane & 15)) * M::kRow + 8 * (lane >> 4));
            const float* xr = X + run * Ge::kPitch;
            // a token's own sums, the large terms in two chains and the small ones in a third, then one rounded addition each: an MMA
            // cuts its sum off where a multiply-add rounds it, which a chain over all tokens would collect
            float part[3][4];
#pragma unroll
            for (int c = 0; c < 12; ++c) part[c >> 2][c & 3] = 0.f;
#pragma unroll 4
            for (int j = 16 * slice, k = 0; j < Ge::kN2; j += 16 * slices, k ^= 1) {
                const uint4 a = matrices(arow + 2u * j);
                const float2 lo = *reinterpret_cast<const float2*>(xr + place(j + 2 * q)), hi = *reinterpret_cast<const float2*>(xr + place(j + 8 + 2 * q));
                uint32_t b0[3], b1[3];
                three_terms(lo.x, lo.y, b0), three_terms(hi.x, hi.y, b1);
                mma_bf16(part[2], a, b0[2], b1[2]);
                mma_bf16(part[2], a, b0[1], b1[1]);
                if (k == 0) mma_bf16(part[0], a, b0[0], b1[0]);
                else mma_bf16(part[1], a, b0[0], b1[0]);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float v = (part[0][c] + part[1][c]) + part[2][c];
                const int r = 16 * mt + g8 + 8 * (c >> 1), k = 8 * (tile / MT) + 2 * q + (c & 1);
                if (!finite(v) && r < n1 && k < n1) {
                    v = 0.f;
                    for (int j = 16 * slice; j < Ge::kN2; j += 16 * slices)
                        for (int e = j; e < j + 16; ++e) v = fmaf(bf16_at(Gb + r * M::kRow + e), X[k * Ge::kPitch + place(e)], v);
                }
                dq[i][c] += v;
            }
        }
        __syncthreads();
        passes_down<L, Ge::kPasses - 1>(X, W, p, row, u, r0, acc);
    }

    // ---- the CTA's sums, in the order of the run lanes and of the slices, to its slot ----
    float* const sm = reinterpret_cast<float*>(sm4);
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
    if (slices > 1) {  // one tile per warp
#pragma unroll
        for (int c = 0; c < 4; ++c) sm[4 * t + c] = dq[0][c];
        __syncthreads();
        if (slice == 0)
            for (int s = 1; s < slices; ++s)
#pragma unroll
                for (int c = 0; c < 4; ++c) dq[0][c] += sm[4 * (t + 32 * s * tiles) + c];
    }
    if (slice == 0) {
#pragma unroll
        for (int i = 0; i < M::kTiles; ++i) {
            const int tile = first_tile + i * kWarps;
            if (tile >= tiles) continue;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int r = 16 * (tile % MT) + g8 + 8 * (c >> 1), k = 8 * (tile / MT) + 2 * q + (c & 1);
                if (r < n1 && k < n1) out[Ge::kAngles + r * n1 + k] = dq[i][c];
            }
        }
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

// runs a kernel on as many CTAs as are resident (and have room for their sums), then adds the CTAs' sums; per_sm: CTAs per SM for
// each n1, found on the first call.  The limit of shared memory is that of every n1 (one per call would be pulled away by another
// thread's call).
static cudaError_t run(const bfq_plan* plan, void (*kern)(Params), size_t smem, int8_t& per_sm, int angles, const Params& p, float* dtheta, float* dq1,
                       cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    if (per_sm == 0) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kBackwardSmem);
        if (e != cudaSuccess) return e;
        int o = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, kThreads, smem);
        if (e != cudaSuccess) return e;
        per_sm = static_cast<int8_t>(o > 0 ? o : 1);
    }
    const int count = angles + p.n1 * p.n1;
    int64_t grid = int64_t(plan->sm_count) * per_sm;
    if (grid > p.rows) grid = p.rows;
    if (grid * count > int64_t(plan->partial_floats)) grid = int64_t(plan->partial_floats) / count;
    if (grid < 1) return cudaErrorInvalidValue;
    kern<<<int(grid), kThreads, smem, st>>>(p);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_reduce_composite<<<(count + 31) / 32, 1024, 0, st>>>(p.partial, int(grid), count, angles, dtheta, dq1);
    return cudaGetLastError();
}

template <int L, int BLOCKS>  // blocks of 16 runs
static cudaError_t launch(const bfq_plan* plan, const Params& p, float* dtheta, float* dq1, cudaStream_t st) {
    using G = Geo<L>;
    static int8_t per_sm[2][kMaxDevices][BFQ_MAX_N1 + 1] = {{{0}}};
    const size_t at_end = sizeof(float) * (G::kAngles > 4 * kThreads ? G::kAngles : 4 * kThreads);  // the sums
    if (p.gt == kBF16) {
        const size_t smem = Mma<L, BLOCKS>::smem(p.n1);
        if (smem <= kBackwardSmem)
            return run(plan, k_composite_backward_mma<L, BLOCKS>, smem > at_end ? smem : at_end, per_sm[1][plan->device][p.n1], G::kAngles, p, dtheta, dq1, st);
    }
    const int n1p = (p.n1 + 7) & ~7;
    const size_t smem = sizeof(float) * (size_t(3) * p.n1 * G::kPitch + size_t(p.n1) * n1p);
    return run(plan, k_composite_backward<L, BLOCKS>, smem > at_end ? smem : at_end, per_sm[0][plan->device][p.n1], G::kAngles, p, dtheta, dq1, st);
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
