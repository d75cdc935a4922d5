// What the kernels of the composite transform on whole tokens in shared memory share (rows of n2 = 2^7 .. 2^10 elements): the
// butterfly's passes of three stages, the loads, and the dense product across the runs.
#pragma once
#include <cuda_runtime.h>

#include "bfq_generic.cuh"
#include "bfq_ptx.cuh"

namespace bfq {
namespace cbw {
using namespace ptx;

constexpr int kThreads = 256;

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

template <int L>
struct Geo {
    static constexpr int kN2 = 1 << L, kPasses = (L + 2) / 3, kU = kN2 / 8, kRuns = kThreads / kU;  // runs side by side
    static constexpr int kPitch = kN2 + 4;
    static constexpr int kAngles = L * kN2 / 2;
};

template <int L, int P>
__device__ __forceinline__ void passes_up(float* X, const float2* __restrict__ tw, int n1, int u, int r0) {
    using G = Geo<L>;
    float2 cs[3][4];
    load_angles<L, P>(tw, u, cs);
    for (int r = r0; r < n1; r += 2 * G::kRuns) {
        const bool two = r + G::kRuns < n1;
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
    if constexpr (P + 1 < G::kPasses) passes_up<L, P + 1>(X, tw, n1, u, r0);
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

// to[k][j] = sum_i qs[i][k] from[i][j] (qs: [n1][n1p], zero from column n1 on), eight output runs x four positions per thread; returns
// the largest magnitude this thread wrote
template <int L>
__device__ __forceinline__ float across_runs(const float* qs, const float* from, float* to, int n1, int n1p) {
    using Ge = Geo<L>;
    float amax = 0.f;
    for (int item = threadIdx.x; item < (n1p / 8) * (Ge::kN2 / 4); item += kThreads) {
        const int j = place(4 * (item % (Ge::kN2 / 4))), k0 = 8 * (item / (Ge::kN2 / 4));
        u64 s[4][4];  // output runs k0 + 2a, k0 + 2a + 1 at position b
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) s[a][b] = 0ull;
#pragma unroll 4
        for (int i = 0; i < n1; ++i) {
            const float4 gv = *reinterpret_cast<const float4*>(from + i * Ge::kPitch + j);
            const ulonglong2 qa = *reinterpret_cast<const ulonglong2*>(qs + i * n1p + k0), qb = *reinterpret_cast<const ulonglong2*>(qs + i * n1p + k0 + 4);
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
            for (int b = 0; b < 4; ++b) unpack2(s[a][b], lo[b], hi[b]), amax = fmaxf(amax, fmaxf(fabsf(lo[b]), fabsf(hi[b])));
            if (k0 + 2 * a < n1) *reinterpret_cast<float4*>(to + (k0 + 2 * a) * Ge::kPitch + j) = make_float4(lo[0], lo[1], lo[2], lo[3]);
            if (k0 + 2 * a + 1 < n1) *reinterpret_cast<float4*>(to + (k0 + 2 * a + 1) * Ge::kPitch + j) = make_float4(hi[0], hi[1], hi[2], hi[3]);
        }
    }
    return amax;
}

}  // namespace cbw
}  // namespace bfq
