// Forward of a few rows of 4096 elements (decoded tokens): bf16 or fp32 rows -> codes and scales, or rows of the same type.
//
// The kernel for many rows (bfq_fwdq4096.cuh) brings all 213 KB of constants into the tensor memory of each SM it runs on, which
// a batch pays for once; for one row that fetch, by one SM, is most of the time.  Here a row is spread over a cluster of eight CTAs
// of 64 threads, each with an eighth of the constants in its registers: stages 0 .. 8 stay inside a CTA's 512 elements
// (three passes of three stages, a thread holds eight elements), then every thread sends each of its eight values to another
// CTA, and stages 9 .. 11 pair what has arrived.  All loads are issued at the start.  The arithmetic is that of the other
// kernel, stage by stage, so a row's results are the same bits in any batch.
// What bounds it: latency (a launch, one round trip to L2, one exchange, and for codes another one for the row's maximum).
#include "bfq_fast.h"
#include "bfq_generic.cuh"
#include "bfq_n4096.cuh"

namespace bfq {
namespace few {
using namespace ptx;
using namespace f4k;

constexpr int kRanks = 8, kThreads = 64, kBlock = kN / kRanks;  // elements of a CTA

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// where element i of a CTA's block lies between passes
__device__ __forceinline__ int place(int i) { return i + (i >> 3); }
// element e (three bits) of thread u in pass P: bits 3 P .. 3 P + 2 of its index are e
template <int P>
__device__ __forceinline__ int index_of(int u, int e) {
    return P == 0 ? (e | (u << 3)) : (P == 1 ? ((u & 7) | (e << 3) | ((u >> 3) << 6)) : (u | (e << 6)));
}
template <int K>
__device__ __forceinline__ constexpr int lo_of(int q) { return ((q >> K) << (K + 1)) | (q & ((1 << K) - 1)); }
__device__ __forceinline__ int angle_of(int lo, int s) { return s * (kN / 2) + (((lo >> (s + 1)) << s) | (lo & ((1 << s) - 1))); }

template <int P, int K = 0>
__device__ __forceinline__ void load_pass(const float2* flat, int rank, int u, float2 (&c)[3][4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) c[K][q] = load_plain(flat + angle_of((rank << 9) | index_of<P>(u, lo_of<K>(q)), 3 * P + K));
    if constexpr (K < 2) load_pass<P, K + 1>(flat, rank, u, c);
}
template <int K>
__device__ __forceinline__ void stage(float (&v)[8], const float2 (&c)[4], bool shear) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int lo = lo_of<K>(q), hi = lo | (1 << K);
        const float a = v[lo], b = v[hi];
        if (!shear) {
            v[lo] = __fmaf_rn(c[q].x, b, a), v[hi] = __fmaf_rn(c[q].y, a, b);
        } else {
            const float a1 = __fmaf_rn(c[q].x, b, a), b1 = __fmaf_rn(c[q].y, a1, b);
            v[lo] = __fmaf_rn(c[q].x, b1, a1), v[hi] = b1;
        }
    }
}
__device__ __forceinline__ void pass(float (&v)[8], const float2 (&c)[3][4], bool shear) {
    stage<0>(v, c[0], shear), stage<1>(v, c[1], shear), stage<2>(v, c[2], shear);
}

// BITS = 0: rows out, else codes and scales
template <bool F32, int BITS>
__global__ void __launch_bounds__(kThreads) k_forward_few(const void* x, int64_t ldx, const float* tables, const int* form,
                                                          uint8_t* __restrict__ codes, uint16_t* __restrict__ scales, void* __restrict__ y, int64_t ldy) {
    __shared__ float buf[kBlock + kBlock / 8];
    __shared__ float arrived[kBlock];       // [rank][64]
    __shared__ uint32_t peak[2 * kRanks];   // [rank][warp]
    const int u = threadIdx.x, warp = u >> 5, lane = u & 31;
    const int rank = static_cast<int>(cluster_ctarank());
    const int64_t row = blockIdx.x / kRanks;
    cluster_arrive();  // the peers have started when this is over: waited for before the first store to one
    grid_dep_launch();
    grid_dep_wait();
    const bool shear = *form != 0;
    // eight elements of the row, and the constants, by loads that stay where they are written: all of them are on their way before the
    // first is waited for.  (k1, k2) of stages 0 .. 10, then the four numbers of the last one
    float v[8];
    if constexpr (F32) {
        const float4* src = reinterpret_cast<const float4*>(static_cast<const float*>(x) + row * ldx + rank * kBlock + 8 * u);
        const float4 a = load_plain(src), b = load_plain(src + 1);
        v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
    } else {
        const uint4 w = *reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(x) + row * ldx + rank * kBlock + 8 * u);
        const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) v[2 * i] = __uint_as_float(ws[i] << 16), v[2 * i + 1] = __uint_as_float(ws[i] & 0xFFFF0000u);
    }
    const float* base = tables + (shear ? kFlatFloats : 0);
    const float2* flat = reinterpret_cast<const float2*>(base);
    const float4* last = reinterpret_cast<const float4*>(base + 11 * kN);
    float2 c0[3][4], c1[3][4], c2[3][4], c9[4], c10[4];
    float4 c11[4];
    load_pass<0>(flat, rank, u, c0);
    load_pass<1>(flat, rank, u, c1);
    load_pass<2>(flat, rank, u, c2);
    const int j = (rank << 6) | u;  // this thread's position in every block after the exchange
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        c9[q] = load_plain(flat + angle_of((lo_of<0>(q) << 9) | j, 9));
        c10[q] = load_plain(flat + angle_of((lo_of<1>(q) << 9) | j, 10));
        c11[q] = load_plain(last + ((q << 9) | j));
    }
    // the rotations start after all loads have been issued
    asm volatile("" : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7])::"memory");
    pass(v, c0, shear);
#pragma unroll
    for (int e = 0; e < 8; ++e) buf[place(index_of<0>(u, e))] = v[e];
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = buf[place(index_of<1>(u, e))];
    pass(v, c1, shear);
#pragma unroll
    for (int e = 0; e < 8; ++e) buf[place(index_of<1>(u, e))] = v[e];  // where this thread read them
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = buf[place(index_of<2>(u, e))];
    pass(v, c2, shear);
    cluster_wait();
    const uint32_t to = smem_u32(arrived) + 4u * static_cast<uint32_t>(rank * kThreads + u);
#pragma unroll
    for (int e = 0; e < 8; ++e) st_cluster_b32(map_to_cta(to, static_cast<uint32_t>(e)), __float_as_uint(v[e]));
    cluster_arrive();
    cluster_wait();
#pragma unroll
    for (int b = 0; b < 8; ++b) v[b] = arrived[b * kThreads + u];
    stage<0>(v, c9, shear);
    stage<1>(v, c10, shear);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float a = v[q], b = v[q + 4];
        v[q] = __fmaf_rn(c11[q].y, b, __fmul_rn(c11[q].x, a));
        v[q + 4] = __fmaf_rn(c11[q].w, b, __fmul_rn(c11[q].z, a));
    }
    // v[b]: element 512 b + j of the result
    if constexpr (BITS == 0) {
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const int64_t at = row * ldy + kBlock * b + j;
            if constexpr (F32) static_cast<float*>(y)[at] = v[b];
            else static_cast<__nv_bfloat16*>(y)[at] = __float2bfloat16_rn(v[b]);
        }
    } else {
        constexpr int kQmax = BITS == 2 ? 1 : (BITS == 8 ? 127 : 7);
        float amax = 0.f;
#pragma unroll
        for (int b = 0; b < 8; ++b) amax = fmaxf(amax, fabsf(v[b]));
        const uint32_t wmax = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(amax));
        if (lane < kRanks) st_cluster_b32(map_to_cta(smem_u32(peak) + 4u * static_cast<uint32_t>(2 * rank + warp), static_cast<uint32_t>(lane)), wmax);
        cluster_arrive();
        cluster_wait();
        amax = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, peak[lane & (2 * kRanks - 1)]));
        float inv;
        const uint16_t s16 = row_scale_fast<kQmax>(amax, &inv);
        if (rank == 0 && u == 0) scales[row] = s16;
        const bool plain = (((s16 >> 10) & 31u) != 0u) && (s16 != 0x7BFFu);  // as in the kernel for many rows
        constexpr int kPer = 8 / BITS;  // codes of a byte, in consecutive lanes
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const float r = plain ? __fmaf_rn(v[b], inv, 12582912.f) - 12582912.f : rintf(__fmul_rn(v[b], inv));
            const int code = static_cast<int>(fminf(fmaxf(r, static_cast<float>(-kQmax - 1)), static_cast<float>(kQmax)));
            uint32_t byte = (static_cast<uint32_t>(code) & ((1u << BITS) - 1u)) << (BITS * (lane & (kPer - 1)));
#pragma unroll
            for (int o = 1; o < kPer; o *= 2) byte |= __shfl_xor_sync(0xFFFFFFFFu, byte, o);
            if ((lane & (kPer - 1)) == 0) codes[row * (kN * BITS / 8) + (kBlock * b + j) / kPer] = static_cast<uint8_t>(byte);
        }
    }
}

}  // namespace few

// Up to this many rows; see k_forward_few
bool forward_few_available(const bfq_plan* plan, int64_t rows) {
    return rows <= f4k::kFewRows && plan->n == f4k::kN && plan->cc_major == 10 && plan->flat4096 != nullptr && !plan->test_stuck_wait;
}

cudaError_t forward_few_launch(const bfq_plan* plan, const void* x, bool f32, int64_t rows, int64_t ldx, int bits, uint8_t* codes, uint16_t* scales, void* y,
                               int64_t ldy, cudaStream_t st) {
    auto go = [&](auto kern) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(unsigned(few::kRanks * rows)), cfg.blockDim = dim3(few::kThreads), cfg.stream = st;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = few::kRanks, attr[0].val.clusterDim.y = 1, attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr, cfg.numAttrs = 2;
        return cudaLaunchKernelEx(&cfg, kern, x, ldx, static_cast<const float*>(plan->flat4096), static_cast<const int*>(plan->form_flag), codes, scales, y, ldy);
    };
    if (f32) {
        return bits == 0 ? go(few::k_forward_few<true, 0>) : bits == 2 ? go(few::k_forward_few<true, 2>)
             : bits == 4 ? go(few::k_forward_few<true, 4>) : go(few::k_forward_few<true, 8>);
    }
    return bits == 0 ? go(few::k_forward_few<false, 0>) : bits == 2 ? go(few::k_forward_few<false, 2>)
         : bits == 4 ? go(few::k_forward_few<false, 4>) : go(few::k_forward_few<false, 8>);
}

}  // namespace bfq
