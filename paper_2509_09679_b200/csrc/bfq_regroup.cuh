// Pieces shared by the backward and inverse kernels on n = 4096 thread roles: the regroupings between the three phases in both
// directions, one row array at a time, and the element a role holds.
#pragma once
#include "bfq_n4096.cuh"
#include "bfq_row_again.cuh"

namespace bfq {
namespace b4k {
using namespace ptx;
using namespace f4k;

constexpr int kThreads = 128;  // a row group

__device__ __forceinline__ void sts128(uint32_t a, uint4 v) {
    asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

struct Addr {
    uint32_t w1, r1, w2, r2;  // per-thread byte offsets inside a regrouping buffer (forward write / read sides)
    uint32_t ex;              // base of the group's regrouping buffers
    int bar;                  // the group's named barrier
};

// ---- regroupings: forward direction (phase 1 -> 2 -> 3) and back, one row array at a time -------------
__device__ __forceinline__ void fwd1_store(const u64 (&P)[16], uint32_t buf, const Addr& a) {
#pragma unroll
    for (int m = 0; m < 16; ++m) sts64(buf + a.w1 + ex1_wr_local(m), P[m]);
}
__device__ __forceinline__ void fwd1_load(u64 (&P)[16], uint32_t buf, const Addr& a) {
#pragma unroll
    for (int m = 0; m < 16; ++m) P[m] = lds64(buf + a.r1 + ex1_rd_local(m));
}
__device__ __forceinline__ void fwd2_store(const u64 (&P)[16], uint32_t buf, const Addr& a) {
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        uint32_t lo, hi;
        unpack2u(P[m], lo, hi);
        sts32(buf + a.w2 + ex2_wr_local(m, 0), lo);
        sts32(buf + a.w2 + ex2_wr_local(m, 1), hi);
    }
}
__device__ __forceinline__ void fwd2_load(u64 (&P)[16], uint32_t buf, const Addr& a) {
#pragma unroll
    for (int m = 0; m < 16; ++m) P[m] = lds64(buf + a.r2 + ex2_rd_local(m));
}
// back from phase 3 to phase 2: the phase-3 owner stores whole packed registers where it read them,
// the phase-2 owner reads scalars where it wrote them
__device__ __forceinline__ void rev2_store(const u64 (&P)[16], uint32_t buf, const Addr& a) {
#pragma unroll
    for (int m = 0; m < 16; ++m) sts64(buf + a.r2 + ex2_rd_local(m), P[m]);
}
__device__ __forceinline__ void rev2_load(u64 (&P)[16], uint32_t buf, const Addr& a) {
#pragma unroll
    for (int m = 0; m < 16; ++m)
        P[m] = pack2u(lds32(buf + a.w2 + ex2_wr_local(m, 0)), lds32(buf + a.w2 + ex2_wr_local(m, 1)));
}
__device__ __forceinline__ void rev1_store(const u64 (&P)[16], uint32_t buf, const Addr& a) {
#pragma unroll
    for (int m = 0; m < 16; ++m) sts64(buf + a.r1 + ex1_rd_local(m), P[m]);
}
__device__ __forceinline__ void rev1_load(u64 (&P)[16], uint32_t buf, const Addr& a) {
#pragma unroll
    for (int m = 0; m < 16; ++m) P[m] = lds64(buf + a.w1 + ex1_wr_local(m));
}

__device__ __forceinline__ uint32_t cvt_bf16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// element index of (phase P, role t, packed register m, half h)
__device__ __forceinline__ int elem_of(int P, int t, int m, int h) {
    if (P == 0) return m | ((t & 15) << 4) | (h << 8) | ((t >> 4) << 9);
    if (P == 1) return (t & 15) | (m << 4) | (h << 8) | ((t >> 4) << 9);
    return h | (t << 1) | (m << 8);
}

// rows shorter than 4096 (SHORT): 2^log rows of n = 4096 >> log elements go through the kernel as one row of 4096 whose last
// stages are the identity (they are passed over, so that no row touches another one's infinities); `rows` counts those, the
// last one may be short (`elems` elements in all, missing ones arrive as zeros).  x, g and dx contiguous.
struct ShortRows {
    int log;
    int64_t elems;
    RowSource from;  // inverse: for rows that are done again
    int64_t ldx;     // inverse: row stride of x
};

}  // namespace b4k
}  // namespace bfq
