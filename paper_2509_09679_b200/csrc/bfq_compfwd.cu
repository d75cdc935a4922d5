// Composite transform Y = Q1 (X Q2^T) of whole tokens, codes or rows out, for n2 = 128 .. 1024 and every n1, in fp32: the shapes
// and types that the tensor-core kernels of 40 x 128 do not take (fp32 rows, INT2, other factors).
//
// A CTA keeps a token in shared memory; the butterfly runs in passes of three stages in registers (two runs packed into one
// instruction), the dense factor with eight output runs x four positions per thread (packed), then one maximum and the codes.
// The kernel for every shape does one stage per barrier, element by element: 32768 tokens of 40 x 128 at INT2 took
// 2.07 ms there and take 0.93 ms here (40000 of 12 x 256: 1.43 -> 0.62 ms, 18000 of 7 x 1024: 1.70 -> 0.47 ms; one token 11.4 us,
// most of it the call).
#include "../../include/bfq.h"

#include <cuda_runtime.h>

#include "bfq_comp_walk.cuh"
#include "bfq_fast.h"
#include "bfq_generic.cuh"

namespace bfq {
namespace cbw {

constexpr int kForwardSmem = 226 * 1024;  // dynamic shared memory of a CTA at most

struct ForwardParams {
    const float2* tw;
    const float* q1;
    int n1;
    const void* x;
    int xt;
    int64_t ldx;
    void* y;  // rows out, or null
    int yt;
    int64_t ldy;
    uint8_t* codes;  // codes out, or null
    uint16_t* scales;
    int bits;
    int64_t rows;
};

template <int L>
__global__ void __launch_bounds__(kThreads, 3) k_composite_forward(const ForwardParams p) {
    using Ge = Geo<L>;
    extern __shared__ __align__(16) float sm[];
    __shared__ uint32_t red[kThreads / 32];
    const int n1 = p.n1, n1p = (n1 + 7) & ~7, t = threadIdx.x;
    float* X = sm;
    float* Y = X + n1 * Ge::kPitch;
    float* q1t = Y + n1 * Ge::kPitch;  // [k][i] = Q1[i][k], columns from n1 on zero
    for (int e = t; e < n1 * n1p; e += kThreads) {
        const int k = e / n1p, i = e % n1p;
        q1t[e] = i < n1 ? p.q1[i * n1 + k] : 0.f;
    }
    const int u = t % Ge::kU, r0 = t / Ge::kU;
    const int64_t code_row = static_cast<int64_t>(n1) * Ge::kN2 * p.bits / 8;
    for (int64_t row = blockIdx.x; row < p.rows; row += gridDim.x) {
        __syncthreads();  // the buffers' readers of the token before are done
        load_token<L>(p.x, p.xt, row, p.ldx, n1, X);
        __syncthreads();
        passes_up<L, 0>(X, p.tw, n1, u, r0);
        const float amax = across_runs<L>(q1t, X, Y, n1, n1p);
        float inv = 0.f;
        if (p.codes != nullptr) {
            // magnitudes order like their bit patterns (a NaN has been dropped by fmaxf)
            const uint32_t wmax = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(amax));
            if ((t & 31) == 0) red[t >> 5] = wmax;
        }
        __syncthreads();
        if (p.codes != nullptr) {
            uint32_t m = red[0];
#pragma unroll
            for (int w = 1; w < kThreads / 32; ++w) m = max(m, red[w]);
            const uint16_t s = row_scale(__uint_as_float(m), (1 << (p.bits - 1)) - 1, &inv);
            if (t == 0) p.scales[row] = s;
        }
        for (int c = t; c < n1 * (Ge::kN2 / 16); c += kThreads) {
            const int r = c / (Ge::kN2 / 16), i = 16 * (c % (Ge::kN2 / 16));
            float v[16];
#pragma unroll
            for (int e = 0; e < 16; e += 4) {
                const float4 f = *reinterpret_cast<const float4*>(Y + r * Ge::kPitch + place(i + e));
                v[e] = f.x, v[e + 1] = f.y, v[e + 2] = f.z, v[e + 3] = f.w;
            }
            if (p.codes != nullptr) store_codes16(p.codes + row * code_row + int64_t(16) * c * p.bits / 8, p.bits, v, inv);
            if (p.y != nullptr) store16(p.y, p.yt, row * p.ldy + 16 * c, v);
        }
    }
}

template <int L>
static cudaError_t launch_forward(const bfq_plan* plan, const ForwardParams& p, cudaStream_t st) {
    const size_t smem = (size_t(2) * p.n1 * Geo<L>::kPitch + size_t(p.n1) * ((p.n1 + 7) & ~7)) * sizeof(float);
    auto kern = k_composite_forward<L>;
    // the limit of every n1, set once (a limit per call would be pulled away by another thread's call with a smaller n1); CTAs
    // per SM for each n1
    static int8_t per_sm[kMaxDevices][BFQ_MAX_N1 + 1] = {{0}};
    int8_t& occ = per_sm[plan->device][p.n1];
    if (occ == 0) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kForwardSmem);
        if (e != cudaSuccess) return e;
        int o = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, kThreads, smem);
        if (e != cudaSuccess) return e;
        occ = static_cast<int8_t>(o > 0 ? o : 1);
    }
    const int64_t cap = int64_t(plan->sm_count) * occ;
    kern<<<int(p.rows < cap ? p.rows : cap), kThreads, smem, st>>>(p);
    return cudaGetLastError();
}

}  // namespace cbw

bool composite_forward_available(const bfq_plan* plan, int n1) {
    const size_t n1p = (n1 + 7) & ~7;
    return plan->n >= 128 && plan->n <= 1024 && (size_t(2) * n1 * (plan->n + 4) + size_t(n1) * n1p) * sizeof(float) <= cbw::kForwardSmem;
}

cudaError_t composite_forward_launch(const bfq_plan* plan, const float* q1, int n1, const void* x, int xt, int64_t rows, int64_t ldx, void* y, int yt,
                                     int64_t ldy, int bits, uint8_t* codes, uint16_t* scales, cudaStream_t st) {
    cbw::ForwardParams p{};
    p.tw = plan->tw, p.q1 = q1, p.n1 = n1, p.x = x, p.xt = xt, p.ldx = ldx, p.y = y, p.yt = yt, p.ldy = ldy;
    p.codes = codes, p.scales = scales, p.bits = bits, p.rows = rows;
    switch (plan->log_n) {
        case 7: return cbw::launch_forward<7>(plan, p, st);
        case 8: return cbw::launch_forward<8>(plan, p, st);
        case 9: return cbw::launch_forward<9>(plan, p, st);
        case 10: return cbw::launch_forward<10>(plan, p, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace bfq
