// Backward pass for rows of 128 .. 4096 elements on sm_100a:  dx = Q^T g  and  d-theta summed over rows.
//
// The gradient comes down first and the row goes up with it: u = Q^T g, then x and u together through the stages, taking
// d[s][pair] += u_hi * x_lo - u_lo * x_hi on the inputs of every stage (a rotation keeps the cross product of two vectors, so
// the inputs serve as well as the outputs).  Neither y nor the last stage of the way up is needed.
//
// One table serves both ways.  The forward kernel keeps true value = d * stored value and rotates by lo' = lo + k1 * hi,
// hi' = hi + k2 * lo, the factors d being folded into its last stage.  A gradient kept the other way round, stored value =
// d * true value, comes down through the transposed stages, lo = lo' + k2 * hi', hi = hi' + k1 * lo': the same constants, with lo
// and hi changing places; so do the three-shear stages.  At the bottom d is 1: u is dx as it stands, and x and u go up with the
// same factors, so that a pair's sum comes out times 1 / (d_lo * d_hi), one number per angle (`weight`), put right when the
// CTAs' sums are added.  560 packed multiply-adds of the rotations and 384 multiplications and additions of the sums per row and thread;
// recomputing y and walking y and g down in the three-shear form (the only one in which one table served that) took 1056 in all.
//
// A CTA per SM runs four groups of 128 threads as a pipeline, a row in each:
//     D  g: stages 11 .. 8 down
//     A  g: stages 7 .. 0 down, dx (or B: kDxByA)
//     B  x and u: stages 0 .. 3 up
//     C  x and u: stages 4 .. 7 up
//     D  x and u: stages 8 .. 10 up, and the sums of 8 .. 11
// so that every scheduler has a warp of each group to take turns with, whatever the others wait for, and a row changes hands
// exactly where it has to be regrouped.  B's and C's sums are in the tensor-memory columns that the constants leave free, D's
// in registers (the groups' register shares differ); half of the last stage's constants are in shared memory instead.
//
// Range: factors of 2^-40 and more (else the three-shear form runs: `form`), and g comes down 2^40 times too large, so that nothing
// is stored smaller than it is: however small g, no bits are lost.  What overflows instead (with the least factors g from about 2^80 on,
// products of u and x from 2^48 on) leaves a sum that is not finite; the CTA then does its rows again in the three-shear form, which
// has no factors, and rewrites only those pieces of dx that were not finite.  The second pass takes 1.7 times as long as the first: 262144
// x 4096 bf16 rows 9.1 ms in all as soon as one CTA meets one, 3.4 otherwise.  An infinity or NaN in g or x is such a row too (and leaves
// no angle's sum finite where it is in g).  A look at g and dx between the passes that leaves the second one out for those cost every
// call 8 %, in registers of the row loops.
#include <type_traits>

#include "bfq_fast.h"
#include "bfq_generic.cuh"
#include "bfq_n4096.cuh"
#include "bfq_regroup.cuh"

namespace bfq {
namespace g4k {
using namespace ptx;
using namespace f4k;
using namespace b4k;

constexpr int kGroups = 4, kCta = kGroups * kThreads;
constexpr int kSlots = 2;                   // rows of x and of g on their way
constexpr int kAccCol = 384;                // sums of stages 0 .. 7: 16 columns each
constexpr int kLastCol = 352;               // constants of the last stage: half of them in tensor memory, the rest in shared memory
constexpr int kSlotFloats = 12 * (kN / 2);  // a CTA's sums
constexpr float kLift = 1099511627776.f;    // 2^40, the inverse of the least factor
// Group A or group B scales u back and writes dx: whichever has the time.  us, written by A / by B: 65536 rows of 4096 bf16 846 / 879,
// fp32 1016 / 932; 2^25 elements of n = 2048 bf16 125 / 116, fp32 152 / 138, n = 1024 119 / 115, 152 / 136, n = 256 117 / 119, 144 / 142,
// n = 128 130 / 137, 166 / 156.
template <bool IN_F32, int STAGES>
constexpr bool kDxByA = !IN_F32 && (STAGES == 12 || STAGES <= 8);
constexpr int kLag = 3;                     // rows between a row's two turns in group D
enum : int { kFullDA = 1, kEmptyDA, kFullAB, kEmptyAB, kFullBC, kEmptyBC, kFullCD, kEmptyCD };

template <bool IN_F32>
struct Smem {
    static constexpr uint32_t kRow = (IN_F32 ? 2 : 1) * kRowBytes;
    static constexpr uint32_t kXOff = 0;                             // [kSlots] rows
    static constexpr uint32_t kGOff = kXOff + kSlots * kRow;         // [kSlots] rows
    // g between phases 3 and 2, index bits i0 .. i11: word (i8 ^ i4) + 2 (i0 ^ i5) + 4 (i1 .. i3) + 32 (i4 .. i7) + 512 (i9 .. i11),
    // so that D's scalar stores (lanes i1 .. i5) and A's 64-bit loads (lanes i0 .. i3) fall into different banks
    static constexpr uint32_t kDAOff = kGOff + kSlots * kRow;
    static constexpr uint32_t kAOff = kDAOff + 4 * kN;               // g between phases 2 and 1
    static constexpr uint32_t kABOff = kAOff + kExBytes;             // u, [8][128] of four numbers
    static constexpr uint32_t kBCOff = kABOff + 4 * kN;              // x, u
    static constexpr uint32_t kCDOff = kBCOff + 2 * kExBytes;        // x, u
    static constexpr uint32_t kLastOff = kCDOff + 2 * kExBytes;      // [8][128] float4: last stage, pairs 4 .. 7
    static constexpr uint32_t kBarOff = kLastOff + 8 * kThreads * 16;  // mbarriers: x [kSlots], g [kSlots]
    static constexpr uint32_t kTmemOff = kBarOff + 16 * kSlots;
    static constexpr uint32_t kBadOff = kTmemOff + 8;  // a sum is not finite
    static constexpr uint32_t kBytes = kBadOff + 8 + 1024;
};
static_assert(Smem<true>::kBytes <= 232448, "shared memory budget of one CTA");

template <int N>
__device__ __forceinline__ void regs_down() {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void regs_up() {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}

// pairs U0 .. U0 + 3 of local stage K, up or (transposed) down
template <int FORM, int K, int U0>
__device__ __forceinline__ void stage_up(u64 (&P)[16], const uint32_t (&T)[16]) {
    if constexpr (FORM == kFormScaled) stage_scaled<K, U0, 4, 16>(P, T);
    else stage_lift<K, U0, 4, 16>(P, T);
}
template <int K>
__device__ __forceinline__ constexpr int pair_lo(int u) { return ((u >> K) << (K + 1)) | (u & ((1 << K) - 1)); }
template <int FORM, int K, int U0>
__device__ __forceinline__ void stage_down(u64 (&P)[16], const uint32_t (&T)[16]) {
    if constexpr (FORM == kFormScaled) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int lo = pair_lo<K>(U0 + i), hi = lo | (1 << K);
            const u64 a = P[lo], b = P[hi];
            P[lo] = fma2(pack2u(T[4 * i + 2], T[4 * i + 3]), b, a);
            P[hi] = fma2(pack2u(T[4 * i], T[4 * i + 1]), a, b);
        }
    } else {
#pragma unroll
        for (int shear = 0; shear < 3; ++shear)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int lo = pair_lo<K>(U0 + i), hi = lo | (1 << K);
                if (shear == 1) P[lo] = fma2(pack2u(T[4 * i + 2], T[4 * i + 3]), P[hi], P[lo]);
                else P[hi] = fma2(pack2u(T[4 * i], T[4 * i + 1]), P[lo], P[hi]);
            }
    }
}
// the last stage, transposed, on pairs (u, u + 8), u = U0 and U0 + 1; DIAGONAL (short rows): it couples nothing
template <int U0, bool DIAGONAL>
__device__ __forceinline__ void last_down(u64 (&P)[16], const uint32_t (&T)[16]) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int lo = U0 + i, hi = lo + 8;
        const u64 k1 = pack2u(T[8 * i], T[8 * i + 1]), k2 = pack2u(T[8 * i + 2], T[8 * i + 3]);
        const u64 k3 = pack2u(T[8 * i + 4], T[8 * i + 5]), k4 = pack2u(T[8 * i + 6], T[8 * i + 7]);
        const u64 a = P[lo], b = P[hi];
        if constexpr (DIAGONAL) {
            P[lo] = mul2(k1, a), P[hi] = mul2(k4, b);
        } else {
            P[lo] = fma2(k3, b, mul2(k1, a));
            P[hi] = fma2(k4, b, mul2(k2, a));
        }
    }
}
// A[i] += u_hi * x_lo - u_lo * x_hi for pairs U0 .. U0 + 3.  The difference first, so that a row is one rounding of the running sum: with
// one product after the other taken into the sum (an instruction less) d-theta of 262144 rows was 1.09e-6 from 64 bits, now 7.5e-7
// (3290 -> 3374 us).
template <int K, int U0>
__device__ __forceinline__ void cross(u64 (&A)[4], const u64 (&X)[16], const u64 (&U)[16]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int lo = pair_lo<K>(U0 + i), hi = lo | (1 << K);
        A[i] = add2(A[i], sub2(mul2(U[hi], X[lo]), mul2(U[lo], X[hi])));
    }
}

// g down through half-stages I .. END - 1, counted from stage 10: half-stage I is half I & 1 of stage 10 - I / 2.  Its
// constants are in Tcur; the next ones are requested right after the wait.  hook(integral_constant<I>) runs after each.
template <int FORM, int I, int END, int STAGES, class F>
__device__ __forceinline__ void walk_down(u64 (&G)[16], uint32_t (&Tcur)[16], uint32_t (&Tnext)[16], uint32_t tlane, F&& hook) {
    constexpr int s = 10 - I / 2, c = I & 1;
    if constexpr (s < STAGES) {
        tmem_wait_ld16(Tcur);
        if constexpr (I + 1 < END) tmem_ld16(tlane + 32 * (10 - (I + 1) / 2) + 16 * ((I + 1) & 1), Tnext);
        stage_down<FORM, s & 3, 4 * c>(G, Tcur);
    }
    hook(std::integral_constant<int, I>());
    if constexpr (I + 1 < END) {
        if constexpr (s < STAGES) walk_down<FORM, I + 1, END, STAGES>(G, Tnext, Tcur, tlane, hook);
        else walk_down<FORM, I + 1, END, STAGES>(G, Tcur, Tnext, tlane, hook);
    }
}
// where the constants of its first half-stage from I on that exists are
template <int I, int STAGES>
__device__ __forceinline__ constexpr int first_col() {
    constexpr int s = 10 - I / 2;
    return s < STAGES ? 32 * s + 16 * (I & 1) : 32 * (STAGES - 1);
}

// x and u up through half-stages C .. END - 1 (half C & 1 of stage C / 2), sums in tensor memory
template <int FORM, int C, int END, int STAGES>
__device__ __forceinline__ void walk_up(u64 (&X)[16], u64 (&U)[16], uint32_t (&Tcur)[16], uint32_t (&Tnext)[16], uint32_t (&Acur)[8],
                                        uint32_t (&Anext)[8], uint32_t tlane) {
    constexpr int s = C / 2, U0 = 4 * (C & 1);
    constexpr bool kMore = C + 1 < END && (C + 1) / 2 < STAGES;
    if constexpr (s >= STAGES) return;
    tmem_wait_ld16_8(Tcur, Acur);
    if constexpr (kMore) {
        tmem_ld16(tlane + 16 * (C + 1), Tnext);
        tmem_ld8(tlane + kAccCol + 8 * (C + 1), Anext);
    }
    u64 A[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) A[i] = pack2u(Acur[2 * i], Acur[2 * i + 1]);
    cross<s & 3, U0>(A, X, U);
#pragma unroll
    for (int i = 0; i < 4; ++i) unpack2u(A[i], Acur[2 * i], Acur[2 * i + 1]);
    tmem_st8(tlane + kAccCol + 8 * C, Acur);
    if constexpr (s + 1 < STAGES) {  // above the last stage nothing is asked for
        stage_up<FORM, s & 3, U0>(X, Tcur);
        stage_up<FORM, s & 3, U0>(U, Tcur);
    }
    if constexpr (kMore) walk_up<FORM, C + 1, END, STAGES>(X, U, Tnext, Tcur, Anext, Acur, tlane);
}
// the same for stages 8 .. 11, sums in registers
template <int FORM, int C, int STAGES>
__device__ __forceinline__ void walk_up_last(u64 (&X)[16], u64 (&U)[16], uint32_t (&Tcur)[16], uint32_t (&Tnext)[16], u64 (&A)[4][2][4], uint32_t tlane) {
    constexpr int s = C / 2, U0 = 4 * (C & 1);
    constexpr bool kRotates = s + 1 < STAGES;
    if constexpr (s >= STAGES) return;
    if constexpr (kRotates) {
        tmem_wait_ld16(Tcur);
        if constexpr ((C + 1) / 2 + 1 < STAGES) tmem_ld16(tlane + 16 * (C + 1), Tnext);
    }
    cross<s & 3, U0>(A[s - 8][C & 1], X, U);
    if constexpr (kRotates) {
        stage_up<FORM, s & 3, U0>(X, Tcur);
        stage_up<FORM, s & 3, U0>(U, Tcur);
    }
    if constexpr (C + 1 < 24) walk_up_last<FORM, C + 1, STAGES>(X, U, Tnext, Tcur, A, tlane);
}

__device__ __forceinline__ bool bad_bits(uint32_t w) { return (w & 0x7F800000u) == 0x7F800000u; }
__device__ __forceinline__ bool bad_bf16x2(uint32_t w) { return bad_bits(w) || (w & 0x7F80u) == 0x7F80u; }

// what a group works with
struct Ctx {
    Addr a;
    uint32_t sbase, tlane;
    int t, count, done;  // done: rows of earlier passes, for the parity of the barriers
    int first, stride;
    void* dx;
    int64_t ld, elems;
    int* status;
    float* out;   // the CTA's sums [12][2048]
    bool again;   // the rows' second pass
};

template <bool IN_F32, int STAGES>
__device__ __forceinline__ void request(const Ctx& cx, const CUtensorMap* map, uint32_t ring, uint32_t bars, int k) {
    const int slot = (cx.done + k) & 1, r = cx.first + k * cx.stride;
    mbar_expect_tx(bars + 8 * slot, Smem<IN_F32>::kRow);
    tma_load_3d(ring + slot * Smem<IN_F32>::kRow, map, 0, 0, r << (12 - STAGES), bars + 8 * slot);
}

// dx of a row, phase 1 ownership: two runs of 16 elements
template <bool IN_F32, int STAGES>
__device__ __forceinline__ void store_dx(const Ctx& cx, const u64 (&U)[16], int row) {
    const int t = cx.t;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int at = 16 * (t & 15) + 512 * (t >> 4) + 256 * h;
        if constexpr (STAGES < 12) {  // a run exists or not as a whole
            if (static_cast<int64_t>(row) * kN + at >= cx.elems) continue;
        }
        constexpr int kWords = IN_F32 ? 16 : 8;
        uint32_t w[kWords];
#pragma unroll
        for (int j = 0; j < kWords; ++j) {
            uint32_t lo0, hi0, lo1, hi1;
            if constexpr (IN_F32) {
                unpack2u(U[j], lo0, hi0);
                w[j] = h ? hi0 : lo0;
            } else {
                unpack2u(U[2 * j], lo0, hi0), unpack2u(U[2 * j + 1], lo1, hi1);
                w[j] = cvt_bf16x2(__uint_as_float(h ? hi0 : lo0), __uint_as_float(h ? hi1 : lo1));
            }
        }
        uint4* dst = reinterpret_cast<uint4*>(static_cast<uint8_t*>(cx.dx) + (static_cast<int64_t>(row) * cx.ld + at) * (IN_F32 ? 4 : 2));
        if (cx.again) {  // only what this thread could not write the first time
            bool bad = false;
#pragma unroll
            for (int c = 0; c < kWords / 4; ++c) {
                const uint4 v = dst[c];
                bad |= IN_F32 ? bad_bits(v.x) || bad_bits(v.y) || bad_bits(v.z) || bad_bits(v.w)
                              : bad_bf16x2(v.x) || bad_bf16x2(v.y) || bad_bf16x2(v.z) || bad_bf16x2(v.w);
            }
            if (!bad) continue;
        }
#pragma unroll
        for (int c = 0; c < kWords / 4; ++c) dst[c] = make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
    }
}

// u at its own size, and dx of the CTA's k-th row
template <int FORM, bool IN_F32, int STAGES>
__device__ __forceinline__ void write_dx(const Ctx& cx, u64 (&U)[16], int k) {
    if constexpr (FORM == kFormScaled) {
        const u64 back = pack2(1.f / kLift, 1.f / kLift);
#pragma unroll
        for (int m = 0; m < 16; ++m) U[m] = mul2(back, U[m]);
    }
    if (cx.dx == nullptr) return;
    const int use = cx.done + k;
    mbar_wait_bounded(cx.sbase + Smem<IN_F32>::kBarOff + 8 * (use & 1), (use >> 1) & 1, cx.status);  // x has arrived: dx may lie over it
    store_dx<IN_F32, STAGES>(cx, U, cx.first + k * cx.stride);
}

// A thread's sixteen sums of one stage to the CTA's slot, in the order of the angles: consecutive lanes fill whole sectors
template <int P>
__device__ __forceinline__ bool write_sums(const Ctx& cx, int s, const uint32_t (&a)[16]) {
    const int t = cx.t;
    float* out = cx.out + s * (kN / 2);
    bool bad = false;
#pragma unroll
    for (int e = 0; e < 16; ++e) bad |= bad_bits(a[e]);  // a[2u + h]: pair u, half h
    if constexpr (P == 0) {  // angle u + 8 (t & 15) + 128 h + 256 (t >> 4)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint4* dst = reinterpret_cast<uint4*>(out + 8 * (t & 15) + 128 * h + 256 * (t >> 4));
            dst[0] = make_uint4(a[h], a[2 + h], a[4 + h], a[6 + h]);
            dst[1] = make_uint4(a[8 + h], a[10 + h], a[12 + h], a[14 + h]);
        }
    } else if constexpr (P == 1) {  // (t & 15) + 16 u + 128 h + 256 (t >> 4)
#pragma unroll
        for (int e = 0; e < 16; ++e) out[(t & 15) + 16 * (e >> 1) + 128 * (e & 1) + 256 * (t >> 4)] = __uint_as_float(a[e]);
    } else {  // h + 2 t + 256 u
#pragma unroll
        for (int u = 0; u < 8; ++u) *reinterpret_cast<uint2*>(out + 2 * t + 256 * u) = make_uint2(a[2 * u], a[2 * u + 1]);
    }
    return bad;
}
template <int P, int STAGES>
__device__ __forceinline__ bool write_tmem_sums(const Ctx& cx) {
    bool bad = false;
    for (int s = 4 * P; s < 4 * P + 4 && s < STAGES; ++s) {
        uint32_t a[16];
        tmem_ld16(cx.tlane + kAccCol + 16 * s, a);
        tmem_wait_ld16(a);
        bad |= write_sums<P>(cx, s, a);
    }
    return bad;
}

template <int FORM, bool IN_F32, int STAGES>
__device__ __forceinline__ void group_a(const Ctx& cx, const CUtensorMap* xmap) {
    using S = Smem<IN_F32>;
    const int t = cx.t;
    const uint32_t xbars = cx.sbase + S::kBarOff, xring = cx.sbase + S::kXOff;
    const uint32_t from_d = cx.sbase + S::kDAOff + 16u * ((t >> 1) & 7) + 2048u * (t >> 4);
    const uint32_t from_d0 = from_d + 8u * (t & 1), from_d1 = from_d + 8u * ((t & 1) ^ 1), own = cx.sbase + S::kAOff, to_b = cx.sbase + S::kABOff + 16u * t;
    if (t == 0) {
        for (int k = 0; k < kSlots && k < cx.count; ++k) request<IN_F32, STAGES>(cx, xmap, xring, xbars, k);
    }
    u64 G[16];
    uint32_t T0[16], T1[16];
    for (int k = 0; k < cx.count; ++k) {
        tmem_ld16(cx.tlane + first_col<6, STAGES>(), T0);
        bar_sync(kFullDA, 2 * kThreads);
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            uint32_t lo, hi;
            unpack2u(lds64(((m >> 1) & 1 ? from_d1 : from_d0) + 128u * m), lo, hi);
            G[m] = (m & 1) ? pack2u(hi, lo) : pack2u(lo, hi);
        }
        if (k + 1 < cx.count) bar_arrive(kEmptyDA, 2 * kThreads);
        walk_down<FORM, 6, 22, STAGES>(G, T0, T1, cx.tlane, [&](auto step) {
            if constexpr (decltype(step)::value == 13) {  // below stage 4: phase 2 -> 1, inside each half-warp
                __syncwarp();
                rev1_store(G, own, cx.a);
                __syncwarp();
                rev1_load(G, own, cx.a);
            }
        });
        if constexpr (kDxByA<IN_F32, STAGES>) write_dx<FORM, IN_F32, STAGES>(cx, G, k);
        if (k > 0) {
            bar_sync(kEmptyAB, 2 * kThreads);  // B has read the row before, x too
            if (t == 0 && k + 1 < cx.count) request<IN_F32, STAGES>(cx, xmap, xring, xbars, k + 1);
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            uint32_t w[4];
            unpack2u(G[2 * c], w[0], w[1]), unpack2u(G[2 * c + 1], w[2], w[3]);
            sts128(to_b + c * kThreads * 16, make_uint4(w[0], w[1], w[2], w[3]));
        }
        __threadfence_block();
        bar_arrive(kFullAB, 2 * kThreads);
    }
}

template <int FORM, bool IN_F32, int STAGES>
__device__ __forceinline__ bool group_b(const Ctx& cx) {
    using S = Smem<IN_F32>;
    const int t = cx.t;
    const uint32_t xbars = cx.sbase + S::kBarOff, from_a = cx.sbase + S::kABOff + 16u * t, to_c = cx.sbase + S::kBCOff;
    // x tile: two runs of 16 elements, as in the forward kernel
    const uint32_t in_line = IN_F32 ? ((t & 15) >> 1) * 128u + (t >> 4) * 2048u : ((t >> 2) & 3) * 128u + (t >> 4) * 1024u;
    const uint32_t in_x = IN_F32 ? ((((t & 1) << 2) ^ ((t >> 1) & 7)) << 4) : ((((t & 3) << 1) ^ ((t >> 2) & 3)) << 4);
    u64 X[16], U[16];
    uint32_t T0[16], T1[16], A0[8], A1[8];
    for (int k = 0; k < cx.count; ++k) {
        const int use = cx.done + k, slot = use & 1;
        bar_sync(kFullAB, 2 * kThreads);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const uint4 w = lds128(from_a + c * kThreads * 16);
            U[2 * c] = pack2u(w.x, w.y), U[2 * c + 1] = pack2u(w.z, w.w);
        }
        tmem_ld16(cx.tlane, T0);
        tmem_ld8(cx.tlane + kAccCol, A0);
        if constexpr (!kDxByA<IN_F32, STAGES>) write_dx<FORM, IN_F32, STAGES>(cx, U, k);
        mbar_wait_bounded(xbars + 8 * slot, (use >> 1) & 1, cx.status);
        const uint32_t src = cx.sbase + S::kXOff + slot * S::kRow + in_line;
        if constexpr (IN_F32) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint4 w0 = lds128(src + (in_x ^ (c << 4))), w1 = lds128(src + 1024u + (in_x ^ (c << 4)));
                X[4 * c + 0] = pack2u(w0.x, w1.x), X[4 * c + 1] = pack2u(w0.y, w1.y);
                X[4 * c + 2] = pack2u(w0.z, w1.z), X[4 * c + 3] = pack2u(w0.w, w1.w);
            }
        } else {
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const uint4 w0 = lds128(src + (in_x ^ (c << 4))), w1 = lds128(src + 512u + (in_x ^ ((c | 4) << 4)));
                const uint32_t a[4] = {w0.x, w0.y, w0.z, w0.w}, b[4] = {w1.x, w1.y, w1.z, w1.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    X[8 * c + 2 * j + 0] = pack2u(bf16_lo(a[j]), bf16_lo(b[j]));
                    X[8 * c + 2 * j + 1] = pack2u(a[j] & 0xFFFF0000u, b[j] & 0xFFFF0000u);
                }
            }
        }
        if (k + 1 < cx.count) bar_arrive(kEmptyAB, 2 * kThreads);
        walk_up<FORM, 0, 8, STAGES>(X, U, T0, T1, A0, A1, cx.tlane);
        if (k > 0) bar_sync(kEmptyBC, 2 * kThreads);
        fwd1_store(X, to_c, cx.a);
        fwd1_store(U, to_c + kExBytes, cx.a);
        __threadfence_block();
        bar_arrive(kFullBC, 2 * kThreads);
        tmem_wait_st();
    }
    return write_tmem_sums<0, STAGES>(cx);
}

template <int FORM, bool IN_F32, int STAGES>
__device__ __forceinline__ bool group_c(const Ctx& cx) {
    using S = Smem<IN_F32>;
    const uint32_t from_b = cx.sbase + S::kBCOff, to_d = cx.sbase + S::kCDOff;
    constexpr bool kMore = STAGES > 8;  // D has something to do
    u64 X[16], U[16];
    uint32_t T0[16], T1[16], A0[8], A1[8];
    for (int k = 0; k < cx.count; ++k) {
        tmem_ld16(cx.tlane + 16 * 8, T0);
        tmem_ld8(cx.tlane + kAccCol + 8 * 8, A0);
        bar_sync(kFullBC, 2 * kThreads);
        fwd1_load(X, from_b, cx.a);
        fwd1_load(U, from_b + kExBytes, cx.a);
        if (k + 1 < cx.count) bar_arrive(kEmptyBC, 2 * kThreads);
        walk_up<FORM, 8, 16, STAGES>(X, U, T0, T1, A0, A1, cx.tlane);
        if constexpr (kMore) {
            if (k > 0) bar_sync(kEmptyCD, 2 * kThreads);
            fwd2_store(X, to_d, cx.a);
            fwd2_store(U, to_d + kExBytes, cx.a);
            __threadfence_block();
            bar_arrive(kFullCD, 2 * kThreads);
        }
        tmem_wait_st();
    }
    return write_tmem_sums<1, STAGES>(cx);
}

template <int FORM, bool IN_F32, int STAGES>
__device__ __forceinline__ bool group_d(const Ctx& cx, const CUtensorMap* gmap) {
    using S = Smem<IN_F32>;
    const int t = cx.t;
    const uint32_t gbars = cx.sbase + S::kBarOff + 8 * kSlots, gring = cx.sbase + S::kGOff;
    if (t == 0) {
        for (int k = 0; k < kSlots && k < cx.count; ++k) request<IN_F32, STAGES>(cx, gmap, gring, gbars, k);
    }
    // bf16: the word of elements 2t + 256m, +1 is word t & 3 of 16-byte chunk (t & 31) >> 2 of 128-byte line (t >> 5) + 4m; the
    // swizzle moves the chunk to chunk ^ (line & 7).  fp32: 8-byte word t & 1 of chunk (t & 15) >> 1 of line (t >> 4) + 8m
    const uint32_t g_x = ((t & 31) >> 2) ^ (t >> 5);
    const uint32_t g_a0 = (t >> 5) * 128u + (g_x << 4) + (t & 3) * 4u, g_a1 = (t >> 5) * 128u + ((g_x ^ 4u) << 4) + (t & 3) * 4u;
    const uint32_t f_a = (t >> 4) * 128u + ((((t & 15) >> 1) ^ (t >> 4)) << 4) + (t & 1) * 8u;
    const uint32_t last = cx.sbase + S::kLastOff + 16u * t, from_c = cx.sbase + S::kCDOff;
    const uint32_t i4 = (t >> 3) & 1, i5 = (t >> 4) & 1, to_a0 = cx.sbase + S::kDAOff + 16u * (t & 7) + 128u * (t >> 3) + 8u * i5;
    const uint32_t to_a[2] = {to_a0 + 4u * i4, to_a0 + 4u * (i4 ^ 1u)};
    constexpr bool kDiagonal = STAGES < 12, kUp = STAGES > 8;
    u64 X[16], U[16], A[4][2][4];
    uint32_t T0[16], T1[16];
#pragma unroll
    for (int i = 0; i < 32; ++i) A[i >> 3][(i >> 2) & 1][i & 3] = 0ull;
    for (int i = 0; i < cx.count + (kUp ? kLag : 0); ++i) {
        if (i < cx.count) {
            const int use = cx.done + i, slot = use & 1;
            tmem_ld16(cx.tlane + kLastCol, T0);
            mbar_wait_bounded(gbars + 8 * slot, (use >> 1) & 1, cx.status);
            const uint32_t src = gring + slot * S::kRow;
#pragma unroll
            for (int m = 0; m < 16; ++m) {
                if constexpr (IN_F32) {
                    U[m] = lds64(src + f_a + 1024u * m);
                } else {
                    const uint32_t w = lds32(src + ((m & 1) ? g_a1 : g_a0) + 512u * m);
                    U[m] = pack2u(bf16_lo(w), w & 0xFFFF0000u);
                }
            }
            tmem_wait_ld16(T0);
            tmem_ld16(cx.tlane + kLastCol + 16, T1);
            last_down<0, kDiagonal>(U, T0);
            tmem_wait_ld16(T1);
            if constexpr (STAGES > 8) tmem_ld16(cx.tlane + first_col<0, STAGES>(), T0);
            last_down<2, kDiagonal>(U, T1);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t K[16];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint4 v = lds128(last + (4 * h + j) * kThreads * 16);
                    K[4 * j] = v.x, K[4 * j + 1] = v.y, K[4 * j + 2] = v.z, K[4 * j + 3] = v.w;
                }
                if (h == 0) last_down<4, kDiagonal>(U, K);
                else last_down<6, kDiagonal>(U, K);
            }
            walk_down<FORM, 0, 6, STAGES>(U, T0, T1, cx.tlane, [](auto) {});
            if (i > 0) {
                bar_sync(kEmptyDA, 2 * kThreads);  // A has read the row before, and every warp here is past its reads of g
                if (t == 0 && i + 1 < cx.count) request<IN_F32, STAGES>(cx, gmap, gring, gbars, i + 1);
            }
#pragma unroll
            for (int m = 0; m < 16; ++m) {
                uint32_t lo, hi;
                unpack2u(U[m], lo, hi);
                sts32(to_a[m & 1] + 2048u * (m >> 1), lo);
                sts32((to_a[m & 1] ^ 8u) + 2048u * (m >> 1), hi);
            }
            __threadfence_block();
            bar_arrive(kFullDA, 2 * kThreads);
        }
        if (kUp && i >= kLag) {
            if constexpr (STAGES > 9) tmem_ld16(cx.tlane + 16 * 16, T0);
            bar_sync(kFullCD, 2 * kThreads);
            fwd2_load(X, from_c, cx.a);
            fwd2_load(U, from_c + kExBytes, cx.a);
            if (i + 1 < cx.count + kLag) bar_arrive(kEmptyCD, 2 * kThreads);
            walk_up_last<FORM, 16, STAGES>(X, U, T0, T1, A, cx.tlane);
        }
    }
    bool bad = false;
#pragma unroll
    for (int s = 8; s < STAGES; ++s) {
        uint32_t a[16];
#pragma unroll
        for (int u = 0; u < 8; ++u) unpack2u(A[s - 8][u >> 2][u & 3], a[2 * u], a[2 * u + 1]);
        bad |= write_sums<2>(cx, s, a);
    }
    return bad;
}

// IN_F32: x, g and dx are fp32.  STAGES = log2 of the row length: below 12, 4096 / n rows of n elements go through as one
// whose last stages are the identity; these are passed over, so that no row touches another one's infinities.  `rows` counts
// joint rows, of which the last one may be short (`elems` elements in all, missing ones arrive as zeros).  `slot_form`: the form each CTA's sums were taken in.  only_shear: no second
// pass is possible (dx lies over x or g).
template <bool IN_F32, int STAGES>
__global__ void __launch_bounds__(kCta, 1)
k_grad4096(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap gmap, const float* img, const int* form,
           void* __restrict__ dx, int64_t ld, float* __restrict__ partial, int* __restrict__ slot_form, int rows, int* __restrict__ status, bool only_shear,
           int64_t elems) {
    using S = Smem<IN_F32>;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const int warp = threadIdx.x >> 5, group = warp >> 2, t = threadIdx.x & (kThreads - 1);
    grid_dep_launch();
    if (warp == 0) tmem_alloc512(sbase + S::kTmemOff);
    if (threadIdx.x < 2 * kSlots) {
        mbar_init(sbase + S::kBarOff + 8 * threadIdx.x, 1);
        mbar_init_fence();
    }
    if (threadIdx.x == 0) sts32(sbase + S::kBadOff, 0u);
    grid_dep_wait();
    bool shear = only_shear || *form != 0;
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    uint32_t tmem_base;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(sbase + S::kTmemOff));

    Ctx cx;
    cx.sbase = sbase, cx.t = t;
    cx.tlane = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    cx.a.w1 = 4u * (2u * (t & 15) + 32u * (t >> 4));
    cx.a.r1 = 4u * (258u * (t & 15) + 32u * (t >> 4));
    cx.a.w2 = 4u * ((t & 15) + 2064u * ((t >> 4) & 1) + 512u * ((t >> 5) & 1) + 1024u * ((t >> 6) & 1));
    cx.a.r2 = 4u * (2u * (t & 15) + 32u * (t >> 4));
    cx.first = blockIdx.x, cx.stride = gridDim.x;
    cx.count = cx.first < rows ? (rows - cx.first + cx.stride - 1) / cx.stride : 0;
    cx.dx = dx, cx.ld = ld, cx.elems = elems, cx.status = status;
    cx.out = partial + static_cast<int64_t>(blockIdx.x) * kSlotFloats;

    for (int pass = 0; pass < 2; ++pass) {
        cx.again = pass != 0, cx.done = pass * cx.count;
        // constants: blocks of 16 columns, [column quad][role][4], all of a thread's loads in flight together; the last two
        // blocks to shared memory; sums to zero
        {
            const float4* base = reinterpret_cast<const float4*>(img) + (shear ? (kCols / 4) * kThreads : 0) + t;
            float4 f[7][4];
#pragma unroll
            for (int j = 0; j < 7; ++j) {
                const int b = group + kGroups * j;
                if (b < kCols / 16) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) f[j][i] = load_plain(base + (4 * b + i) * kThreads);
                }
            }
            const float lift = shear ? 1.f : kLift;
#pragma unroll
            for (int j = 0; j < 7; ++j) {
                const int b = group + kGroups * j;
                if (b >= kCols / 16) continue;
                uint32_t v[16];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float m = 16 * b >= kLastCol ? lift : 1.f;
                    v[4 * i] = __float_as_uint(f[j][i].x * m), v[4 * i + 1] = __float_as_uint(f[j][i].y * m);
                    v[4 * i + 2] = __float_as_uint(f[j][i].z * m), v[4 * i + 3] = __float_as_uint(f[j][i].w * m);
                }
                if (16 * b < kAccCol) {
                    tmem_st16(cx.tlane + 16 * b, v);
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        sts128(sbase + S::kLastOff + (4 * (b - kAccCol / 16) + i) * kThreads * 16 + 16u * t, make_uint4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]));
                }
            }
            uint32_t z[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) z[i] = 0u;
            for (int c = kAccCol + 16 * group; c < 512; c += 16 * kGroups) tmem_st16(cx.tlane + c, z);
            tmem_wait_st();
        }
        tmem_fence_before();
        __syncthreads();
        tmem_fence_after();

        bool bad = false;
        auto run = [&](auto form_tag) {
            constexpr int FORM = decltype(form_tag)::value;
            if (group == 0) {
                regs_down<80>();
                group_a<FORM, IN_F32, STAGES>(cx, &xmap);
                regs_up<128>();
            } else if (group == 1) {
                bad = group_b<FORM, IN_F32, STAGES>(cx);
            } else if (group == 2) {
                bad = group_c<FORM, IN_F32, STAGES>(cx);
            } else {
                regs_up<176>();
                bad = group_d<FORM, IN_F32, STAGES>(cx, &gmap);
                regs_down<128>();
            }
        };
        if (shear) run(std::integral_constant<int, kFormShear>());
        else run(std::integral_constant<int, kFormScaled>());
        if (!shear && bad) sts32(sbase + S::kBadOff, 1u);
        tmem_fence_before();
        __syncthreads();
        tmem_fence_after();
        if (shear || lds32(sbase + S::kBadOff) == 0u) break;
        shear = true;
    }
    if (threadIdx.x == 0) slot_form[blockIdx.x] = shear ? 1 : 0;
    if (warp == 0) tmem_dealloc512(tmem_base);
}

// dtheta [levels][half] from the slots' [12][2048]: stage s, angle j = the sum over the slots and the 2048 / half row
// positions r of entry s * 2048 + r * half + j, times the angle's weight in the form of the slot.  A block = 32 lanes x 32
// angles (half is a multiple of 32): lane y adds terms y, y + 32, ... (term = slot * positions + r) in groups of four, then the
// lanes are added as four sums, so that the roundings at the size of the whole sum are few.  (64 bits throughout were no closer, and
// one row of 4096 took 1.3 us longer.)
__global__ void __launch_bounds__(1024) k_reduce_grad(const float* partial, const int* slot_form, int slots, int half_log,
                                                      const float* weight, float* __restrict__ out) {
    __shared__ float sh[32][33];
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
    const int k = blockIdx.x * 32 + x, s = k >> half_log, j = k & ((1 << half_log) - 1);
    const int pos_log = 11 - half_log, terms = slots << pos_log, at = s * (kN / 2) + j;
    grid_dep_launch();
    grid_dep_wait();
    const float w[2] = {weight[at], weight[kSlotFloats + at]};
    auto weighted = [&](int i, float add) {
        const int slot = i >> pos_log;
        const float v = partial[static_cast<int64_t>(slot) * kSlotFloats + ((i & ((1 << pos_log) - 1)) << half_log) + at];
        return fmaf(v, slot_form[slot] != 0 ? w[1] : w[0], add);
    };
    float acc = 0.f;
    int i = y;
    for (; i + 96 < terms; i += 128) acc += weighted(i, weighted(i + 32, weighted(i + 64, weighted(i + 96, 0.f))));
    for (; i < terms; i += 32) acc = weighted(i, acc);
    sh[y][x] = acc;
    __syncthreads();
    if (y == 0) {
        float a[4] = {};
#pragma unroll
        for (int e = 0; e < 32; ++e) a[e & 3] += sh[e][x];
        out[k] = (a[0] + a[1]) + (a[2] + a[3]);
    }
}

// f(IN_F32, STAGES) for a type and a row length
template <class F>
static cudaError_t choose(bool f32, int levels, F&& f) {
    auto with = [&](auto stages) { return f32 ? f(std::true_type(), stages) : f(std::false_type(), stages); };
    switch (levels) {
        case 7: return with(std::integral_constant<int, 7>());
        case 8: return with(std::integral_constant<int, 8>());
        case 9: return with(std::integral_constant<int, 9>());
        case 10: return with(std::integral_constant<int, 10>());
        case 11: return with(std::integral_constant<int, 11>());
        case 12: return with(std::integral_constant<int, 12>());
        default: return cudaErrorInvalidValue;
    }
}
}  // namespace g4k

size_t grad4096_weight_bytes() { return size_t(2) * g4k::kSlotFloats * sizeof(float); }
size_t grad4096_partial_floats(int ctas) { return size_t(ctas) * g4k::kSlotFloats; }

bool grad4096_available(const bfq_plan* plan) {
    return plan->n >= 128 && plan->n <= f4k::kN && plan->cc_major == 10 && plan->img4096 != nullptr && plan->weight4096 != nullptr &&
           plan->partial_floats >= grad4096_partial_floats(plan->sm_count) && encode_tiled() != nullptr;
}

// what the kernels need once per device (a caller that captures does this before)
cudaError_t grad4096_prepare(int device) {
    static bool attr_set[kMaxDevices] = {false};
    if (attr_set[device]) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    for (int levels = 7; levels <= 12; ++levels)
        for (int f32 = 0; f32 < 2; ++f32)
            if (e == cudaSuccess)
                e = g4k::choose(f32 != 0, levels, [](auto type, auto stages) {
                    constexpr bool kF32Rows = decltype(type)::value;
                    return cudaFuncSetAttribute(g4k::k_grad4096<kF32Rows, decltype(stages)::value>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                int(g4k::Smem<kF32Rows>::kBytes));
                });
    attr_set[device] = e == cudaSuccess;
    return e;
}

// x, g and dx: rows of plan->n elements, ld apart (n < 4096: contiguous), all fp32 or all bf16
cudaError_t grad4096_launch(bfq_plan* plan, const void* x, const void* g, int64_t rows, int64_t ld, void* dx, float* dtheta, bool f32, cudaStream_t st) {
    cudaError_t e = grad4096_prepare(plan->device);
    if (e != cudaSuccess) return e;
    const int n = plan->n;
    CUtensorMap xmap, gmap;
    const bool maps = f32 ? (encode_row_map_f32(&xmap, x, rows, ld, n) && encode_row_map_f32(&gmap, g, rows, ld, n))
                          : (encode_row_map(&xmap, x, rows, ld, n) && encode_row_map(&gmap, g, rows, ld, n));
    if (!maps) return cudaErrorInvalidValue;
    const int64_t elems = rows * n, joint = n < f4k::kN ? (elems + f4k::kN - 1) / f4k::kN : rows, pairs = (joint + 1) / 2;
    const int grid = int(pairs < plan->sm_count ? pairs : plan->sm_count);
    const size_t bytes = size_t(rows - 1) * ld * (f32 ? 4 : 2) + size_t(n) * (f32 ? 4 : 2);
    auto meets = [&](const void* p) {
        const uintptr_t a = reinterpret_cast<uintptr_t>(dx), b = reinterpret_cast<uintptr_t>(p);
        return dx != nullptr && a < b + bytes && b < a + bytes;
    };
    const bool over = meets(x) || meets(g);
    e = g4k::choose(f32, plan->log_n, [&](auto type, auto stages) {
        constexpr bool kF32Rows = decltype(type)::value;
        return launch_overlapped(g4k::k_grad4096<kF32Rows, decltype(stages)::value>, dim3(grid), dim3(g4k::kCta), g4k::Smem<kF32Rows>::kBytes, st, xmap, gmap,
                                 plan->img4096, plan->form_flag + 3, dx, n < f4k::kN ? int64_t(f4k::kN) : ld, plan->partial, plan->slot_form, int(joint),
                                 plan->status_word, over, elems);
    });
    if (e != cudaSuccess) return e;
    plan->last_backward_partials = grid;
    return launch_overlapped(g4k::k_reduce_grad, dim3(plan->log_n * (n / 2) / 32), dim3(1024), 0, st, plan->partial, plan->slot_form, grid, plan->log_n - 1,
                             plan->weight4096, dtheta);
}

}  // namespace bfq
