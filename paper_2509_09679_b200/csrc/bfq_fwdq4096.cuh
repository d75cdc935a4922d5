// The forward kernel of n = 4096 (and of shorter rows, several as one); the description is in bfq_fwdq4096.cu.
#pragma once
#include <type_traits>

#include "bfq_fast.h"
#include "bfq_generic.cuh"
#include "bfq_n4096.cuh"
#include "bfq_row_again.cuh"

namespace bfq {
namespace f4k {

// G row groups per CTA; XB regrouping buffers per group (2: one per regrouping; 1: shared, at the
// price of one more barrier per row)
template <int G, int XB>
struct Smem {
    static constexpr uint32_t kInOff = 0;  // [G][kInSlots][kRowBytes], 1024-byte aligned tiles
    static constexpr uint32_t kExOff = kInOff + G * kInSlots * kRowBytes;  // [G][XB][kExBytes]
    static constexpr uint32_t kBarOff = kExOff + G * XB * kExBytes;       // mbarriers [G][kInSlots]
    static constexpr uint32_t kAmaxOff = kBarOff + 8 * G * kInSlots;      // float [G][2 parities][4 warps]
    static constexpr uint32_t kStatOff = kAmaxOff + 32 * G;               // float [G][2 parities][4 warps][2]: row moments
    static constexpr uint32_t kTmemOff = kStatOff + 64 * G;               // tensor-memory base address
    static constexpr uint32_t kBinsOff = kTmemOff + 16;                   // u64 [16]: the CTA's code counts (statistics)
    static constexpr uint32_t kHistOff = kBinsOff + 128;                  // u32 [G][256]: counts of packed code bytes
    static constexpr uint32_t kUsed = kHistOff + 1024 * G;
    static constexpr uint32_t kBytes = kUsed + 1024;  // slack for the 1024-byte alignment of the TMA tiles
};

// last stage (local bit 3 of phase 3): out_lo = k1*a + k2*b, out_hi = k3*a + k4*b for pairs U0..U0+NU-1
template <int U0, int NU, int CW>
__device__ __forceinline__ void stage_general(u64 (&P)[16], const uint32_t (&T)[CW]) {
    static_assert(8 * NU <= CW, "chunk too small");
#pragma unroll
    for (int i = 0; i < NU; ++i) {
        const int m_lo = U0 + i, m_hi = m_lo | 8;
        const u64 K1 = pack2u(T[8 * i], T[8 * i + 1]), K2 = pack2u(T[8 * i + 2], T[8 * i + 3]);
        const u64 K3 = pack2u(T[8 * i + 4], T[8 * i + 5]), K4 = pack2u(T[8 * i + 6], T[8 * i + 7]);
        const u64 a = P[m_lo], b = P[m_hi];
        P[m_lo] = fma2(K2, b, mul2(K1, a));
        P[m_hi] = fma2(K4, b, mul2(K3, a));
    }
}

// the last stage where it couples nothing (rows shorter than 4096): the factors of the elements are taken off
template <int U0, int NU, int CW>
__device__ __forceinline__ void stage_diagonal(u64 (&P)[16], const uint32_t (&T)[CW]) {
#pragma unroll
    for (int i = 0; i < NU; ++i) {
        const int m_lo = U0 + i, m_hi = m_lo | 8;
        P[m_lo] = mul2(pack2u(T[8 * i], T[8 * i + 1]), P[m_lo]);
        P[m_hi] = mul2(pack2u(T[8 * i + 6], T[8 * i + 7]), P[m_hi]);
    }
}

struct ExAddr {
    uint32_t w1, r1, w2, r2;  // per-thread byte addresses of the two regroupings (write / read side)
    int bar;                  // named barrier of the group
};

// rows shorter than 4096: see SUB at the kernel
__host__ __device__ __forceinline__ constexpr int stages_of_sub(int sub) { return 12 - sub; }

// chunk C of CW words: columns [C*CW, C*CW + CW) of the thread's strip
template <int CW, int STAGES = 12>
struct Chunks {
    static constexpr int kPerStage = 32 / CW;             // chunks per lifting stage
    static constexpr int kLift = 11 * kPerStage;          // chunks of the 11 lifting stages
    static constexpr int kCount = kLift + 64 / CW;        // + the general last stage
    static constexpr int kAfterPhase1 = 4 * kPerStage - 1;  // last chunk of stage 3
    static constexpr int kAfterPhase2 = (STAGES < 8 ? STAGES : 8) * kPerStage - 1;  // last chunk of stage 7, or of the last one before it
    static constexpr int kLastLift = (STAGES < 11 ? STAGES : 11) * kPerStage - 1;
    // the chunk after C: stages that do not exist are passed over, the last one always runs
    __host__ __device__ static constexpr int next(int c) { return c == kLastLift ? kLift : c + 1; }
    static constexpr int kPhase3 = next(kAfterPhase2);
};

template <int FORM, int C, int CW, int SUB>
__device__ __forceinline__ void run_chunk(u64 (&P)[16], const uint32_t (&T)[CW]) {
    using CH = Chunks<CW>;
    constexpr int NU = CW / 4;
    if constexpr (C < CH::kLift) {
        if constexpr (FORM == kFormScaled) {
            stage_scaled<(C / CH::kPerStage) & 3, (C % CH::kPerStage) * NU, NU, CW>(P, T);
        } else {
            stage_lift<(C / CH::kPerStage) & 3, (C % CH::kPerStage) * NU, NU, CW>(P, T);
        }
    } else if constexpr (SUB == 0) {
        stage_general<(C - CH::kLift) * (CW / 8), CW / 8, CW>(P, T);
    } else {
        stage_diagonal<(C - CH::kLift) * (CW / 8), CW / 8, CW>(P, T);
    }
}

__device__ __forceinline__ void regroup1(u64 (&P)[16], const ExAddr& ex) {
#pragma unroll
    for (int m = 0; m < 16; ++m) sts64(ex.w1 + ex1_wr_local(m), P[m]);
    __syncwarp();
#pragma unroll
    for (int m = 0; m < 16; ++m) P[m] = lds64(ex.r1 + ex1_rd_local(m));
}
template <int XB>
__device__ __forceinline__ void regroup2(u64 (&P)[16], const ExAddr& ex) {
    // with one shared buffer, every warp of the group must be past its reads of the first layout
    if constexpr (XB == 1) bar_sync(ex.bar, kGroupThreads);
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        uint32_t lo, hi;
        unpack2u(P[m], lo, hi);
        sts32(ex.w2 + ex2_wr_local(m, 0), lo);
        sts32(ex.w2 + ex2_wr_local(m, 1), hi);
    }
    bar_sync(ex.bar, kGroupThreads);
#pragma unroll
    for (int m = 0; m < 16; ++m) P[m] = lds64(ex.r2 + ex2_rd_local(m));
}

// Chunk C is in Tcur (load already issued); the load of chunk C+1 is issued right after the wait so
// that exactly one tensor-memory load is in flight while chunk C is being used.  `issue_next` runs
// once per row, after the second regrouping's barrier (all reads of the input slot are done by then).
template <int FORM, int C, int CW, int XB, int SUB, class F>
__device__ __forceinline__ void run_chunks(u64 (&P)[16], uint32_t (&Tcur)[CW], uint32_t (&Tnext)[CW], uint32_t tbase,
                                           const ExAddr& ex, const Turn& turn, F&& issue_next) {
    using CH = Chunks<CW, stages_of_sub(SUB)>;
    constexpr int N = CH::next(C);
    if constexpr (C == 0 || C == CH::kAfterPhase1 + 1 || C == CH::kPhase3) turn.acquire();
    tmem_wait_ld(Tcur);
    if constexpr (N < CH::kCount) tmem_ld(tbase + CW * N, Tnext);
    run_chunk<FORM, C, CW, SUB>(P, Tcur);
    if constexpr (C == CH::kAfterPhase1) {
        turn.pass();
        regroup1(P, ex);
    }
    if constexpr (C == CH::kAfterPhase2) {
        turn.pass();
        regroup2<XB>(P, ex);
        issue_next();
    }
    if constexpr (N == CH::kCount) turn.pass();
    if constexpr (N < CH::kCount) run_chunks<FORM, N, CW, XB, SUB>(P, Tnext, Tcur, tbase, ex, turn, issue_next);
}

template <int XB, class F>
__device__ __forceinline__ void run_hadamard(u64 (&P)[16], const ExAddr& ex, F&& issue_next) {
    stage_hadamard<0>(P), stage_hadamard<1>(P), stage_hadamard<2>(P), stage_hadamard<3>(P);
    regroup1(P, ex);
    stage_hadamard<0>(P), stage_hadamard<1>(P), stage_hadamard<2>(P), stage_hadamard<3>(P);
    regroup2<XB>(P, ex);
    issue_next();
    stage_hadamard<0>(P), stage_hadamard<1>(P), stage_hadamard<2>(P), stage_hadamard<3>(P);
}

enum : int { kButterfly = 0, kHadamard = 1 };  // TRANSFORM
enum : int { kOutInt4 = 0, kOutBf16 = 1, kOutInt4Stats = 2, kOutInt2 = 3, kOutInt8 = 4, kOutF32 = 5 };  // OUT

// TRANSFORM: learned butterfly (constants in tensor memory) or the fixed Walsh-Hadamard transform (no constants,
// no tensor memory).  OUT: INT4 codes + fp16 scales, or the rotated rows in bf16 (`yout`, leading dimension ldy), or
// codes + scales + the second and fourth moment of every rotated row (`yout` then points to float [rows][2]) + the
// tensor-wide counts of the 16 code values added to `hist`, or INT2 / INT8 codes + scales.
// STEP: group g passes its token to group (g + STEP) % G, so gcd(STEP, G) groups rotate at a time (0: no tokens).
// ROWS (code outputs only): the rotated rows are written as well, in the type of the input, to `yout` (weight folding that
// keeps W Q^T).
// IN_F32: the rows are fp32 (16 KB each): one input slot per group instead of two, re-armed as soon as the group has
// read it (after the second regrouping's barrier), so the load still has most of a row's time to arrive.
// SUB: rows of n = 4096 >> SUB elements.  Q on 2^SUB consecutive rows is a transform of 4096 elements whose stages from
// log2 n on are the identity, so 2^SUB rows go through the kernel as one ("rows" then counts these; `elems` = all
// elements, the last one may be short: its missing rows arrive as zeros and are not stored).  The absent stages are passed
// over, not multiplied by 1 and 0 (no row may touch another one's infinities); the general last stage becomes a diagonal
// that takes the factors off.  A quantized row's maximum is taken over its own part of the 4096.  A row whose results are not
// finite is done again at the end (bfq_row_again.cuh); to know of one takes sixteen maxima per thread and joint row where
// rows go out.
// STRIDED (rows out alone): the short rows of the output lie ldy >> SUB apart instead of one after the other.
template <int G, int CW, int XB, int TRANSFORM, int OUT, int STEP = 2, bool ROWS = false, bool IN_F32 = false, int SUB = 0, bool STRIDED = false>
__global__ void __launch_bounds__(G * kGroupThreads, 1)
k_fwdq4096(const __grid_constant__ CUtensorMap tmap, const float* img, const int* form,
           uint8_t* __restrict__ codes,
           uint16_t* __restrict__ scales, __nv_bfloat16* __restrict__ yout, int64_t ldy, int rows,
           int* __restrict__ status, uint32_t tx_bytes, int wait_limit, unsigned long long* __restrict__ hist, int64_t elems,
           const __grid_constant__ typename std::conditional<SUB != 0, Again, Never>::type again) {
    using S = Smem<G, XB>;
    constexpr bool kTmem = TRANSFORM == kButterfly;
    constexpr bool kCount = OUT == kOutInt4Stats;
    constexpr float kPost = TRANSFORM == kHadamard ? 1.0f / 64.0f : 1.0f;  // 1/sqrt(4096), exact
    extern __shared__ uint8_t smem_raw[];
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q = warp & 3, g = warp >> 2;
    const int t = q * 32 + lane;  // role within the group: 0..127
    // Constants of this thread's role: the image is stored [column quad][role][4], a warp's load is 512 contiguous
    // bytes, and all of a thread's loads are in flight together, issued before the set-up barrier.  The G warps of a lane quarter share its 26 blocks of 16 columns.  The scaled-form
    // image is fetched on the assumption that the table build selected it; the flag is checked below.
    constexpr int kFillBlocks = (kCols / 16 + G - 1) / G;
    float4 fill[kTmem ? kFillBlocks : 1][4];
    auto fetch_image = [&](const float4* base) {
#pragma unroll
        for (int j = 0; j < kFillBlocks; ++j) {
            const int b = g + j * G;
            if (b < kCols / 16) {
#pragma unroll
                for (int i = 0; i < 4; ++i) fill[j][i] = load_plain(base + (4 * b + i) * 128 + t);
            }
        }
    };
    grid_dep_launch();
    if constexpr (kTmem) {
        if (warp == 0) tmem_alloc512(sbase + S::kTmemOff);
    }
    if (threadIdx.x < G * kInSlots) {
        mbar_init(sbase + S::kBarOff + 8 * threadIdx.x, 1);
        mbar_init_fence();
    }
    if constexpr (kCount) {
        for (uint32_t e = threadIdx.x; e < (128u + 1024u * G) / 4u; e += G * kGroupThreads) sts32(sbase + S::kBinsOff + 4u * e, 0u);
    }
    if constexpr (SUB != 0) {
        if (threadIdx.x < G) sts32(sbase + S::kHistOff + 1024u * threadIdx.x + 256u, 0u);
    }
    // everything above overlaps the end of the kernel before this one; global memory is touched from here on
    grid_dep_wait();
    bool shear = false;
    if constexpr (kTmem) {
        fetch_image(reinterpret_cast<const float4*>(img));
        shear = load_plain(form) != 0;
    }
    if constexpr (kTmem) tmem_fence_before();
    __syncthreads();
    if constexpr (kTmem) tmem_fence_after();
    uint32_t tmem_base = 0;
    if constexpr (kTmem) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(sbase + S::kTmemOff));
    const uint32_t tlane = tmem_base + (static_cast<uint32_t>(q * 32) << 16);

    // row r belongs to group (r / gridDim.x) % G of CTA r % gridDim.x: a last, partial round of rows spreads over
    // the CTAs instead of filling all groups of the first few
    const int first = g * gridDim.x + blockIdx.x;
    const int stride = gridDim.x * G;
    const int count = first < rows ? (rows - first + stride - 1) / stride : 0;
    // rows of group 0, the largest count of the CTA: every group takes that many turns with a token
    const int turns = static_cast<int>(blockIdx.x) < rows ? (rows - blockIdx.x + stride - 1) / stride : 0;
    const uint32_t in_base = sbase + S::kInOff + g * kInSlots * kRowBytes;
    const uint32_t bar_base = sbase + S::kBarOff + 8 * g * kInSlots;
    static_assert(STEP >= 0 && (STEP == 0 || G % STEP == 0), "the rings must have equal length");
    constexpr int kRings = STEP == 0 ? 1 : STEP;  // gcd(STEP, G)
    Turn turn;
    turn.on = kTmem && STEP > 0;
    turn.wait_id = kTurnBar0 + g;
    turn.pass_id = kTurnBar0 + (g + STEP) % G;
    const bool seeds_ring = (g + STEP) % G < kRings;  // this group's successor starts with the token

    // first rows of this group
    constexpr int kSlotsUsed = IN_F32 ? 1 : kInSlots;                // fp32 rows: one slot of 2 * kRowBytes per group
    constexpr uint32_t kSlotBytes = IN_F32 ? 2 * kRowBytes : kRowBytes;
    static_assert(kInSlots == 2, "an fp32 row takes the group's two bf16 slots");
    if (t == 0) {
        for (int k = 0; k < kSlotsUsed && k < count; ++k) {
            mbar_expect_tx(bar_base + 8 * k, tx_bytes);
            tma_load_3d(in_base + k * kSlotBytes, &tmap, 0, 0, (first + k * stride) << SUB, bar_base + 8 * k);
        }
    }
    // fill tensor memory
    if constexpr (kTmem) {
        if (shear) fetch_image(reinterpret_cast<const float4*>(img) + (kCols / 4) * 128);  // the other image after all
#pragma unroll
        for (int j = 0; j < kFillBlocks; ++j) {
            const int b = g + j * G;
            if (b < kCols / 16) {
                uint32_t v[16];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    v[4 * i + 0] = __float_as_uint(fill[j][i].x), v[4 * i + 1] = __float_as_uint(fill[j][i].y);
                    v[4 * i + 2] = __float_as_uint(fill[j][i].z), v[4 * i + 3] = __float_as_uint(fill[j][i].w);
                }
                tmem_st16(tlane + 16 * b, v);
            }
        }
        tmem_wait_st();
        tmem_fence_before();
    }
    __syncthreads();
    if constexpr (kTmem) tmem_fence_after();

    ExAddr ex;
    {
        const uint32_t eb1 = sbase + S::kExOff + g * XB * kExBytes;
        const uint32_t eb2 = eb1 + (XB - 1) * kExBytes;
        const uint32_t t4 = (t >> 4) & 1, t5 = (t >> 5) & 1, t6 = (t >> 6) & 1;
        ex.w1 = eb1 + 4u * (2u * (t & 15) + 32u * (t >> 4));
        ex.r1 = eb1 + 4u * (258u * (t & 15) + 32u * (t >> 4));
        ex.w2 = eb2 + 4u * ((t & 15) + 2064u * t4 + 512u * t5 + 1024u * t6);
        ex.r2 = eb2 + 4u * (2u * (t & 15) + 32u * (t >> 4));
        ex.bar = 1 + g;
    }
    // input tile: thread t owns two runs of 32 bytes, at byte 32 (t & 15) + 1024 (t >> 4) + 512 h of the
    // row, i.e. 16-byte chunks 2 (t & 3) + c of 128-byte line ((t >> 2) & 3) + 8 (t >> 4) + 4 h; the TMA
    // swizzle stores chunk j of line l at position j ^ (l & 7)
    // (fp32 rows: runs of 64 bytes at byte 64 (t & 15) + 2048 (t >> 4) + 1024 h: chunks 4 (t & 1) + c of line
    // ((t & 15) >> 1) + 16 (t >> 4) + 8 h)
    const uint32_t in_line = IN_F32 ? ((t & 15) >> 1) * 128u + (t >> 4) * 2048u : ((t >> 2) & 3) * 128u + (t >> 4) * 1024u;
    const uint32_t in_x = IN_F32 ? ((((t & 1) << 2) ^ ((t >> 1) & 7)) << 4) : ((((t & 3) << 1) ^ ((t >> 2) & 3)) << 4);
    const uint32_t amax_base = sbase + S::kAmaxOff + g * 32;
    uint8_t* const out_t = codes + t;
    const uint32_t bad_flag = sbase + S::kHistOff + 1024u * g + 256u;  // SUB > 0: the group has met a result that is not finite
    const uint32_t hist_g = sbase + S::kHistOff + 1024u * g;  // this group's counts of packed code bytes

    // the whole row loop exists once per stage form: the choice is made once per launch, outside the loop
    auto row_loop = [&](auto form_tag) {
    constexpr int FORM = decltype(form_tag)::value;
    u64 P[16];
    uint32_t T0[CW], T1[CW];

    if (seeds_ring) turn.pass();
    for (int k = 0; k < count; ++k) {
        const int row = first + k * stride;
        const int slot = IN_F32 ? 0 : (k & 1);
        if constexpr (kTmem) tmem_ld(tlane, T0);
        mbar_wait_bounded(bar_base + 8 * slot, (IN_F32 ? k : (k >> 1)) & 1, status, wait_limit);
        const uint32_t src = in_base + slot * kSlotBytes + in_line;
        if constexpr (IN_F32) {
            // run h holds elements 4c .. 4c+3 in 16-byte chunk c; element m of half h is half h of P[m]
            uint4 w[2][4];
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int c = 0; c < 4; ++c) w[h][c] = lds128(src + 1024u * h + (in_x ^ (c << 4)));
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                P[4 * c + 0] = pack2u(w[0][c].x, w[1][c].x);
                P[4 * c + 1] = pack2u(w[0][c].y, w[1][c].y);
                P[4 * c + 2] = pack2u(w[0][c].z, w[1][c].z);
                P[4 * c + 3] = pack2u(w[0][c].w, w[1][c].w);
            }
        } else {
            // run (h, c) holds elements 8c..8c+7 of half h; element m of half h is half h of P[m]
            uint4 w[2][2];
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int c = 0; c < 2; ++c) w[h][c] = lds128(src + 512u * h + (in_x ^ ((c | (h << 2)) << 4)));
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const uint32_t a[4] = {w[0][c].x, w[0][c].y, w[0][c].z, w[0][c].w};
                const uint32_t b[4] = {w[1][c].x, w[1][c].y, w[1][c].z, w[1][c].w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    P[8 * c + 2 * j + 0] = pack2u(bf16_lo(a[j]), bf16_lo(b[j]));
                    P[8 * c + 2 * j + 1] = pack2u(a[j] & 0xFFFF0000u, b[j] & 0xFFFF0000u);
                }
            }
        }
        auto issue_next = [&]() {
            if (t == 0 && k + kSlotsUsed < count) {
                mbar_expect_tx(bar_base + 8 * slot, tx_bytes);
                tma_load_3d(in_base + slot * kSlotBytes, &tmap, 0, 0, (first + (k + kSlotsUsed) * stride) << SUB,
                            bar_base + 8 * slot);
            }
        };
        if constexpr (kTmem) {
            run_chunks<FORM, 0, CW, XB, SUB>(P, T0, T1, tlane, ex, turn, issue_next);
        } else {
            run_hadamard<XB>(P, ex, issue_next);
        }

        static_assert(!ROWS || OUT == kOutInt4 || OUT == kOutInt2 || OUT == kOutInt8, "rows beside codes only");
        static_assert(SUB == 0 || (kTmem && OUT != kOutInt4Stats), "not built for short rows");
        static_assert(!(ROWS && IN_F32 && SUB == 0), "not built for fp32 rows of 4096");
        // elements of this row that exist; thread t's pair of register m is 2t + 256m, +1
        const int64_t left = elems - static_cast<int64_t>(row) * kN;
        const int lim = SUB == 0 || left >= kN ? kN : static_cast<int>(left);
        auto there = [&](int m) { return SUB == 0 || 2 * t + 256 * m < lim; };
        static_assert(!STRIDED || (SUB != 0 && (OUT == kOutBf16 || OUT == kOutF32)), "rows out alone");
        // pairs of elements between where register m's would lie in contiguous rows and where they lie
        auto gap = [&](int m) -> int64_t {
            if constexpr (!STRIDED) return 0;
            else return (SUB < 5 ? m >> (4 - SUB) : 2 * m + (q >> 1)) * (((ldy >> SUB) - (kN >> SUB)) / 2);
        };
        if constexpr (OUT == kOutBf16 || (ROWS && !IN_F32)) {
            // thread t holds elements 2t + 256m, +1: one 32-bit word of the bf16 row per packed register
            uint32_t* out = reinterpret_cast<uint32_t*>(yout + static_cast<int64_t>(row) * ldy) + t;
#pragma unroll
            for (int m = 0; m < 16; ++m) {
                float a, b;
                unpack2(P[m], a, b);
                const __nv_bfloat162 v = __floats2bfloat162_rn(a * kPost, b * kPost);
                if (there(m)) out[128 * m + gap(m)] = *reinterpret_cast<const uint32_t*>(&v);
            }
        }
        if constexpr (OUT == kOutF32 || (ROWS && IN_F32)) {
            // thread t holds elements 2t + 256m, +1: one 64-bit word of the fp32 row per packed register
            u64* out = reinterpret_cast<u64*>(reinterpret_cast<float*>(yout) + static_cast<int64_t>(row) * ldy) + t;
#pragma unroll
            for (int m = 0; m < 16; ++m) {
                float a, b;
                unpack2(P[m], a, b);
                if (there(m)) out[128 * m + gap(m)] = pack2(a * kPost, b * kPost);
            }
        }
        if constexpr (OUT == kOutBf16 || OUT == kOutF32) {
            bar_sync(ex.bar, kGroupThreads);  // every warp is past its reads of the second regrouping buffer
            if constexpr (SUB != 0) sts32_if(__float_as_uint(largest<0>(P)) >= not_finite(OUT == kOutBf16), bad_flag, 1u);
            continue;
        }

        constexpr int kQmax = OUT == kOutInt2 ? 1 : (OUT == kOutInt8 ? 127 : 7);
        // rows that a thread holds parts of (short rows: register m belongs to part m >> kPartShift), and the multiplier of
        // each register
        constexpr int kPartLog = SUB < 4 ? SUB : 4, kParts = 1 << kPartLog, kPartShift = 4 - kPartLog;
        bool plain;         // every scale here is a normal, unsaturated fp16 number: nothing needs clipping
        uint32_t plain_parts = 0u;  // SUB > 0: the same of each part
        uint16_t s16 = 0;
        float inv = 0.f;    // SUB == 0: the row's; else lane s < kParts holds part s's
        if constexpr (SUB == 0) {
            // per-row absmax: thread, warp, then the group's four warps
            float m0 = 0.f, m1 = 0.f;
#pragma unroll
            for (int m = 0; m < 16; ++m) {
                float a, b;
                unpack2(P[m], a, b);
                m0 = fmaxf(m0, fabsf(a));
                m1 = fmaxf(m1, fabsf(b));
            }
            // non-negative floats order like their bit patterns: one integer max-reduction over the warp (fmaxf has
            // already dropped NaNs)
            float amax = fmaxf(m0, m1);
            const uint32_t aslot = amax_base + (k & 1) * 16;
            {
                const uint32_t wmax = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(amax));
                sts32_if(lane == 0, aslot + q * 4, wmax);
            }
            const uint32_t mslot = sbase + S::kStatOff + g * 64 + (k & 1) * 32;
            if constexpr (OUT == kOutInt4Stats) {
                // sum y^2 and sum y^4 of the row: thread (fixed order), warp (xor tree), then the four warps in order
                u64 s2v = pack2(0.f, 0.f), s4v = pack2(0.f, 0.f);
#pragma unroll
                for (int m = 0; m < 16; ++m) {
                    const u64 sq = mul2(P[m], P[m]);
                    s2v = add2(s2v, sq);
                    s4v = fma2(sq, sq, s4v);
                }
                float a2, b2, a4, b4;
                unpack2(s2v, a2, b2), unpack2(s4v, a4, b4);
                float s2 = a2 + b2, s4 = a4 + b4;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    s2 += __shfl_xor_sync(0xFFFFFFFFu, s2, o);
                    s4 += __shfl_xor_sync(0xFFFFFFFFu, s4, o);
                }
                if (lane == 0) sts64(mslot + q * 8, pack2(s2, s4));
            }
            bar_sync(ex.bar, kGroupThreads);
            if constexpr (OUT == kOutInt4Stats) {
                if (t == 0) {
                    float s2 = 0.f, s4 = 0.f;
#pragma unroll
                    for (int w4 = 0; w4 < 4; ++w4) {
                        float a, b;
                        unpack2(lds64(mslot + w4 * 8), a, b);
                        s2 += a, s4 += b;
                    }
                    float* rs = reinterpret_cast<float*>(yout) + 2 * static_cast<int64_t>(row);
                    rs[0] = s2 * (kPost * kPost), rs[1] = s4 * (kPost * kPost * kPost * kPost);
                }
            }
            {
                const uint4 o = lds128(aslot);
                amax = fmaxf(fmaxf(__uint_as_float(o.x), __uint_as_float(o.y)),
                             fmaxf(__uint_as_float(o.z), __uint_as_float(o.w)));
            }
            s16 = row_scale_fast<kQmax>(amax * kPost, &inv);
            inv *= kPost;  // the registers still hold the un-normalised values (kPost is a power of two)
            stg16_if(t == 0, scales + row, s16);
            plain = (((s16 >> 10) & 31u) != 0u) && (s16 != 0x7BFFu);
        } else {
            // lane s of each warp collects the warp's maximum of part s, then the warps' maxima of the part: a part is the
            // whole group's, or (n = 128) that of its lower or upper two warps
            float mx[kParts];
#pragma unroll
            for (int s = 0; s < kParts; ++s) mx[s] = 0.f;
#pragma unroll
            for (int m = 0; m < 16; ++m) {
                float a, b;
                unpack2(P[m], a, b);
                mx[m >> kPartShift] = max_abs_nan(mx[m >> kPartShift], a, b);
            }
            uint32_t mine = 0u;
#pragma unroll
            for (int s = 0; s < kParts; ++s) {
                const uint32_t wmax = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(mx[s]));
                if (lane == s) mine = wmax;
            }
            const int part = lane & (kParts - 1);
            const uint32_t slots = sbase + S::kHistOff + 1024u * g + 512u * (k & 1);  // [part][warp]
            sts32_if(lane < kParts, slots + 16 * part + 4 * q, mine);
            bar_sync(ex.bar, kGroupThreads);
            const uint4 o = lds128(slots + 16 * part);
            const uint32_t lower = max(o.x, o.y), upper = max(o.z, o.w);
            const uint32_t amax = SUB < 5 ? max(lower, upper) : (q < 2 ? lower : upper);
            sts32_if(amax >= not_finite(false), bad_flag, 1u);
            s16 = row_scale_fast<kQmax>(__uint_as_float(amax), &inv);
            const int64_t short_row = SUB < 5 ? (static_cast<int64_t>(row) << SUB) + part
                                              : (static_cast<int64_t>(row) << SUB) + 2 * part + (q >> 1);
            const bool writes = lane < kParts && (SUB < 5 ? q == 0 : (q & 1) == 0) && (short_row << stages_of_sub(SUB)) < elems;
            stg16_if(writes, scales + short_row, s16);
            plain_parts = __ballot_sync(0xFFFFFFFFu, (((s16 >> 10) & 31u) != 0u) && (s16 < 0x7BFFu));  // NaN is not
            plain = plain_parts == 0xFFFFFFFFu;
        }
        float invp[kParts];
#pragma unroll
        for (int s = 0; s < kParts; ++s) invp[s] = SUB == 0 ? inv : __shfl_sync(0xFFFFFFFFu, inv, s);
        auto inv_of = [&](int m) { return invp[m >> kPartShift]; };
        // The code of one value where some scale is not plain.  A part whose own scale is rounds as it does when all are, once
        // (v * inv + the constant, then the constant off): a row's codes must not depend on the rows beside it.
        auto code_of = [&](float v, int m) {
            const bool once = SUB != 0 && ((plain_parts >> (m >> kPartShift)) & 1u) != 0u;
            const float r = once ? __fmaf_rn(v, inv_of(m), 12582912.f) - 12582912.f : rintf(v * inv_of(m));
            return static_cast<int>(fminf(fmaxf(r, static_cast<float>(-kQmax - 1)), static_cast<float>(kQmax)));
        };

        if constexpr (OUT == kOutInt8) {
            // |v * inv| <= qmax (1 + 2^-10) < qmax + 1/2 for a normal, unsaturated fp16 scale: no clipping; v * inv +
            // 1.5 * 2^23 then has the code (two's complement) in its low mantissa bits
            // thread t holds elements 2t + 256m, +1 = bytes 2t + 256m, +1 of the row
            uint16_t* out16 = reinterpret_cast<uint16_t*>(codes + static_cast<size_t>(row) * kN) + t;
            if (plain) {
                // u = code + 128 in the low byte of v * inv + (1.5 * 2^23 + 128), whose other low bits are zero:
                // hi * 256 + lo has u_hi, u_lo in its two low bytes; the XOR turns offset binary into two's complement
                const u64 magic2 = pack2(12583040.0f, 12583040.0f);
#pragma unroll
                for (int m = 0; m < 16; ++m) {
                    uint32_t lo, hi;
                    unpack2u(fma2(P[m], pack2(inv_of(m), inv_of(m)), magic2), lo, hi);
                    if (there(m)) out16[128 * m] = static_cast<uint16_t>((hi * 256u + lo) ^ 0x8080u);
                }
            } else {
#pragma unroll
                for (int m = 0; m < 16; ++m) {
                    float a, b;
                    unpack2(P[m], a, b);
                    const uint32_t lo = static_cast<uint32_t>(code_of(a, m)), hi = static_cast<uint32_t>(code_of(b, m));
                    if (there(m)) out16[128 * m] = static_cast<uint16_t>((lo & 0xFFu) | ((hi & 0xFFu) << 8));
                }
            }
            continue;
        }
        if constexpr (OUT == kOutInt2) {
            // elements 2t + 256m, +1 are half of byte t/2 + 64m: the low half for even t, the high half for odd t.
            // The sixteen 4-bit halves (two codes each) travel in the low halves of the bytes of four words, registers
            // 4w .. 4w+3 in word w.
            uint32_t w[4] = {0u, 0u, 0u, 0u};
            if (plain) {
                // |v * inv| <= 1.0005: v * inv + (1.5 * 2^23 + 2) has u = code + 2 in {1, 2, 3} in its low bits above
                // the constant pattern C = 0x4B400000, so hi * 4 + lo = 5 C + (4 u_hi + u_lo); a Horner chain over four
                // registers gives the nibbles times 256^i plus a constant, one subtraction removes it and one XOR turns
                // every u into the two's complement code
                const u64 magic2 = pack2(12582914.0f, 12582914.0f);
                constexpr uint32_t kBias = static_cast<uint32_t>((5ull * 0x4B400000ull * 0x01010101ull) & 0xFFFFFFFFull);
#pragma unroll
                for (int q4 = 0; q4 < 4; ++q4) {
#pragma unroll
                    for (int i = 3; i >= 0; --i) {
                        uint32_t lo, hi;
                        unpack2u(fma2(P[4 * q4 + i], pack2(inv_of(4 * q4 + i), inv_of(4 * q4 + i)), magic2), lo, hi);
                        w[q4] = w[q4] * 256u + (hi * 4u + lo);
                    }
                    w[q4] = (w[q4] - kBias) ^ 0x0A0A0A0Au;
                }
            } else {
#pragma unroll
                for (int m = 0; m < 16; ++m) {
                    float a, b;
                    unpack2(P[m], a, b);
                    const uint32_t c = (static_cast<uint32_t>(code_of(a, m)) & 3u) | ((static_cast<uint32_t>(code_of(b, m)) & 3u) << 2);
                    w[m >> 2] |= c << (8 * (m & 3));
                }
            }
            // the even thread writes bytes m = 0..7 (its nibbles + the odd thread's), the odd one 8..15 (the even
            // thread's nibbles + its own): one exchange per word, then the two nibbles of a byte side by side
            const bool odd = t & 1;
            uint8_t* out2 = codes + static_cast<size_t>(row) * (kN / 4) + (t >> 1) + (odd ? 64 * 8 : 0);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, odd ? w[h] : w[2 + h], 1);
                const uint32_t bytes = (odd ? other : w[h]) + ((odd ? w[2 + h] : other) << 4);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (SUB == 0 || there((odd ? 8 : 0) + 4 * h + j)) out2[64 * (4 * h + j)] = static_cast<uint8_t>(bytes >> (8 * j));
            }
            continue;
        }

        // codes: thread t holds elements 2t + 256m (+1) = byte t + 128m of the row's packed codes
        uint8_t* out = out_t + static_cast<size_t>(row) * (kN / 2);
        if (plain) {  // |v*inv| <= 7.004
            // q + 8 lands in the low nibble of the fp32 bit pattern of v*inv + (1.5*2^23 + 8), whose other
            // low bits are zero: hi*16 + lo has (q_hi + 8) << 4 | (q_lo + 8) in its low byte
            const u64 magic2 = pack2(12582920.0f, 12582920.0f);
#pragma unroll
            for (int m = 0; m < 16; ++m) {
                uint32_t lo, hi;
                unpack2u(fma2(P[m], pack2(inv_of(m), inv_of(m)), magic2), lo, hi);
                const uint32_t ob = hi * 16u + lo;  // 17 * 0x4B400000 + the offset-binary byte
                if (there(m)) out[128 * m] = static_cast<uint8_t>(ob ^ 0x88u);  // offset binary -> two's complement
                // counted by its offset-binary value; the constant is taken off the base address instead of the index
                if constexpr (kCount) red_shared_inc(hist_g - 4u * (17u * 0x4B400000u) + 4u * ob);
            }
        } else {
#pragma unroll
            for (int m = 0; m < 16; ++m) {
                float a, b;
                unpack2(P[m], a, b);
                const int qa = code_of(a, m), qb = code_of(b, m);
                const uint32_t byte = static_cast<uint32_t>((qa & 0xF) | ((qb & 0xF) << 4));
                if (there(m)) out[128 * m] = static_cast<uint8_t>(byte);
                if constexpr (kCount) red_shared_inc(hist_g + 4u * (byte ^ 0x88u));
            }
        }
    }
    // a group with fewer rows than group 0 keeps the tokens moving
    for (int k = count; k < turns; ++k) {
#pragma unroll
        for (int ph = 0; ph < 3; ++ph) turn.acquire(), turn.pass();
    }
    if (g < kRings) turn.acquire();  // each ring's first group takes its token back: no arrival stays pending
    };
    if (!shear) {
        row_loop(std::integral_constant<int, kFormScaled>());
    } else if constexpr (kTmem) {
        row_loop(std::integral_constant<int, kFormShear>());
    }

    if constexpr (SUB != 0) {
        bar_sync(ex.bar, kGroupThreads);  // the group's stores are done
        if (lds32(bad_flag) != 0u) rows_again(again, first, stride, count, sbase + S::kExOff + g * XB * kExBytes, ex.bar, t);
    }

    if constexpr (kCount) {
        // counts of the G groups per offset-binary byte (two nibbles code + 8) -> the CTA's 16 code counts -> the caller's
        // histogram, indexed by code + 8.  Integer additions: the result does not depend on their order.
        __syncthreads();
        if (threadIdx.x < 256) {
            uint32_t n = 0;
#pragma unroll
            for (int gg = 0; gg < G; ++gg) n += lds32(sbase + S::kHistOff + 1024u * gg + 4u * threadIdx.x);
            if (n != 0u) {
                red_shared_add64(sbase + S::kBinsOff + 8u * (threadIdx.x & 15u), n);
                red_shared_add64(sbase + S::kBinsOff + 8u * (threadIdx.x >> 4), n);
            }
        }
        __syncthreads();
        if (threadIdx.x < 16) {
            const unsigned long long c = lds64(sbase + S::kBinsOff + 8u * threadIdx.x);
            if (c != 0ull) atomicAdd(hist + threadIdx.x, c);
        }
    }
    if constexpr (kTmem) {
        tmem_fence_before();
        __syncthreads();
        if (warp == 0) tmem_dealloc512(tmem_base);
    }
}

}  // namespace f4k

template <int G, int CW, int XB, int TRANSFORM, int OUT, bool ROWS = false, bool IN_F32 = false, int SUB = 0, bool STRIDED = false>
static cudaError_t launch_variant(const bfq_plan* plan, const CUtensorMap& tmap, int64_t rows, uint8_t* codes,
                                  uint16_t* scales, void* y, int64_t ldy, cudaStream_t st,
                                  unsigned long long* hist = nullptr, int64_t elems = 0, const RowSource& source = RowSource{}) {
    using S = f4k::Smem<G, XB>;
    static bool attr_set[kMaxDevices] = {false};
    auto kern = f4k::k_fwdq4096<G, CW, XB, TRANSFORM, OUT, 2, ROWS, IN_F32, SUB, STRIDED>;
    if (!attr_set[plan->device]) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(S::kBytes));
        if (e != cudaSuccess) return e;
        attr_set[plan->device] = true;
    }
    const int64_t want = (rows + G - 1) / G;
    const int grid = int(want < plan->sm_count ? want : plan->sm_count);
    // bytes a row's load is expected to deliver and the bound on polls of its barrier; the test hook announces more
    // bytes than arrive, so that every wait runs out (quickly) and reports through the status word
    const uint32_t tx_bytes = (IN_F32 ? 2 : 1) * f4k::kRowBytes + (plan->test_stuck_wait ? 16u : 0u);
    const int wait_limit = plan->test_stuck_wait ? 4096 : (1 << 22);
    typename std::conditional<SUB != 0, Again, Never>::type again{};
    if constexpr (SUB != 0) {
        using namespace f4k;
        constexpr int kBits = OUT == kOutInt2 ? 2 : (OUT == kOutInt4 ? 4 : (OUT == kOutInt8 ? 8 : 0)), kType = IN_F32 ? kF32 : kBF16;
        again = Again{source, kType, false, stages_of_sub(SUB), elems, kBits, kBits == 0 || ROWS ? y : nullptr, ldy >> SUB, kType, codes, scales};
    }
    return launch_overlapped(kern, dim3(grid), dim3(G * f4k::kGroupThreads), S::kBytes, st, tmap, plan->img4096,
                             plan->form_flag, codes, scales, static_cast<__nv_bfloat16*>(y), ldy, int(rows),
                             plan->status_word, tx_bytes, wait_limit, hist, elems, again);
}

}  // namespace bfq
