// Dense products of the layer-calibration step on the tensor cores, with the low-bit operands dequantized on the fly:
//     C[i][j] = alpha * sum_k A(i, k) * B(j, k),   i < M, j < N, k < K
// where each operand is given as rows of fp32 / bf16 numbers or as packed two's-complement codes with one fp16 scale
// per stored row (the output format of bfq_forward_quant / bfq_fold_weights), stored either [rows][K] or transposed
// [K][rows].  This covers the three products of the reconstruction loss (paper Sec. 3.4):
//     Dequant(Quant(B x)) . Dequant(Quant(W B^T))^T,   err . Dequant(Quant(W B^T)),   err^T . Dequant(Quant(B x)).
//
// Tensor-core side: pairs of CTAs (tcgen05 cta_group::2).  The rows of B are the M side of the MMA (256 per pair, 128 per
// CTA) and the rows of A its N side (`nt` = 32 .. 256 per pair, half per CTA), so that the lanes of an accumulator are
// consecutive columns of C and every store of the epilogue is 128 contiguous bytes.  K blocks of 64.  An operand tile in
// shared memory is up to 128 rows of 128 bytes (64 bf16) with the 128-byte swizzle, and every row is 64 elements that are
// CONTIGUOUS IN THE STORED OPERAND:
//   * stored [rows][K]: shared-memory row r = tile row r, 64 consecutive k (the K-major layout of the tensor core);
//   * stored [K][rows]: shared-memory row 64 h + k = stored row k0 + k, tile rows 64 h .. 64 h + 63 (the MN-major
//     layout: blocks of 64 tile rows 8192 bytes apart, groups of 8 k 1024 bytes apart).
// So one producer thread always turns contiguous stored elements into 16-byte pieces of a 128-byte row, whatever the
// orientation; the instruction descriptor tells the tensor core which layout each operand has.  bf16 operands need no
// conversion and come by TMA straight into the same layout.  Terms per operand:
//   * codes contracted along their stored row: the integer codes are exact in bf16 (one term); the row scale multiplies
//     the finished row / column of C;
//   * codes contracted across stored rows: the scale varies along k.  If the other operand is fp32 the scale multiplies
//     THAT operand before it is split (one fp32 rounding, 2^-24, in front of a split that keeps 2^-17) and the codes stay
//     one exact term; otherwise code x scale (at most 15 significant bits) is stored as hi + lo, exactly;
//   * fp32 numbers: hi + lo = 16 significant bits (relative error 2^-17 per element); bf16 numbers: one term, exact.  Given a
//     workspace, a pass of its own splits an fp32 operand into two bf16 matrices, which then come by TMA; without one every
//     tile splits the rows it needs again, which takes three times as long as the products.
// The MMA thread issues one product per pair of terms (1, 2 or 4 per K step), accumulating all of them in fp32.
//
// What bounds it: per K block a CTA's tensor core works 512 cycles on nt = 256 (one term pair) and reads 64 KB of
// operands from shared memory, while 32 KB are written there: with one CTA per 128 x 128 tile, which this replaces, both
// figures per product were twice as large and the conversion of an element served half as many products.
// Measured on a B200, before -> now (bf16 rows x 2-bit codes, 1000 x 28672 x 8192: 0.98 -> 0.334 ms = 1.40 PFLOP/s; bf16 x bf16,
// 4096 x 8192 x 8192: 0.386 ms = 1.42 PFLOP/s; 8-bit x 2-bit codes, 1000 x 28672 x 8192: 0.270 ms; 4-bit x 4-bit codes,
// 2048 x 4096 x 4096: 0.181 -> 0.057 ms; fp32 x 4-bit codes stored [K][rows]: 0.445 -> 0.175 ms, 0.115 ms split
// beforehand; both stored [K][rows]: 0.400 -> 0.227 ms, 0.126 ms split beforehand).
#include "../../include/bfq.h"

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "bfq_n4096.cuh"
#include "bfq_plan.h"
#include "bfq_ptx.cuh"

namespace bfq {
namespace dqg {
using namespace ptx;

constexpr int kRows = 128;       // shared-memory rows of an operand tile; rows of B per CTA
constexpr int kKB = 64;          // K block: one 128-byte swizzle atom of bf16
constexpr int kMaxNt = 256;      // rows of A per pair of CTAs
constexpr int kMaxStages = 6;
constexpr int kEpi = 128;        // threads 0 .. 127: epilogue, one tensor-memory lane each
constexpr int kProd = 256;       // producers per operand: threads 128 .. 383 build B's tiles, 384 .. 639 A's
constexpr int kIssuer = kEpi + 2 * kProd;  // thread 640: MMAs (even CTA of a pair) or forwarding (odd CTA)
constexpr int kLoader = kIssuer + 32;      // thread 672: TMA loads of bf16 operands
constexpr int kThreads = kLoader + 32;
constexpr uint32_t kTileBytes = kRows * kKB * 2;  // one bf16 term of one operand: 16 KB
// shared memory: operand tiles, and raw pieces of converted operands on their way (128 bytes for each of 512 producers)
constexpr uint32_t kRingTiles = 12, kRingTilesStaged = 9;
constexpr int kStagedPieces = 8;                        // per producer thread
constexpr uint32_t kStagingBytes = 512 * kStagedPieces * 16;
constexpr uint32_t kBarsOff = kRingTilesStaged * kTileBytes + kStagingBytes;  // the larger of the two uses
static_assert(kRingTiles * kTileBytes <= kBarsOff, "both uses lie below the barriers");
constexpr int kWaitLimit = 1 << 22;

struct Operand {
    const void* data;
    const uint16_t* scales;  // fp16 bits, one per stored row (codes only)
    int64_t ld;              // elements (numbers) or codes per stored row pitch
    int kind;                // BFQ_OP_*
    int transposed;          // 0: [rows][K], 1: [K][rows]
    int rows;                // M or N
    int terms;               // bf16 terms an element is stored in
    int scaled;              // codes times their scales go into shared memory (two terms)
    const void* lo;          // kind bf16, two terms: the second matrix of an fp32 operand that was split beforehand
};

__host__ __device__ __forceinline__ bool is_codes(int kind) { return kind >= BFQ_OP_CODES2; }
__host__ __device__ __forceinline__ int stages_of(bool staged, int terms_u, int terms_v) {
    const int fit = static_cast<int>(staged ? kRingTilesStaged : kRingTiles) / (terms_u + terms_v);
    return fit < kMaxStages ? fit : kMaxStages;
}

__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ bool elect_one() {
    uint32_t r;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
    return r != 0;
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool wait_bounded(uint32_t bar, uint32_t parity, int* status) {
    for (int i = 0; i < kWaitLimit; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
    }
    atomicExch(status, 3);
    return false;
}
// Arrival on another CTA's barrier.  What it announces is read by the tensor core of the CTA that wrote it (or is an
// accumulator), never by another CTA's threads, so no fence at cluster scope is needed (one would cost more than the
// products of a K block).
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// both CTAs of a pair allocate and free together
__device__ __forceinline__ void tmem_alloc_pair(uint32_t smem_dst) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_dst) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(taddr) : "memory");
}
// Shared-memory descriptor of a 128-byte-swizzled tile.  K-major operand: rows of 128 bytes, 8-row groups 1024 bytes
// apart (stride field), the leading field unused; one K step of 16 elements is 32 bytes further along the row.
// MN-major operand: rows of 128 bytes hold 64 tile rows for one k, groups of 8 k are 1024 bytes apart (stride field),
// blocks of 64 tile rows 8192 bytes apart (leading field); one K step of 16 is two groups = 2048 bytes further.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t addr, uint32_t leading_bytes) {
    return static_cast<uint64_t>((addr & 0x3FFFFu) >> 4) | (static_cast<uint64_t>(leading_bytes >> 4) << 16) |
           (static_cast<uint64_t>(1024 >> 4) << 32) | (static_cast<uint64_t>(1) << 46) | (static_cast<uint64_t>(2) << 61);
}
// M = 256 over the pair, N = nt; bf16 x bf16 -> fp32 (bit 15 / 16: the M / N operand is MN-major), or 8-bit x 8-bit -> 32-bit
// signed integers
__device__ __forceinline__ uint32_t make_idesc(bool int8, int nt, int u_mn_major, int v_mn_major) {
    return ((int8 ? 2u : 1u) << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(u_mn_major) << 15) |
           (static_cast<uint32_t>(v_mn_major) << 16) | (static_cast<uint32_t>(nt >> 3) << 17) | (uint32_t(2 * kRows >> 4) << 24);
}
// Issued by the one thread of a converged warp whose `lead` is set: a predicate on the instruction and no branch around it,
// so that the operands can stay in uniform registers.
template <bool INT8>
__device__ __forceinline__ void mma_pair(uint32_t lead, uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    if constexpr (INT8) {
        asm volatile(
            "{\n\t.reg .pred p, q;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "setp.ne.b32 q, %5, 0;\n\t"
            "@q tcgen05.mma.cta_group::2.kind::i8 [%0], %1, %2, %3, p;\n\t}"
            ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(lead)
            : "memory");
    } else {
        asm volatile(
            "{\n\t.reg .pred p, q;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "setp.ne.b32 q, %5, 0;\n\t"
            "@q tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
            ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(lead)
            : "memory");
    }
}
// arrives on the barrier at this offset of every CTA in `mask` when the MMAs that this thread has issued so far have finished
__device__ __forceinline__ void mma_commit(uint32_t lead, uint32_t bar, uint16_t mask) {
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "setp.ne.b32 q, %2, 0;\n\t"
        "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n\t}"
        ::"r"(bar), "h"(mask), "r"(lead)
        : "memory");
}
// whether a phase is over, without waiting for it
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// the wait of a converged warp
__device__ __forceinline__ bool wait_warp(uint32_t bar, uint32_t parity, int* status) {
    for (int i = 0; i < kWaitLimit; ++i) {
        if (__all_sync(0xFFFFFFFFu, mbar_try_wait(bar, parity))) return true;
    }
    atomicExch(status, 3);
    return false;
}

// ---- one shared-memory row: 64 elements that are contiguous in the stored operand -------------------------------
__device__ __forceinline__ void sts128(uint32_t at, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(at), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {  // lo in bits 0..15
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ uint32_t sub_bf16x2(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("sub.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}

// Where chunk j (16 bytes = 8 bf16) of shared-memory row `srow` of a tile goes
__device__ __forceinline__ uint32_t chunk_addr(uint32_t tile, int srow, int j) {
    return tile + static_cast<uint32_t>(srow) * 128u + static_cast<uint32_t>((j ^ (srow & 7)) << 4);
}

// two fp32 values -> their bf16 words (hi term, remainder term)
__device__ __forceinline__ void split2(float a, float b, uint32_t& hi, uint32_t& lo) {
    hi = pack_bf16(a, b);
    lo = pack_bf16(a - __uint_as_float(hi << 16), b - __uint_as_float(hi & 0xFFFF0000u));
}

// How the 128 shared-memory rows of an operand tile are cut into 16-byte pieces of the stored operand.  INT8: a row is 128
// codes as bytes instead of 64 elements as bf16.  A group of kThreads threads builds a whole tile by itself; several groups
// of an operand work on different K blocks, because one block's chain (wait for the stage, convert, make the writes
// visible to the tensor core) takes longer than the tensor core takes for the block.
template <int KIND, bool INT8>
struct Pieces {
    static constexpr int kBits = KIND == BFQ_OP_F32 ? 32 : KIND;
    static constexpr int kRowElems = INT8 ? 2 * kKB : kKB;
    static constexpr int kPerRow = kRowElems * kBits / 128;
    static constexpr int kElems = 128 / kBits;
    static constexpr int kThreads = KIND == BFQ_OP_F32 ? 256 : 128;
    static constexpr int kPerThread = kRows * kPerRow / kThreads;
    // of the group's own blocks, how many are on their way
    static constexpr int kDepth = kStagedPieces / kPerThread < 4 ? kStagedPieces / kPerThread : 4;
};

// 8 codes of 4 bits (one word, element e in bits 4e..4e+3, two's complement) -> 4 words of bf16 pairs in element order
__device__ __forceinline__ void codes4_to_bf16(uint32_t w, uint32_t (&o)[4]) {
    const uint32_t x = w ^ 0x88888888u;  // u = code + 8
    // (128 + u_e, 128 + u_{e+4}) as a bf16 pair: the field sits in the low mantissa bits of 128.0 = 0x4300
    const uint32_t t0 = (x & 0x000F000Fu) | 0x43004300u, t1 = ((x >> 4) & 0x000F000Fu) | 0x43004300u;
    const uint32_t t2 = ((x >> 8) & 0x000F000Fu) | 0x43004300u, t3 = ((x >> 12) & 0x000F000Fu) | 0x43004300u;
    const uint32_t off = 0x43084308u;  // 136.0 twice
    const uint32_t c0 = sub_bf16x2(t0, off), c1 = sub_bf16x2(t1, off), c2 = sub_bf16x2(t2, off), c3 = sub_bf16x2(t3, off);
    o[0] = prmt(c0, c1, 0x5410u), o[1] = prmt(c2, c3, 0x5410u);  // elements (0,1), (2,3)
    o[2] = prmt(c0, c1, 0x7632u), o[3] = prmt(c2, c3, 0x7632u);  // elements (4,5), (6,7)
}
// 16 codes of 2 bits (one word) -> 8 words of bf16 pairs in element order
__device__ __forceinline__ void codes2_to_bf16(uint32_t w, uint32_t (&o)[8]) {
    const uint32_t x = w ^ 0xAAAAAAAAu;  // u = code + 2
    uint32_t c[8];                       // c[j] = (code_j, code_{j+8})
#pragma unroll
    for (int j = 0; j < 8; ++j) c[j] = sub_bf16x2(((x >> (2 * j)) & 0x00030003u) | 0x43004300u, 0x43024302u);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        o[j] = prmt(c[2 * j], c[2 * j + 1], 0x5410u);      // elements (2j, 2j+1)
        o[4 + j] = prmt(c[2 * j], c[2 * j + 1], 0x7632u);  // elements (8+2j, 9+2j)
    }
}
// 4 codes of 8 bits (one word) -> 2 words of bf16 pairs: byte u = code + 128 in the low mantissa bits of 2^23
__device__ __forceinline__ void codes8_to_bf16(uint32_t w, uint32_t (&o)[2]) {
    const uint32_t x = w ^ 0x80808080u;
    const float m = 8388736.0f;  // 2^23 + 128
    const float f0 = __uint_as_float(prmt(x, 0x4B000000u, 0x7440u)) - m, f1 = __uint_as_float(prmt(x, 0x4B000000u, 0x7441u)) - m;
    const float f2 = __uint_as_float(prmt(x, 0x4B000000u, 0x7442u)) - m, f3 = __uint_as_float(prmt(x, 0x4B000000u, 0x7443u)) - m;
    o[0] = pack_bf16(f0, f1), o[1] = pack_bf16(f2, f3);
}

// The same codes as 8-bit integers for the integer tensor path, 16 codes -> one 16-byte chunk.  Codes stay where they are
// in their bytes, so that a 2-bit code counts 64 times and a 4-bit code 16 times (kShift; taken off in the epilogue,
// exactly); byte b of word j is code 4 b + j of the 16, the order the 2-bit codes fall into, for every width.
template <int KIND>
struct Int8Chunk {
    static constexpr int kShift = KIND == BFQ_OP_CODES2 ? 6 : (KIND == BFQ_OP_CODES4 ? 4 : 0);
    // w: the 16 codes' words (1, 2 or 4)
    __device__ __forceinline__ static void make(const uint32_t* w, uint32_t (&o)[4]) {
        if constexpr (KIND == BFQ_OP_CODES2) {
            o[0] = (w[0] << 6) & 0xC0C0C0C0u, o[1] = (w[0] << 4) & 0xC0C0C0C0u;
            o[2] = (w[0] << 2) & 0xC0C0C0C0u, o[3] = w[0] & 0xC0C0C0C0u;
        } else if constexpr (KIND == BFQ_OP_CODES4) {
            const uint32_t al = (w[0] << 4) & 0xF0F0F0F0u, ah = w[0] & 0xF0F0F0F0u;  // codes 0, 2, 4, 6 and 1, 3, 5, 7
            const uint32_t bl = (w[1] << 4) & 0xF0F0F0F0u, bh = w[1] & 0xF0F0F0F0u;
            o[0] = prmt(al, bl, 0x6420u), o[1] = prmt(ah, bh, 0x6420u);
            o[2] = prmt(al, bl, 0x7531u), o[3] = prmt(ah, bh, 0x7531u);
        } else {
            const uint32_t a = prmt(w[0], w[1], 0x5140u), b = prmt(w[2], w[3], 0x5140u);
            const uint32_t c = prmt(w[0], w[1], 0x7362u), d = prmt(w[2], w[3], 0x7362u);
            o[0] = prmt(a, b, 0x5410u), o[1] = prmt(a, b, 0x7632u);
            o[2] = prmt(c, d, 0x5410u), o[3] = prmt(c, d, 0x7632u);
        }
    }
};

struct Params {
    Operand u, v;  // B (M side of the MMA) and A (N side)
    float* c;
    int64_t ldc;
    int k;        // length of the contraction
    int kblocks;  // in blocks of 64, or of 128 on the integer path
    int int8;     // both operands are codes along K: kind::i8 products of the integer codes
    float unit;   // integer path: 2^-(the places the codes were left in)
    float alpha;
    int nt;       // rows of A per tile
    int tiles_v;  // tiles along A's rows; consecutive tiles share the rows of B
    int tiles;
    int split;    // pairs per cluster that share a tile, each with its part of K (1: a cluster is one pair, many tiles)
    int* status;
};

// zeroes the elements >= valid of the c-th chunk of a piece (its elements 8c .. 8c+7, two per word)
__device__ __forceinline__ void mask_chunk(uint32_t (&o)[4], int c, int valid) {
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        const int e = 8 * c + 2 * w;
        o[w] = e >= valid ? 0u : (e + 1 >= valid ? (o[w] & 0xFFFFu) : o[w]);
    }
}

// One chunk (8 elements as 4 words of exact bf16 pairs) to chunk j of row `srow`: as it is, or times the scale in two
// terms.  c = which chunk of its piece this is (for the masking of a partial piece).
template <bool SCALED, bool PARTIAL>
__device__ __forceinline__ void store_bf16_chunk(uint32_t tile, int srow, int j, int c, uint32_t (&o)[4], float s, int valid) {
    if constexpr (PARTIAL) mask_chunk(o, c, valid);
    const uint32_t at = chunk_addr(tile, srow, j);
    if constexpr (!SCALED) {
        sts128(at, o[0], o[1], o[2], o[3]);
    } else {
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) split2(__uint_as_float(o[w] << 16) * s, __uint_as_float(o[w] & 0xFFFF0000u) * s, hi[w], lo[w]);
        sts128(at, hi[0], hi[1], hi[2], hi[3]);
        sts128(at + kTileBytes, lo[0], lo[1], lo[2], lo[3]);
    }
}

// Piece p of shared-memory row `srow`.  SCALED (codes contracted across their stored rows): times `s`, two terms; fp32
// numbers: times the scales `f` of the other operand's codes where those vary along k (1 otherwise).  PARTIAL: only the
// first `valid` elements of the piece exist; the others are stored as zero.
template <int KIND, bool SCALED, bool PARTIAL>
__device__ __forceinline__ void convert_piece(const uint4 raw, uint32_t tile, int srow, int p, float s, const float (&f)[4], int valid) {
    if constexpr (KIND == BFQ_OP_F32) {
        // 4 numbers = half of chunk p / 2
        uint32_t hi[2], lo[2];
        split2(__uint_as_float(raw.x) * f[0], __uint_as_float(raw.y) * f[1], hi[0], lo[0]);
        split2(__uint_as_float(raw.z) * f[2], __uint_as_float(raw.w) * f[3], hi[1], lo[1]);
        if constexpr (PARTIAL) {
#pragma unroll
            for (int w = 0; w < 2; ++w) {
                const uint32_t m = 2 * w >= valid ? 0u : (2 * w + 1 >= valid ? 0xFFFFu : 0xFFFFFFFFu);
                hi[w] &= m, lo[w] &= m;
            }
        }
        const uint32_t at = chunk_addr(tile, srow, p >> 1) + 8u * (p & 1);
        asm volatile("st.shared.v2.u32 [%0], {%1,%2};" ::"r"(at), "r"(hi[0]), "r"(hi[1]) : "memory");
        asm volatile("st.shared.v2.u32 [%0], {%1,%2};" ::"r"(at + kTileBytes), "r"(lo[0]), "r"(lo[1]) : "memory");
    } else if constexpr (KIND == BFQ_OP_CODES4) {
        const uint32_t ws[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            uint32_t o[4];
            codes4_to_bf16(ws[w], o);
            store_bf16_chunk<SCALED, PARTIAL>(tile, srow, 4 * p + w, w, o, s, valid);
        }
    } else if constexpr (KIND == BFQ_OP_CODES2) {
        const uint32_t ws[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            uint32_t o8[8];
            codes2_to_bf16(ws[w], o8);
            uint32_t oa[4] = {o8[0], o8[1], o8[2], o8[3]}, ob[4] = {o8[4], o8[5], o8[6], o8[7]};
            store_bf16_chunk<SCALED, PARTIAL>(tile, srow, 8 * p + 2 * w, 2 * w, oa, s, valid);
            store_bf16_chunk<SCALED, PARTIAL>(tile, srow, 8 * p + 2 * w + 1, 2 * w + 1, ob, s, valid);
        }
    } else {
        const uint32_t ws[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t o2a[2], o2b[2];
            codes8_to_bf16(ws[2 * h], o2a);
            codes8_to_bf16(ws[2 * h + 1], o2b);
            uint32_t o[4] = {o2a[0], o2a[1], o2b[0], o2b[1]};
            store_bf16_chunk<SCALED, PARTIAL>(tile, srow, 2 * p + h, h, o, s, valid);
        }
    }
}

// Piece p of shared-memory row `srow` on the integer path
template <int KIND>
__device__ __forceinline__ void convert_piece_int8(const uint4 raw, uint32_t tile, int srow, int p) {
    constexpr int kWords = KIND / 2;          // of 16 codes
    constexpr int kChunks = 4 / kWords;       // 16-byte chunks that a 16-byte piece turns into
    const uint32_t ws[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
    for (int c = 0; c < kChunks; ++c) {
        uint32_t o[4];
        Int8Chunk<KIND>::make(ws + c * kWords, o);
        sts128(chunk_addr(tile, srow, kChunks * p + c), o[0], o[1], o[2], o[3]);
    }
}

// What a role of a CTA walks through: tiles first, first + step, ... below `tiles`, K blocks [kb0, kb1) of each.
struct Walk {
    int first, step, tiles, kb0, kb1;
    __device__ __forceinline__ int blocks() const {
        return first < tiles ? ((tiles - first + step - 1) / step) * (kb1 - kb0) : 0;
    }
};

struct Ring {
    uint32_t sbase, stage_bytes, bar_full, bar_empty;
    int stages;
};

// the tile rows of one operand that this CTA holds
struct Span {
    int tiles_v, row_tile, lim;  // lim: rows of the operand in this CTA's half of a tile
    bool is_u;
    int half;                    // 0 / 1: which CTA of the pair
    __device__ __forceinline__ int row0(int tile) const {
        const int t = is_u ? tile / tiles_v : tile % tiles_v;
        return t * row_tile + half * lim;
    }
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t bytes) {  // bytes = 0: sixteen zeros
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Producer loop of thread r of one of the `groups` groups that build one operand's tiles; group g has blocks g, g + groups,
// ... of the walk.  Piece id = i * kThreads + r (i = 0 .. kPerThread - 1) is piece id % kPerRow of row id / kPerRow, so the
// lanes of a warp read consecutive pieces of the same stored row: global loads are coalesced as far as the stored row
// allows.  Raw pieces go through shared memory (`staging`, `pitch16` bytes between a thread's slots), each thread reading
// only what it copied itself: kDepth blocks ahead cost no registers (with the pieces in registers an fp32 block waited
// most of 3400 cycles for its loads).  ACROSS: the operand is stored [K][rows]; shared-memory row 64 h + k is stored row
// k0 + k, tile rows 64 h .. 64 h + 63.  SCALED / fold: see convert_piece.
template <int KIND, bool ACROSS, bool SCALED, bool INT8>
__device__ __forceinline__ void produce(const Operand& op, int k_len, int g, int groups, int r, uint32_t staging, uint32_t pitch16,
                                        const Span& span, uint32_t tile_off, const Ring& ring, const Walk& walk, const uint16_t* fold,
                                        int* status) {
    using PC = Pieces<KIND, INT8>;
    constexpr int kBits = PC::kBits, kElems = PC::kElems, kPer = PC::kPerThread, kDepth = PC::kDepth;
    constexpr int kRowStep = PC::kThreads / PC::kPerRow;  // rows between a thread's consecutive pieces
    constexpr int kBlockBytes = PC::kRowElems * kBits / 8;  // a K block of a row stored along K
    constexpr bool kFold = KIND == BFQ_OP_F32;
    const int p = r % PC::kPerRow, row_first = r / PC::kPerRow;
    const uint8_t* const base = static_cast<const uint8_t*>(op.data);
    const int64_t pitch = op.ld * kBits / 8;  // bytes of a stored row
    auto srow_of = [&](int i) { return row_first + i * kRowStep; };
    auto active = [&](int i) { return ACROSS ? 64 * (srow_of(i) >> 6) < span.lim : srow_of(i) < span.lim; };
    // how many of piece i's elements exist (0: zeros are staged)
    auto valid_of = [&](int i, int row0, int kb) -> int {
        if constexpr (!ACROSS) {
            return row0 + srow_of(i) < op.rows && (!INT8 || kb * PC::kRowElems + p * kElems < k_len) ? kElems : 0;
        } else {
            const int left = op.rows - (row0 + 64 * (srow_of(i) >> 6) + p * kElems);
            return left < 0 ? 0 : (left > kElems ? kElems : left);
        }
    };
    struct At {
        int tile, kb, row0;
        const uint8_t* src;  // this thread's first piece of the tile, K block 0
    };
    auto enter = [&](At& a) {
        a.row0 = span.row0(a.tile);
        if constexpr (!ACROSS) {
            a.src = base + int64_t(a.row0 + row_first) * pitch + 16 * p;
        } else {
            a.src = base + int64_t(row_first) * pitch + int64_t(a.row0) * kBits / 8 + 16 * p;
        }
    };
    auto advance = [&](At& a, int by) {
        a.kb += by;
        if (a.kb >= walk.kb1) {
            do {
                a.kb -= walk.kb1 - walk.kb0, a.tile += walk.step;
            } while (a.kb >= walk.kb1);
            enter(a);
        }
    };
    auto stage_in = [&](uint32_t slot, const At& a) {
        if (a.tile < walk.tiles) {
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                const uint8_t* src;
                if constexpr (!ACROSS) {
                    src = a.src + int64_t(i * kRowStep) * pitch + int64_t(a.kb) * kBlockBytes;
                } else {
                    // rows repeat every 64: the next 64 tile rows of the same stored rows
                    constexpr int kHalfBytes = 64 * kBits / 8;
                    const int sr = srow_of(i);
                    src = a.src + (int64_t(a.kb) * kKB + ((sr & 63) - row_first)) * pitch + (sr >> 6) * kHalfBytes;
                }
                const bool there = active(i) && valid_of(i, a.row0, a.kb) > 0;
                cp_async16(staging + (slot * kPer + i) * pitch16, there ? src : base, there ? 16u : 0u);
            }
        }
        cp_async_commit();
    };
    constexpr int kScales = SCALED ? kPer : (kFold ? 4 : 1);
    float sc[kScales];
    auto half_at = [](const uint16_t* q) { return __half2float(__ushort_as_half(*q)); };
    auto load_scales = [&](const At& a) {
        if constexpr (SCALED) {
#pragma unroll
            for (int i = 0; i < kPer; ++i) sc[i] = a.tile < walk.tiles ? half_at(op.scales + a.kb * kKB + (srow_of(i) & 63)) : 0.f;
        }
        if constexpr (kFold) {
            // along k: this thread's four k; across: the stored rows of its pieces, which repeat after four
#pragma unroll
            for (int i = 0; i < 4; ++i)
                sc[i] = fold != nullptr && a.tile < walk.tiles ? half_at(fold + a.kb * kKB + (ACROSS ? (srow_of(i) & 63) : 4 * p + i)) : 1.f;
        }
    };
    At ahead{walk.first, walk.kb0, 0, nullptr};
    enter(ahead);
    advance(ahead, g);
    At now = ahead;
    load_scales(now);
#pragma unroll
    for (int d = 0; d < kDepth; ++d) {
        stage_in(d, ahead);
        advance(ahead, groups);
    }
    int s = g % ring.stages;
    uint32_t round = g / ring.stages;  // how many times the ring has wrapped
    uint32_t slot = 0;
    while (now.tile < walk.tiles) {
        cp_async_wait<kDepth - 1>();
        uint4 raw[kPer];
#pragma unroll
        for (int i = 0; i < kPer; ++i) raw[i] = f4k::lds128(staging + (slot * kPer + i) * pitch16);
        float si[kScales];
#pragma unroll
        for (int i = 0; i < kScales; ++i) si[i] = sc[i];
        At next = now;
        advance(next, groups);
        load_scales(next);
        stage_in(slot, ahead);
        advance(ahead, groups);
        slot = slot + 1 == kDepth ? 0 : slot + 1;
        if (round > 0) {  // one answer for the warp
            const bool ok = wait_bounded(ring.bar_empty + 8 * s, (round - 1) & 1, status);
            if (!__all_sync(0xFFFFFFFFu, ok)) break;
        }
        const uint32_t dst = ring.sbase + s * ring.stage_bytes + tile_off;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            if (!active(i)) continue;
            if constexpr (INT8) {
                convert_piece_int8<KIND>(raw[i], dst, srow_of(i), p);
            } else {
                float f[4] = {1.f, 1.f, 1.f, 1.f};
                if constexpr (kFold) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) f[j] = si[ACROSS ? (i & 3) : j];
                }
                const float scale = SCALED ? si[SCALED ? i : 0] : 1.f;
                const int v = ACROSS ? valid_of(i, now.row0, now.kb) : kElems;  // rows that do not exist were staged as zeros
                if (v == kElems) {
                    convert_piece<KIND, SCALED, false>(raw[i], dst, srow_of(i), p, scale, f, v);
                } else {
                    convert_piece<KIND, SCALED, true>(raw[i], dst, srow_of(i), p, scale, f, v);
                }
            }
        }
        fence_proxy_async();  // written through the generic proxy, read by the tensor core through the async one
        __syncwarp();
        if ((threadIdx.x & 31) == 0) mbar_arrive(ring.bar_full + 8 * s);
        now = next;
        s += groups;
        while (s >= ring.stages) s -= ring.stages, ++round;
    }
    cp_async_wait<0>();  // no copy of this CTA may be in flight when it leaves
}

// bf16 operands come by TMA (elements outside the operand arrive as zeros), issued like the products: a converged warp, one
// thread's predicate on the instructions, the next stage's barrier tested ahead.  (One thread's loop behind a branch took 800
// cycles per block and was what the whole kernel waited for.)
__device__ __forceinline__ void expect_if(uint32_t lead, uint32_t bar, uint32_t bytes) {
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n\t}" ::"r"(bar), "r"(bytes), "r"(lead)
                 : "memory");
}
__device__ __forceinline__ void tma_if(uint32_t lead, uint32_t dst, const CUtensorMap* tmap, int c0, int c1, uint32_t bar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t"
        "@q cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n\t}"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tmap)), "r"(c0), "r"(c1), "r"(bar), "r"(lead)
        : "memory");
}
__device__ __forceinline__ void load_tiles(uint32_t lead, const Operand& op, const CUtensorMap* map, int lim, int row0, int kb, uint32_t dst, uint32_t bar) {
    if (op.transposed) {
        for (int h = 0; h < lim; h += 64) tma_if(lead, dst + 128u * h, map, row0 + h, kb * kKB, bar);
    } else {
        tma_if(lead, dst, map, kb * kKB, row0, bar);
    }
}

// `threads` producers (256, or 512 when the other operand comes by TMA) as groups of one tile each
template <int KIND, bool ACROSS, bool SCALED, bool INT8 = false>
__device__ __forceinline__ void produce_groups(const Operand& op, int k_len, int t, int threads, uint32_t staging, const Span& span, uint32_t tile_off,
                                               const Ring& ring, const Walk& walk, const uint16_t* fold, int* status) {
    constexpr int kGroup = Pieces<KIND, INT8>::kThreads;
    // never more groups than stages: a group that skips a whole turn of the ring would meet a barrier two phases behind
    const int groups = threads / kGroup < ring.stages ? threads / kGroup : ring.stages;
    if (t / kGroup >= groups) return;
    produce<KIND, ACROSS, SCALED, INT8>(op, k_len, t / kGroup, groups, t % kGroup, staging + 16u * t, 16u * threads, span, tile_off, ring, walk, fold, status);
}
__device__ __forceinline__ void produce_any(const Params& p, const Operand& op, int t, int threads, uint32_t staging, const Span& span, uint32_t tile_off,
                                            const Ring& ring, const Walk& walk, const uint16_t* fold) {
    if (p.int8) {
        switch (op.kind) {
            case BFQ_OP_CODES2: return produce_groups<BFQ_OP_CODES2, false, false, true>(op, p.k, t, threads, staging, span, tile_off, ring, walk, fold, p.status);
            case BFQ_OP_CODES4: return produce_groups<BFQ_OP_CODES4, false, false, true>(op, p.k, t, threads, staging, span, tile_off, ring, walk, fold, p.status);
            default: return produce_groups<BFQ_OP_CODES8, false, false, true>(op, p.k, t, threads, staging, span, tile_off, ring, walk, fold, p.status);
        }
    }
    if (op.scaled) {
        switch (op.kind) {
            case BFQ_OP_CODES2: return produce_groups<BFQ_OP_CODES2, true, true>(op, p.k, t, threads, staging, span, tile_off, ring, walk, fold, p.status);
            case BFQ_OP_CODES4: return produce_groups<BFQ_OP_CODES4, true, true>(op, p.k, t, threads, staging, span, tile_off, ring, walk, fold, p.status);
            default: return produce_groups<BFQ_OP_CODES8, true, true>(op, p.k, t, threads, staging, span, tile_off, ring, walk, fold, p.status);
        }
    }
    if (op.transposed) {
        switch (op.kind) {
            case BFQ_OP_F32: return produce_groups<BFQ_OP_F32, true, false>(op, p.k, t, threads, staging, span, tile_off, ring, walk, fold, p.status);
            case BFQ_OP_CODES2: return produce_groups<BFQ_OP_CODES2, true, false>(op, p.k, t, threads, staging, span, tile_off, ring, walk, fold, p.status);
            case BFQ_OP_CODES4: return produce_groups<BFQ_OP_CODES4, true, false>(op, p.k, t, threads, staging, span, tile_off, ring, walk, fold, p.status);
            default: return produce_groups<BFQ_OP_CODES8, true, false>(op, p.k, t, threads, staging, span, tile_off, ring, walk, fold, p.status);
        }
    }
    switch (op.kind) {
        case BFQ_OP_F32: return produce_groups<BFQ_OP_F32, false, false>(op, p.k, t, threads, staging, span, tile_off, ring, walk, fold, p.status);
        case BFQ_OP_CODES2: return produce_groups<BFQ_OP_CODES2, false, false>(op, p.k, t, threads, staging, span, tile_off, ring, walk, fold, p.status);
        case BFQ_OP_CODES4: return produce_groups<BFQ_OP_CODES4, false, false>(op, p.k, t, threads, staging, span, tile_off, ring, walk, fold, p.status);
        default: return produce_groups<BFQ_OP_CODES8, false, false>(op, p.k, t, threads, staging, span, tile_off, ring, walk, fold, p.status);
    }
}
// warps that arrive on a stage's barrier for one operand
__device__ __forceinline__ uint32_t arrivals_of(const Operand& op) {
    return op.kind == BFQ_OP_BF16 ? 1u : (op.kind == BFQ_OP_F32 ? 8u : 4u);
}

// The MMA warp of a pair's even CTA: every pair of terms, four K steps of 32 bytes per block.  The issue of a block must
// take less than its MMAs (512 cycles at nt = 256 and one term pair): with a branch around one thread's loop, descriptors
// built per MMA and a blocking wait per block it took 850.  So the warp stays converged, one thread's predicate is on the
// instructions, the steps between descriptors are constants, and the next block's barrier is tested before this block's
// products are issued.
template <bool INT8, bool U_MN, bool V_MN>
__device__ __forceinline__ void issue_products(const Params& p, const Ring& ring, const Walk& walk, uint32_t tmem_base, uint32_t bar_acc_full,
                                               uint32_t bar_acc_empty, uint16_t mask) {
    const uint32_t lead = elect_one() ? 1u : 0u;
    const uint32_t idesc = make_idesc(INT8, p.nt, U_MN, V_MN);
    // descriptors: start address in 16-byte units in the low bits, so steps are additions
    constexpr uint64_t kUStep = (U_MN ? 2048u : 32u) >> 4, kVStep = (V_MN ? 2048u : 32u) >> 4, kTerm = kTileBytes >> 4;
    const uint64_t u_desc = desc_sw128(ring.sbase, U_MN ? 8192u : 16u);
    const uint64_t v_desc = desc_sw128(ring.sbase + p.u.terms * kTileBytes, V_MN ? 8192u : 16u);
    const uint64_t stage_step = ring.stage_bytes >> 4;
    const int blocks = walk.kb1 - walk.kb0;
    int s = 0, n = 0;
    uint32_t parity = 0;
    bool ready = false;
    for (int tile = walk.first; tile < walk.tiles; tile += walk.step, ++n) {
        const int buf = n & 1;
        if (n >= 2 && !wait_warp(bar_acc_empty + 8 * buf, ((n >> 1) - 1) & 1, p.status)) return;
        tmem_fence_after();
        const uint32_t d = tmem_base + buf * kMaxNt;
        uint32_t accumulate = 0u;
        for (int kb = 0; kb < blocks; ++kb) {
            if (!ready && !wait_warp(ring.bar_full + 8 * s, parity, p.status)) return;
            const int s_next = s + 1 == ring.stages ? 0 : s + 1;
            const uint32_t parity_next = s_next == 0 ? parity ^ 1u : parity;
            const bool next = mbar_test(ring.bar_full + 8 * s_next, parity_next);
            tmem_fence_after();
            const uint64_t ud = u_desc + s * stage_step, vd = v_desc + s * stage_step;
            if (INT8 || (p.u.terms == 1 && p.v.terms == 1)) {
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) {
                    mma_pair<INT8>(lead, d, ud + ks * kUStep, vd + ks * kVStep, idesc, accumulate);
                    accumulate = 1u;
                }
            } else {
                for (int iu = 0; iu < p.u.terms; ++iu)
                    for (int iv = 0; iv < p.v.terms; ++iv) {
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks) {
                            mma_pair<false>(lead, d, ud + iu * kTerm + ks * kUStep, vd + iv * kTerm + ks * kVStep, idesc, accumulate);
                            accumulate = 1u;
                        }
                    }
            }
            mma_commit(lead, ring.bar_empty + 8 * s, mask);  // both CTAs may refill the stage
            s = s_next, parity = parity_next;
            ready = __all_sync(0xFFFFFFFFu, next);
        }
        mma_commit(lead, bar_acc_full + 8 * buf, mask);
    }
}

__global__ void __launch_bounds__(kThreads, 1)
k_dequant_gemm(const __grid_constant__ Params p, const __grid_constant__ CUtensorMap map_u, const __grid_constant__ CUtensorMap map_v,
               const __grid_constant__ CUtensorMap map_u_lo, const __grid_constant__ CUtensorMap map_v_lo) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;  // the same offset in both CTAs of a pair
    const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
    // clusters are consecutive CTAs: the rank in the cluster from the (warp-uniform) block index
    const uint32_t rank = p.split == 1 ? blockIdx.x & 1u : blockIdx.x % (2u * p.split), leader = rank & ~1u;
    const int half = static_cast<int>(rank & 1u);
    Ring ring;
    ring.sbase = sbase;
    ring.stage_bytes = static_cast<uint32_t>(p.u.terms + p.v.terms) * kTileBytes;
    ring.stages = stages_of(!(p.u.kind == BFQ_OP_BF16 && p.v.kind == BFQ_OP_BF16), p.u.terms, p.v.terms);
    // barriers: full[6] (a stage's operand tiles are in place: this CTA's and, in the even CTA, the odd CTA's too),
    // empty[6], acc_full[2], acc_empty[2] (even CTA), then the tensor-memory address
    const uint32_t bars = sbase + kBarsOff;
    ring.bar_full = bars, ring.bar_empty = bars + 8 * kMaxStages;
    const uint32_t bar_acc_full = bars + 16 * kMaxStages, bar_acc_empty = bar_acc_full + 16;
    const uint32_t tmem_slot = bar_acc_empty + 16;

    grid_dep_launch();
    if (warp == 0) tmem_alloc_pair(tmem_slot);
    if (tid == kIssuer) {
        const uint32_t arrivals = arrivals_of(p.u) + arrivals_of(p.v) + (half == 0 ? 1u : 0u);
        for (int s = 0; s < kMaxStages; ++s) {
            mbar_init(ring.bar_full + 8 * s, arrivals);
            mbar_init(ring.bar_empty + 8 * s, 1);
        }
        for (int b = 0; b < 2; ++b) mbar_init(bar_acc_full + 8 * b, 1), mbar_init(bar_acc_empty + 8 * b, 2 * kEpi / 32);
        mbar_init_fence();
    }
    tmem_fence_before();
    __syncthreads();
    cluster_sync_all();  // the peers' barriers are initialised
    tmem_fence_after();
    uint32_t tmem_base;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(tmem_base) : "r"(tmem_slot));
    grid_dep_wait();

    Walk walk;
    int slice = 0;
    if (p.split == 1) {
        walk.first = blockIdx.x >> 1, walk.step = gridDim.x >> 1, walk.tiles = p.tiles, walk.kb0 = 0, walk.kb1 = p.kblocks;
    } else {
        slice = static_cast<int>(rank >> 1);
        walk.first = blockIdx.x / (2 * p.split), walk.step = p.tiles, walk.tiles = p.tiles;
        walk.kb0 = p.kblocks * slice / p.split, walk.kb1 = p.kblocks * (slice + 1) / p.split;
    }
    const int hv = p.nt >> 1;  // rows of A per CTA

    // scales that do not vary along k multiply the finished column / row of C
    const bool u_scales = is_codes(p.u.kind) && !p.u.transposed, v_scales = is_codes(p.v.kind) && !p.v.transposed;
    auto u_scale = [&](int j) { return u_scales && j < p.u.rows ? p.alpha * __half2float(__ushort_as_half(p.u.scales[j])) : p.alpha; };
    auto v_scale = [&](int i) { return v_scales && i < p.v.rows ? __half2float(__ushort_as_half(p.v.scales[i])) : 1.f; };

    auto span_of = [&](bool u) {
        Span span;
        span.tiles_v = p.tiles_v, span.is_u = u, span.half = half;
        span.row_tile = u ? 2 * kRows : p.nt, span.lim = u ? kRows : hv;
        return span;
    };
    // an accumulator as a number: the integer path's come with the places its codes were left in
    auto number = [&](uint32_t acc) { return p.int8 ? __int2float_rn(static_cast<int>(acc)) * p.unit : __uint_as_float(acc); };

    if (tid < kEpi) {
        // ---- epilogue: lane = column of C, accumulator column = row of C ----
        const uint32_t tlane = tmem_base + (static_cast<uint32_t>(warp * 32) << 16);
        const uint32_t empty_at_leader = map_to_cta(bar_acc_empty, leader);
        bool ok = true;
        int n = 0;
        for (int tile = walk.first; tile < walk.tiles; tile += walk.step, ++n) {
            const int buf = n & 1;
            ok = wait_bounded(bar_acc_full + 8 * buf, (n >> 1) & 1, p.status);
            ok = __all_sync(0xFFFFFFFFu, ok);  // the tensor-memory loads below are warp-wide
            if (!ok || p.split > 1) break;
            tmem_fence_after();
            const int j = (tile / p.tiles_v) * (2 * kRows) + half * kRows + tid, i0 = (tile % p.tiles_v) * p.nt;
            const bool col_ok = j < p.u.rows;
            const float us = u_scale(j);
            float* out = p.c + int64_t(i0) * p.ldc + j;
            for (int c0 = 0; c0 < p.nt; c0 += 32) {
                uint32_t acc[32];
                tmem_ld32(tlane + buf * kMaxNt + c0, acc);
                tmem_wait_ld32(acc);
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const float v = number(acc[i]) * (us * v_scale(i0 + c0 + i));
                    if (col_ok && i0 + c0 + i < p.v.rows) out[int64_t(c0 + i) * p.ldc] = v;
                }
            }
            tmem_fence_before();
            __syncwarp();
            if ((tid & 31) == 0) mbar_arrive_remote(empty_at_leader + 8 * buf);
        }
    } else if (tid < kIssuer) {
        // ---- producers ----
        // both operands converted: 256 threads each; one of them bf16 (TMA): all 512 convert the other
        const bool u_tma = p.u.kind == BFQ_OP_BF16, v_tma = p.v.kind == BFQ_OP_BF16;
        const int t = tid - kEpi;
        // staging: 64 KB above the ring, half of it for each operand when both are converted
        const uint32_t staging = sbase + kRingTilesStaged * kTileBytes;
        auto convert = [&](bool u, int tt, int threads) {
            const Operand& op = u ? p.u : p.v;
            const Operand& other = u ? p.v : p.u;
            const uint16_t* fold = is_codes(other.kind) && other.transposed && !other.scaled ? other.scales : nullptr;
            produce_any(p, op, tt, threads, staging + (u || threads > kProd ? 0u : kStagingBytes / 2), span_of(u), u ? 0u : static_cast<uint32_t>(p.u.terms) * kTileBytes, ring, walk, fold);
        };
        if (u_tma != v_tma) {
            convert(!u_tma, t, 2 * kProd);
        } else if (!u_tma) {
            convert(t < kProd, t & (kProd - 1), kProd);
        }
    } else if (warp == kLoader / 32) {
        const bool u_tma = p.u.kind == BFQ_OP_BF16, v_tma = p.v.kind == BFQ_OP_BF16;
        if (u_tma || v_tma) {
            const uint32_t lead = elect_one() ? 1u : 0u;
            auto bytes_of = [&](const Operand& op, int lim) { return 128u * static_cast<uint32_t>(op.terms * (op.transposed ? (lim + 63) / 64 * 64 : lim)); };
            const uint32_t u_bytes = bytes_of(p.u, kRows), v_bytes = bytes_of(p.v, hv);
            int s = 0, issued = 0;
            uint32_t parity = 1u;  // of the phase before the first: over, as far as a fresh barrier tells
            bool ok = true, ready = false;
            for (int tile = walk.first; ok && tile < walk.tiles; tile += walk.step) {
                const int u0 = (tile / p.tiles_v) * (2 * kRows) + half * kRows, v0 = (tile % p.tiles_v) * p.nt + half * hv;
                for (int kb = walk.kb0; kb < walk.kb1; ++kb) {
                    if (!ready && !wait_warp(ring.bar_empty + 8 * s, parity, p.status)) {
                        // no copy of this CTA may be in flight when it leaves
                        for (int i = issued > ring.stages ? issued - ring.stages : 0; i < issued; ++i)
                            wait_bounded(ring.bar_full + 8 * (i % ring.stages), (i / ring.stages) & 1, p.status);
                        ok = false;
                        break;
                    }
                    const int s_next = s + 1 == ring.stages ? 0 : s + 1;
                    const uint32_t parity_next = s_next == 0 ? parity ^ 1u : parity;
                    const bool next = mbar_test(ring.bar_empty + 8 * s_next, parity_next);
                    const uint32_t dst = sbase + s * ring.stage_bytes, bar = ring.bar_full + 8 * s;
                    if (u_tma) {
                        expect_if(lead, bar, u_bytes);
                        load_tiles(lead, p.u, &map_u, kRows, u0, kb, dst, bar);
                        if (p.u.terms == 2) load_tiles(lead, p.u, &map_u_lo, kRows, u0, kb, dst + kTileBytes, bar);
                    }
                    if (v_tma) {
                        expect_if(lead, bar, v_bytes);
                        load_tiles(lead, p.v, &map_v, hv, v0, kb, dst + p.u.terms * kTileBytes, bar);
                        if (p.v.terms == 2) load_tiles(lead, p.v, &map_v_lo, hv, v0, kb, dst + (p.u.terms + 1) * kTileBytes, bar);
                    }
                    ++issued;
                    s = s_next, parity = parity_next;
                    ready = __all_sync(0xFFFFFFFFu, next);
                }
            }
        }
    } else if (warp == kIssuer / 32 && half == 0) {
        const uint16_t mask = static_cast<uint16_t>(3u << leader);
        const uint32_t base = __shfl_sync(0xFFFFFFFFu, tmem_base, 0);
        if (p.int8) {
            issue_products<true, false, false>(p, ring, walk, base, bar_acc_full, bar_acc_empty, mask);
        } else if (p.u.transposed) {
            if (p.v.transposed) issue_products<false, true, true>(p, ring, walk, base, bar_acc_full, bar_acc_empty, mask);
            else issue_products<false, true, false>(p, ring, walk, base, bar_acc_full, bar_acc_empty, mask);
        } else {
            if (p.v.transposed) issue_products<false, false, true>(p, ring, walk, base, bar_acc_full, bar_acc_empty, mask);
            else issue_products<false, false, false>(p, ring, walk, base, bar_acc_full, bar_acc_empty, mask);
        }
    } else if (tid == kIssuer) {
        // ---- odd CTA: tell the even CTA which stages are in place here ----
        const uint32_t leader_full = map_to_cta(ring.bar_full, leader);
        const int total = walk.blocks();
        int s = 0;
        uint32_t round = 0;
        for (int at = 0; at < total; ++at) {
            if (!wait_bounded(ring.bar_full + 8 * s, round & 1, p.status)) break;
            mbar_arrive_remote(leader_full + 8 * s);
            if (++s == ring.stages) s = 0, ++round;
        }
    }
    __syncwarp();

    if (p.split > 1) {
        // The pairs of the cluster hold partial sums of one tile.  Every CTA sends accumulator columns [w q, w (q + 1)) to
        // the CTA of its parity in pair q (w = nt / split), into the ring that no MMA reads any more, and adds what it
        // gets in the order of the pairs: layout [sending pair][column][lane].
        cluster_sync_all();
        const int w = p.nt / p.split;
        if (tid < kEpi) {
            tmem_fence_after();
            const uint32_t tlane = tmem_base + (static_cast<uint32_t>(warp * 32) << 16);
            for (int c0 = 0; c0 < p.nt; c0 += 8) {
                uint32_t acc[8];
                tmem_ld8(tlane + c0, acc);
                tmem_wait_ld8(acc);
                const int q = c0 / w;
                const uint32_t dst = map_to_cta(sbase, static_cast<uint32_t>(2 * q + half)) +
                                     4u * static_cast<uint32_t>((slice * w + (c0 - q * w)) * kRows + tid);
#pragma unroll
                for (int i = 0; i < 8; ++i) st_cluster_b32(dst + 4u * kRows * i, acc[i]);
            }
            tmem_fence_before();
        }
        cluster_sync_all();
        const int tile = walk.first, lane = tid & (kRows - 1);
        const int j = (tile / p.tiles_v) * (2 * kRows) + half * kRows + lane, i0 = (tile % p.tiles_v) * p.nt + slice * w;
        if (tid < kIssuer && j < p.u.rows) {
            const float us = u_scale(j);
            for (int c = tid / kRows; c < w && i0 + c < p.v.rows; c += kIssuer / kRows) {
                float sum = 0.f;
                int isum = 0;
                for (int q = 0; q < p.split; ++q) {
                    uint32_t bits;
                    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(bits) : "r"(sbase + 4u * static_cast<uint32_t>((q * w + c) * kRows + lane)));
                    isum += static_cast<int>(bits), sum += __uint_as_float(bits);
                }
                if (p.int8) sum = number(static_cast<uint32_t>(isum));
                p.c[int64_t(i0 + c) * p.ldc + j] = sum * (us * v_scale(i0 + c));
            }
        }
    }
    tmem_fence_before();
    cluster_sync_all();  // nobody's barriers or operand tiles are in use by a peer any more
    if (warp == 0) tmem_dealloc_pair(tmem_base);
}

// ---- a few rows of A against coded rows of B -----------------------------------------------------------------------
// A decoded token or a few: the product is a pass over B's codes, and a 256-row tile of the pair kernel keeps 32 to 128
// CTAs in a chain of K blocks (one token, 4096 x 4096 at 2 bits: 17 - 25 us).  Here a CTA of eight warps takes 16 rows of B, each
// warp every eighth part of K, and the partial sums are added in the order of the warps.  mma.sync m16n8k16 with the codes as
// the 16-row operand straight from registers: a lane's 16 bytes of a row are its k values, in whatever order they come, as
// long as the lanes that hold A's rows take the same ones.  Two code operands are multiplied as integers (m16n8k32), so that a
// row of C is the same exact number here and in the pair kernel's integer products.
// What bounds it: on a small layer the latency of one pass; on a wide one the instructions that turn codes into bf16 pairs and
// feed them to the m16n8k16 products, and with eight bf16 rows the reading of all of A for every 16 rows of B.  us, one row /
// eight: 4096 x 4096 at 2 bits bf16 9.4 / 13.2, INT4 codes 7.7 / 7.8 as bf16 pairs -> 4.5 / 4.5 as integers; 28672 x 8192 bf16
// 44 / 76, INT4 52 / 52 -> 16 / 16, INT8 53 / 54 -> 18 / 24 (its codes alone take 9).
constexpr int kFewWarps = 8;

__device__ __forceinline__ void mma_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_16832(int (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// 16 bytes of codes -> 64 / KIND * 2 bf16 pairs in element order
template <int KIND>
__device__ __forceinline__ void codes_to_pairs(const uint4& raw, uint32_t (&o)[64 / KIND]) {
    const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if constexpr (KIND == BFQ_OP_CODES2) {
            uint32_t t[8];
            codes2_to_bf16(w[i], t);
#pragma unroll
            for (int j = 0; j < 8; ++j) o[8 * i + j] = t[j];
        } else if constexpr (KIND == BFQ_OP_CODES4) {
            uint32_t t[4];
            codes4_to_bf16(w[i], t);
#pragma unroll
            for (int j = 0; j < 4; ++j) o[4 * i + j] = t[j];
        } else {
            uint32_t t[2];
            codes8_to_bf16(w[i], t);
            o[2 * i] = t[0], o[2 * i + 1] = t[1];
        }
    }
}
// UK: kind of B's codes, VK: kind of A
template <int UK, int VK>
__global__ void __launch_bounds__(32 * kFewWarps) k_few_rows(const Operand u, const Operand v, float* __restrict__ c, int64_t ldc, int k, float alpha) {
    constexpr int kElems = 128 / UK;  // codes of 16 bytes of B
    constexpr int kVBits = VK == BFQ_OP_BF16 ? 16 : VK;
    constexpr int kVElems = VK == BFQ_OP_BF16 ? 8 : 128 / VK;           // of 16 bytes of A
    constexpr int kRound = kElems > kVElems ? kElems : kVElems;          // codes of B and elements of A taken together
    constexpr int kVLoads = kRound / kVElems, kULoads = kRound / kElems;
    constexpr bool kInts = VK != BFQ_OP_BF16;                            // exact sums: K < 2^17
    using Sum = typename std::conditional<kInts, int, float>::type;
    __shared__ Sum part[kFewWarps][8][16 + 1];
    grid_dep_launch();
    grid_dep_wait();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
    const int j0 = blockIdx.x * 16;
    const uint8_t* urow[2];
    bool there[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int j = j0 + g + 8 * h;
        there[h] = j < u.rows;
        urow[h] = static_cast<const uint8_t*>(u.data) + int64_t(there[h] ? j : 0) * (u.ld * UK / 8);
    }
    const int i0 = 8 * blockIdx.y;  // the MMA's eight columns
    const bool has_v = i0 + g < v.rows;
    const uint8_t* vrow = static_cast<const uint8_t*>(v.data) + int64_t(has_v ? i0 + g : 0) * (v.ld * kVBits / 8);
    Sum acc[4] = {0, 0, 0, 0};
    // a lane's kRound elements of each row start at a multiple of kRound: inside K as a whole, or cut at a 16-byte piece
    auto piece = [&](const uint8_t* row, bool yes, int at, int bits) {
        return yes && at < k ? *reinterpret_cast<const uint4*>(row + int64_t(at) * bits / 8) : make_uint4(0u, 0u, 0u, 0u);
    };
    constexpr int kStride = kFewWarps * 4 * kRound;
    uint4 w[2][kULoads];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < kULoads; ++i) w[h][i] = piece(urow[h], there[h], k0 + i * kElems, UK);
    };
    int kl = (4 * warp + q) * kRound;
    fetch(kl);
    for (; kl - q * kRound < k; kl += kStride) {
        uint4 x[kVLoads], now[2][kULoads];
#pragma unroll
        for (int i = 0; i < kVLoads; ++i) x[i] = piece(vrow, has_v, kl + i * kVElems, kVBits);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < kULoads; ++i) now[h][i] = w[h][i];
        fetch(kl + kStride);
        if constexpr (kInts) {
            auto words = [](const uint4& r) { return reinterpret_cast<const uint32_t*>(&r); };
#pragma unroll
            for (int e = 0; e < kRound; e += 16) {  // sixteen codes of each row
                uint32_t a[4], b[4], xi[4];
                constexpr int kUWords = UK / 2, kVWords = VK / 2;
                Int8Chunk<UK>::make(words(now[0][e / kElems]) + (e % kElems) / 16 * kUWords, a);
                Int8Chunk<UK>::make(words(now[1][e / kElems]) + (e % kElems) / 16 * kUWords, b);
                Int8Chunk<VK>::make(words(x[e / kVElems]) + (e % kVElems) / 16 * kVWords, xi);
                mma_16832(acc, a[0], b[0], a[1], b[1], xi[0], xi[1]);
                mma_16832(acc, a[2], b[2], a[3], b[3], xi[2], xi[3]);
            }
        } else {
#pragma unroll
            for (int part_u = 0; part_u < kULoads; ++part_u) {
                uint32_t a[64 / UK], b[64 / UK];
                codes_to_pairs<UK>(now[0][part_u], a);
                codes_to_pairs<UK>(now[1][part_u], b);
#pragma unroll
                for (int s = 0; s < kElems / 4; ++s) {
                    const int e = part_u * kElems + 4 * s;  // element of the round: half of a 16-byte piece of A
                    const uint4& xe = x[e / 8];
                    mma_16816(acc, a[2 * s], b[2 * s], a[2 * s + 1], b[2 * s + 1], e % 8 == 0 ? xe.x : xe.z, e % 8 == 0 ? xe.y : xe.w);
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) part[warp][2 * q + (i & 1)][g + 8 * (i >> 1)] = acc[i];
    __syncthreads();
    for (int e = threadIdx.x; e < 8 * 16; e += 32 * kFewWarps) {
        const int i = i0 + (e >> 4), j = e & 15;
        if (i >= v.rows || j0 + j >= u.rows) continue;
        Sum sum = 0;
#pragma unroll
        for (int x = 0; x < kFewWarps; ++x) sum += part[x][e >> 4][j];
        float scale = alpha * __half2float(__ushort_as_half(u.scales[j0 + j]));
        if (is_codes(VK)) scale *= __half2float(__ushort_as_half(v.scales[i]));
        float value = sum;
        if constexpr (kInts) value = __int2float_rn(sum) * (1.f / float(1 << (Int8Chunk<UK>::kShift + Int8Chunk<VK>::kShift)));
        c[int64_t(i) * ldc + j0 + j] = value * scale;
    }
}

// ---- host side ---------------------------------------------------------------------------------------------------
static Operand make_operand(const void* data, const uint16_t* scales, int64_t ld, int kind, int transposed, int rows, int other_kind) {
    Operand op{data, scales, ld, kind, transposed, rows, 1, 0, nullptr};
    op.scaled = is_codes(kind) && transposed && other_kind != BFQ_OP_F32;  // else the scales go into the fp32 operand
    op.terms = kind == BFQ_OP_F32 || op.scaled ? 2 : 1;
    return op;
}

// An fp32 operand as two bf16 matrices hi + lo of its stored rows (pitch: the row's length rounded up to 8), times the other
// operand's scales where those vary along k: `row_scales` per stored row (stored [K][rows]), `col_scales` per element of a row.
// The same arithmetic as in the tiles, so the products come out the same.  Bound by memory: 8 bytes per element.
__global__ void __launch_bounds__(256) k_split_rows(const float* x, int64_t ld, int64_t rows, int width, const uint16_t* row_scales,
                                                    const uint16_t* col_scales, uint16_t* __restrict__ hi, uint16_t* __restrict__ lo) {
    grid_dep_launch();
    grid_dep_wait();
    const int chunks = (width + 7) / 8;
    const int64_t total = rows * chunks, step = int64_t(gridDim.x) * blockDim.x;
    auto half_at = [](const uint16_t* q) { return __half2float(__ushort_as_half(*q)); };
    for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < total; e += step) {
        const int64_t r = e / chunks;
        const int c = 8 * static_cast<int>(e - r * chunks);
        const float4* src = reinterpret_cast<const float4*>(x + r * ld + c);
        const float4 none = make_float4(0.f, 0.f, 0.f, 0.f), a = *src, b = c + 4 < width ? src[1] : none;
        float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        const float rs = row_scales != nullptr ? half_at(row_scales + r) : 1.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            v[i] *= rs;
            if (c + i >= width) v[i] = 0.f;
            else if (col_scales != nullptr) v[i] *= half_at(col_scales + c + i);
        }
        uint32_t h[4], l[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) split2(v[2 * i], v[2 * i + 1], h[i], l[i]);
        *reinterpret_cast<uint4*>(hi + 8 * e) = make_uint4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<uint4*>(lo + 8 * e) = make_uint4(l[0], l[1], l[2], l[3]);
    }
}

static int code_shift(int kind) {
    return kind == BFQ_OP_CODES2 ? Int8Chunk<BFQ_OP_CODES2>::kShift : (kind == BFQ_OP_CODES4 ? Int8Chunk<BFQ_OP_CODES4>::kShift : 0);
}

static bool encode_operand(CUtensorMap* map, const Operand& op, int64_t k, int box_rows) {
    // stored [rows][K]: box of 64 k x box_rows rows; stored [K][rows]: box of 64 rows x 64 k
    const cuuint64_t inner = static_cast<cuuint64_t>(op.transposed ? op.rows : k), outer = static_cast<cuuint64_t>(op.transposed ? k : op.rows);
    const cuuint64_t dims[2] = {inner, outer};
    const cuuint64_t strides[1] = {static_cast<cuuint64_t>(op.ld) * 2};
    const cuuint32_t box[2] = {kKB, static_cast<cuuint32_t>(op.transposed ? kKB : box_rows)};
    const cuuint32_t estr[2] = {1, 1};
    return encode_tiled() != nullptr &&
           encode_tiled()(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(op.data), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct Shape {
    int nt, tiles_v, tiles, split;
};
// Rows of A per tile and pairs per tile.  Model in SM cycles: a round of a pair is its K blocks at the slower of the
// tensor core (nt / 2 cycles per K step and term pair) and shared memory (operands written once and read once, 128 bytes
// a cycle: 64 + nt / 4), plus what a tile costs besides (filling the ring, draining the accumulators); a tile shared by
// 2 or 4 pairs has that much less of K and an exchange more, and is worth it only while all the pairs run at once.
// nt_step: 32 (the MMA's N step), or more where A is codes stored [K][rows]: a CTA's half of the tile has to start on a
// whole 16-byte piece.
static Shape choose_shape(int64_t m, int64_t n, int kblocks, int term_pairs, int nt_step, int sms) {
    const int64_t pairs = sms / 2 > 0 ? sms / 2 : 1, tiles_u = (n + 2 * kRows - 1) / (2 * kRows);
    Shape best{};
    double best_cost = 0.0;
    for (int nt = kMaxNt; nt >= nt_step; nt -= nt_step) {
        const int64_t tiles_v = (m + nt - 1) / nt, tiles = tiles_u * tiles_v;
        const int step = nt / 2 > 64 + nt / 4 ? nt / 2 : 64 + nt / 4;
        for (int split = 1; split <= 4; split *= 2) {
            // eight-CTA clusters: only about half of the chip's pairs run at once as such (4096 x 4096, 64 rows: 28 us with four
            // pairs to a tile against 21 with two)
            if (split > 1 && (tiles * split > (split == 4 ? pairs / 2 : pairs) || kblocks < 4 * split)) break;
            const int64_t rounds = split > 1 ? 1 : (tiles + pairs - 1) / pairs;
            const double cost = double(rounds) * ((kblocks + split - 1) / split) * (kKB / 16) * step * term_pairs +
                                double(rounds) * 500 + 2000 + 16 * nt + (split > 1 ? 2000 : 0);
            if (best.nt == 0 || cost < best_cost) best_cost = cost, best = Shape{nt, int(tiles_v), int(tiles), split};
        }
    }
    return best;
}

// Up to eight rows of A one pass over the codes is faster than tiles at every size measured (1 row, us, tiles -> pass:
// 1024 x 1024 at 2 bits 7.7 -> 2.8, 4096 x 4096 25 -> 9.4, 28672 x 8192 104 -> 44; 8 rows 8.1 -> 3.2, 26 -> 13, 105 -> 76).  More
// rows are more passes, worth it while they are small together.
static bool use_few_rows(const Operand& u, const Operand& v, int64_t k) {
    if (!is_codes(u.kind) || u.transposed || v.kind == BFQ_OP_F32 || v.transposed || k >= (is_codes(v.kind) ? 1 << 17 : 1 << 30)) return false;
    const int64_t passes = (int64_t(v.rows) + 7) / 8;
    return passes == 1 || (passes <= 8 && passes * u.rows * k <= int64_t(1) << 25);
}
template <int UK, int VK>
static cudaError_t launch_few(const Operand& u, const Operand& v, float* c, int64_t ldc, int k, float alpha, cudaStream_t st) {
    return launch_overlapped(k_few_rows<UK, VK>, dim3(unsigned((u.rows + 15) / 16), unsigned((v.rows + 7) / 8)), dim3(32 * kFewWarps), 0, st, u, v, c, ldc, k, alpha);
}
template <int UK>
static cudaError_t launch_few(const Operand& u, const Operand& v, float* c, int64_t ldc, int k, float alpha, cudaStream_t st) {
    if (v.kind == BFQ_OP_BF16) return launch_few<UK, BFQ_OP_BF16>(u, v, c, ldc, k, alpha, st);
    if (v.kind == BFQ_OP_CODES2) return launch_few<UK, BFQ_OP_CODES2>(u, v, c, ldc, k, alpha, st);
    if (v.kind == BFQ_OP_CODES4) return launch_few<UK, BFQ_OP_CODES4>(u, v, c, ldc, k, alpha, st);
    return launch_few<UK, BFQ_OP_CODES8>(u, v, c, ldc, k, alpha, st);
}

// Bytes of one of an fp32 operand's two matrices, and whether splitting it beforehand pays: a pair that works on 16 K blocks
// or more loses 20 us and up in its own tiles (2900 cycles a block against 1000), the pass takes 3 us and 8 bytes per element.
static size_t plane_bytes(const Operand& op, int64_t k) {
    const int64_t stored = op.transposed ? k : op.rows, width = op.transposed ? op.rows : k;
    return (size_t(stored) * ((width + 7) / 8 * 8) * 2 + 255) / 256 * 256;
}
static bool split_pays(const Operand& u, const Operand& v, int64_t k, int sms) {
    if (u.kind != BFQ_OP_F32 && v.kind != BFQ_OP_F32) return false;
    const Shape shape = choose_shape(v.rows, u.rows, int(k / kKB), u.terms * v.terms, 32, sms);
    const int64_t pairs = sms / 2 > 0 ? sms / 2 : 1, rounds = shape.split > 1 ? 1 : (shape.tiles + pairs - 1) / pairs;
    return rounds * (k / kKB) / shape.split >= 16;
}
// replaces an fp32 operand by its two matrices at *workspace and moves the pointer on
static cudaError_t split_operand(Operand& op, const Operand& other, int64_t k, uint8_t** workspace, cudaStream_t st) {
    if (op.kind != BFQ_OP_F32) return cudaSuccess;
    const int64_t stored = op.transposed ? k : op.rows, width = op.transposed ? op.rows : k, pitch = (width + 7) / 8 * 8;
    const size_t bytes = plane_bytes(op, k);
    uint16_t *hi = reinterpret_cast<uint16_t*>(*workspace), *lo = reinterpret_cast<uint16_t*>(*workspace + bytes);
    *workspace += 2 * bytes;
    const uint16_t* fold = is_codes(other.kind) && other.transposed && !other.scaled ? other.scales : nullptr;
    const int64_t blocks = (stored * (pitch / 8) + 255) / 256;
    const cudaError_t e = launch_overlapped(k_split_rows, dim3(unsigned(blocks < (1 << 20) ? blocks : (1 << 20))), dim3(256), 0, st, static_cast<const float*>(op.data),
                                            op.ld, stored, int(width), op.transposed ? fold : nullptr, op.transposed ? nullptr : fold, hi, lo);
    op.data = hi, op.lo = lo, op.kind = BFQ_OP_BF16, op.ld = pitch;
    return e;
}

static cudaError_t launch(const Params& p, const CUtensorMap& map_u, const CUtensorMap& map_v, const CUtensorMap& map_u_lo, const CUtensorMap& map_v_lo, int sms,
                          size_t smem, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    const int pairs = p.split > 1 ? p.tiles * p.split : (p.tiles < sms / 2 ? p.tiles : (sms / 2 > 0 ? sms / 2 : 1));
    cfg.gridDim = dim3(unsigned(2 * pairs)), cfg.blockDim = dim3(kThreads), cfg.dynamicSmemBytes = smem, cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = unsigned(2 * p.split), attr[0].val.clusterDim.y = 1, attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr, cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, k_dequant_gemm, p, map_u, map_v, map_u_lo, map_v_lo);
}

}  // namespace dqg
}  // namespace bfq

extern "C" size_t bfq_dequant_gemm_workspace(const bfq_plan* plan, int64_t m, int64_t n, int64_t k, int a_kind, int a_transposed, int b_kind,
                                            int b_transposed) {
    using namespace bfq::dqg;
    if (plan == nullptr || m <= 0 || n <= 0 || k <= 0 || k % kKB != 0 || m >= (int64_t(1) << 31) || n >= (int64_t(1) << 31) || k >= (int64_t(1) << 31)) return 0;
    const Operand u = make_operand(nullptr, nullptr, 0, b_kind, b_transposed, int(n), a_kind);
    const Operand v = make_operand(nullptr, nullptr, 0, a_kind, a_transposed, int(m), b_kind);
    if (!split_pays(u, v, k, plan->sm_count)) return 0;
    return 2 * ((a_kind == BFQ_OP_F32 ? plane_bytes(v, k) : 0) + (b_kind == BFQ_OP_F32 ? plane_bytes(u, k) : 0));
}

extern "C" int bfq_dequant_gemm(bfq_plan* plan, int64_t m, int64_t n, int64_t k, float alpha, const void* a, int a_kind,
                                int a_transposed, int64_t lda, const uint16_t* a_scales, const void* b, int b_kind,
                                int b_transposed, int64_t ldb, const uint16_t* b_scales, float* c, int64_t ldc, void* stream) {
    return bfq_dequant_gemm_split(plan, m, n, k, alpha, a, a_kind, a_transposed, lda, a_scales, b, b_kind, b_transposed, ldb, b_scales, c, ldc, nullptr, 0,
                                  stream);
}

extern "C" int bfq_dequant_gemm_split(bfq_plan* plan, int64_t m, int64_t n, int64_t k, float alpha, const void* a, int a_kind,
                                      int a_transposed, int64_t lda, const uint16_t* a_scales, const void* b, int b_kind,
                                      int b_transposed, int64_t ldb, const uint16_t* b_scales, float* c, int64_t ldc, void* workspace,
                                      size_t workspace_bytes, void* stream) {
    using namespace bfq::dqg;
    if (plan == nullptr) return BFQ_ERR_NULL;
    if (m < 0 || n < 0 || k < 0 || k % kKB != 0 || m >= (int64_t(1) << 31) || n >= (int64_t(1) << 31) || k >= (int64_t(1) << 31))
        return BFQ_ERR_STRIDE;
    if (m == 0 || n == 0) return BFQ_OK;
    if (a == nullptr || b == nullptr || c == nullptr) return BFQ_ERR_NULL;
    auto check = [&](const void* data, int kind, int transposed, int64_t ld, const uint16_t* scales, int64_t rows) -> int {
        const bool codes = kind == BFQ_OP_CODES2 || kind == BFQ_OP_CODES4 || kind == BFQ_OP_CODES8;
        if (!codes && kind != BFQ_OP_F32 && kind != BFQ_OP_BF16) return BFQ_ERR_DTYPE;
        if (codes && scales == nullptr) return BFQ_ERR_NULL;
        if ((reinterpret_cast<uintptr_t>(data) & 15u) != 0) return BFQ_ERR_ALIGN;
        const int64_t width = transposed ? rows : k;  // elements of a stored row in use
        if (ld < width) return BFQ_ERR_STRIDE;
        const int ebits = kind == BFQ_OP_F32 ? 32 : (kind == BFQ_OP_BF16 ? 16 : kind);
        if ((ld * ebits) % 128 != 0) return BFQ_ERR_STRIDE;  // stored rows start on 16-byte boundaries
        return BFQ_OK;
    };
    int rc = check(a, a_kind, a_transposed, lda, a_scales, m);
    if (rc == BFQ_OK) rc = check(b, b_kind, b_transposed, ldb, b_scales, n);
    if (rc != BFQ_OK) return rc;
    if (ldc < n || (reinterpret_cast<uintptr_t>(c) & 3u) != 0) return BFQ_ERR_STRIDE;
    const size_t wanted = workspace != nullptr ? bfq_dequant_gemm_workspace(plan, m, n, k, a_kind, a_transposed, b_kind, b_transposed) : 0;
    if (workspace != nullptr && (reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return BFQ_ERR_ALIGN;
    if (workspace != nullptr && workspace_bytes < wanted) return BFQ_ERR_WORKSPACE;
    int prev = -1;
    if (cudaGetDevice(&prev) != cudaSuccess) return BFQ_ERR_CUDA;
    if (prev != plan->device && cudaSetDevice(plan->device) != cudaSuccess) return BFQ_ERR_CUDA;
    cudaError_t e = cudaSuccess;
    const Operand u = make_operand(b, b_scales, ldb, b_kind, b_transposed, int(n), a_kind);
    const Operand v = make_operand(a, a_scales, lda, a_kind, a_transposed, int(m), b_kind);
    if (k == 0) {
        e = cudaMemset2DAsync(c, size_t(ldc) * 4, 0, size_t(n) * 4, size_t(m), static_cast<cudaStream_t>(stream));
    } else if (use_few_rows(u, v, k)) {
        cudaStream_t st = static_cast<cudaStream_t>(stream);
        e = b_kind == BFQ_OP_CODES2 ? launch_few<BFQ_OP_CODES2>(u, v, c, ldc, int(k), alpha, st)
            : b_kind == BFQ_OP_CODES4 ? launch_few<BFQ_OP_CODES4>(u, v, c, ldc, int(k), alpha, st)
                                      : launch_few<BFQ_OP_CODES8>(u, v, c, ldc, int(k), alpha, st);
    } else {
        constexpr size_t smem = size_t(kBarsOff) + 8 * (2 * kMaxStages + 4) + 16 + 1024;
        static bool attr_set[bfq::kMaxDevices] = {false};
        if (!attr_set[plan->device]) {
            e = cudaFuncSetAttribute(k_dequant_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
            attr_set[plan->device] = (e == cudaSuccess);
        }
        if (e == cudaSuccess) {
            Params p{};
            p.u = u, p.v = v;
            if (wanted > 0) {
                uint8_t* at = static_cast<uint8_t*>(workspace);
                e = split_operand(p.u, v, k, &at, static_cast<cudaStream_t>(stream));
                if (e == cudaSuccess) e = split_operand(p.v, u, k, &at, static_cast<cudaStream_t>(stream));
            }
            p.c = c, p.ldc = ldc, p.k = int(k), p.alpha = alpha, p.status = plan->status_word;
            // Two code operands along K are an integer product: exact in 32 bits up to K = 2^17 - 1 (codes left in place are at
            // most 128 in size), at twice the rate of the bf16 products.
            p.int8 = is_codes(a_kind) && is_codes(b_kind) && !a_transposed && !b_transposed && k < (1 << 17);
            p.unit = 1.f / float(1 << (code_shift(a_kind) + code_shift(b_kind)));
            p.kblocks = p.int8 ? int((k + 2 * kKB - 1) / (2 * kKB)) : int(k / kKB);
            const Shape shape = choose_shape(m, n, p.kblocks, p.u.terms * p.v.terms,
                                             is_codes(a_kind) && a_transposed ? (a_kind == BFQ_OP_CODES8 ? 32 : 256 / a_kind) : 32,
                                             plan->sm_count);
            p.nt = shape.nt, p.tiles_v = shape.tiles_v, p.tiles = shape.tiles, p.split = shape.split;
            CUtensorMap map_u{}, map_v{}, map_u_lo{}, map_v_lo{};
            auto encode = [&](CUtensorMap* map, CUtensorMap* map_lo, Operand op, int box_rows) {
                if (op.kind != BFQ_OP_BF16) return true;
                if (!encode_operand(map, op, k, box_rows)) return false;
                op.data = op.lo;
                return op.terms == 1 || encode_operand(map_lo, op, k, box_rows);
            };
            const bool ok = encode(&map_u, &map_u_lo, p.u, kRows) && encode(&map_v, &map_v_lo, p.v, p.nt / 2);
            if (e == cudaSuccess)
                e = ok ? launch(p, map_u, map_v, map_u_lo, map_v_lo, plan->sm_count, smem, static_cast<cudaStream_t>(stream)) : cudaErrorInvalidValue;
        }
    }
    if (prev != plan->device) cudaSetDevice(prev);
    if (e != cudaSuccess) {
        plan->last_cuda_error = static_cast<int>(e);
        return BFQ_ERR_CUDA;
    }
    return BFQ_OK;
}
