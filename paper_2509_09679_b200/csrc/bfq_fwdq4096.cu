// Tuned forward for n = 4096 bf16 rows on sm_100a: learned butterfly or fixed Walsh-Hadamard rotation, fused with
// INT4 quantization or writing the rotated rows in bf16.  The description below is the butterfly + INT4 case.
//
// Design (one persistent CTA per SM, G row groups of 128 threads):
//  * A row is owned by one group of four warps, one warp per scheduler and per tensor-memory lane
//    quarter.  The 12 stages run as three phases of four stages.  In each phase a thread holds 32
//    elements of the row as 16 packed fp32x2 registers: four index bits are the phase's stage bits
//    (so all partners are in the thread's own registers) and the fifth selects the half of the
//    packed register and is never a stage bit of that phase, so every rotation is a packed FMA.
//        phase 1: stage bits 0-3, packed along bit 8     (two runs of 16 consecutive elements)
//        phase 2: stage bits 4-7, packed along bit 8
//        phase 3: stage bits 8-11, packed along bit 0    (adjacent elements -> one code byte)
//    Between phases the row is regrouped through shared memory.  The first regrouping swaps bits
//    0-3 with bits 4-7 among the 16 lanes of a half-warp: 64-bit stores and loads of whole packed
//    registers and a warp-level sync only.  The second crosses warps: scalar stores, 64-bit loads,
//    one named barrier.  The buffer layouts are additive in the index bits (padded, not
//    XOR-swizzled) so that every access is base + immediate and bank-conflict free.
//  * Rotations use the scaled form  lo' = lo + k1*hi, hi' = hi + k2*lo  (two independent FMAs and two constants
//    per pair): every element carries an implicit factor d, the product of the cosines of the rotations it has
//    been through, which the table build folds into k1, k2 and into the general 2x2 of the last stage, so the
//    kernel sees only constants.  The form is singular where a cosine vanishes; when some element's factor leaves
//    [2^-64, 1] the table build raises a flag and the kernel takes the three-shear (lifting) form instead:
//    a += -t*b; b += s*a; a += -t*b  with t = tan(phi/2), s = sin(phi), three FMAs per pair, angles reduced to
//    |phi| <= pi/2 (so |t| <= 1), the sign flips of the reduction tracked per element at table-build time.  Both
//    images have the same layout.
//  * The constants (416 words per thread role, 53248 in all) live in tensor memory, one strip per
//    lane; every group reads the same strips.  They are streamed into registers with tcgen05.ld,
//    one chunk ahead of use.
//  * Rows arrive by TMA (128-byte swizzled tiles, two-deep ring per group, mbarrier completion).
//    The per-row absmax is a warp reduction plus one step across the group's four warps; INT4
//    codes are produced with the magic-number rounding trick, one byte per packed register.
#include "bfq_fwdq4096.cuh"

namespace bfq {
namespace f4k {

// ---- table preparation -----------------------------------------------------------------------------------
// Step 1 (one thread per angle of the 4096-element transform; rows of n = 2^levels < 4096 elements: the angles of 4096 / n
// rows side by side, stages from log2 n on the identity): the generic (cos, sin) table entry, cos and sin in double for step 2, the
// reduced-angle lifting constants and whether the reduction negates the pair.  The pair is negated iff
// cos(theta) < 0, and phi = theta -+ pi in that case; tan(phi/2) and sin(phi) are odd in phi, so the constants for
// the mirrored rotation G(-theta) are the negatives of the stored ones.
__global__ void __launch_bounds__(256) k_prep_angles4096(const float* theta, float2* __restrict__ tw,
                                                          float4* __restrict__ prep, uint8_t* __restrict__ flip,
                                                          double2* __restrict__ cs, int* __restrict__ form, int levels) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    grid_dep_launch();
    grid_dep_wait();
    // step 2 raises the first word when the scaled form is out of range, and the fourth (backward); the build of the reverse
    // walk the second
    if (k == 0) form[0] = kFormScaled, form[1] = kFormScaled, form[3] = kFormScaled;
    if (k >= 12 * (kN / 2)) return;
    const int s = k / (kN / 2), j = k % (kN / 2), half = 1 << (levels - 1);
    const int src = s * half + (j & (half - 1));
    const double th = s < levels ? static_cast<double>(theta[src]) : 0.0;
    double sn, c;
    sincos(th, &sn, &c);
    if (s < levels && j < half) tw[src] = make_float2(static_cast<float>(c), static_cast<float>(sn));
    cs[k] = make_double2(c, sn);
    // phi = theta -+ pi when cos(theta) < 0 (|phi| <= pi/2 then): sin(phi) = -sin(theta), cos(phi) = -cos(theta), and
    // tan(phi/2) = sin(phi) / (1 + cos(phi)) with a denominator >= 1: no second reduction, no tan
    const bool f = c < 0.0;
    const double sp = f ? -sn : sn, cp = f ? -c : c;
    flip[k] = f ? 1 : 0;
    prep[k] = make_float4(static_cast<float>(-sp / (1.0 + cp)), static_cast<float>(sp), static_cast<float>(c),
                          static_cast<float>(sn));
}

// Step 2 (one thread per angle): build_image_fwd in bfq_n4096.cuh
__global__ void __launch_bounds__(256) k_build_image4096(const float4* prep, const double2* cs,
                                                          float* __restrict__ img, int* __restrict__ form, float* __restrict__ weight, float* __restrict__ flat) {
    grid_dep_launch();
    grid_dep_wait();
    build_image_fwd(blockIdx.x * blockDim.x + threadIdx.x, prep, cs, img, form, weight, flat);
}

}  // namespace f4k

// ---- host side ---------------------------------------------------------------------------------------------
// two images: scaled form, three-shear form
size_t fwdq4096_image_bytes() { return size_t(2) * 128 * f4k::kCols * sizeof(float); }
// per angle: float4 (three-shear constants, cos, sin), double2 (cos, sin), one negation flag
size_t fwdq4096_prep_bytes() { return size_t(12) * (f4k::kN / 2) * (sizeof(float4) + sizeof(double2) + 1); }

// The generic (cos, sin) table and the staging entries of every image (one launch).
static cudaError_t fwdq4096_prep_angles(const bfq_plan* plan, const float* theta, cudaStream_t st) {
    const int count = 12 * (f4k::kN / 2);
    float4* prep = reinterpret_cast<float4*>(plan->prep4096);
    double2* cs = reinterpret_cast<double2*>(prep + count);
    uint8_t* flip = reinterpret_cast<uint8_t*>(cs + count);
    return launch_overlapped(f4k::k_prep_angles4096, dim3((count + 255) / 256), dim3(256), 0, st, theta, plan->tw, prep, flip, cs,
                             plan->form_flag, plan->log_n);
}

// That and the tensor-memory image of the forward kernels (two launches).  Rows shorter than 4096: the second launch builds the
// reverse tables too, so that later calls on any stream find all tables built here (with a third launch for them bfq_set_angles took
// 7.7 us on the GPU, now 5.4; the table of the kernels for every n
// alone takes 3.1 - 3.6).
cudaError_t fwdq4096_set_angles(const bfq_plan* plan, const float* theta, cudaStream_t st) {
    if (plan->n == f4k::kN) return fwdq4096_build_forward(plan, theta, st);
    const cudaError_t e = fwdq4096_prep_angles(plan, theta, st);
    return e == cudaSuccess ? bwd4096_build_tables(plan, st, true) : e;
}

// the forward tables alone, which are the backward kernel's too
cudaError_t fwdq4096_build_forward(const bfq_plan* plan, const float* theta, cudaStream_t st) {
    const int count = 12 * (f4k::kN / 2);
    const cudaError_t e = fwdq4096_prep_angles(plan, theta, st);
    if (e != cudaSuccess) return e;
    float4* prep = reinterpret_cast<float4*>(plan->prep4096);
    double2* cs = reinterpret_cast<double2*>(prep + count);
    return launch_overlapped(f4k::k_build_image4096, dim3((count + 255) / 256), dim3(256), 0, st, prep, cs, plan->img4096,
                             plan->form_flag, plan->weight4096, plan->flat4096);
}

// rows of 128 .. 2048 elements: several as one of 4096.  bits = 0: the rotated rows, in the type of x.
bool fwdq_short_available(const bfq_plan* plan) {
    return plan->n >= 128 && plan->n < f4k::kN && plan->cc_major == 10 && plan->img4096 != nullptr && encode_tiled() != nullptr;
}
cudaError_t fwdq_short_launch(const bfq_plan* plan, const void* x, bool f32, int64_t rows, int64_t ldx, int bits, uint8_t* codes,
                              uint16_t* scales, void* y, int64_t ldy, cudaStream_t st) {
    switch (plan->n) {
        case 128: return fwdq128_launch(plan, x, f32, rows, ldx, bits, codes, scales, y, ldy, st);
        case 256: return fwdq256_launch(plan, x, f32, rows, ldx, bits, codes, scales, y, ldy, st);
        case 512: return fwdq512_launch(plan, x, f32, rows, ldx, bits, codes, scales, y, ldy, st);
        case 1024: return fwdq1024_launch(plan, x, f32, rows, ldx, bits, codes, scales, y, ldy, st);
        case 2048: return fwdq2048_launch(plan, x, f32, rows, ldx, bits, codes, scales, y, ldy, st);
        default: return cudaErrorInvalidValue;
    }
}

bool fwdq4096_available(const bfq_plan* plan) {
    return plan->n == f4k::kN && plan->cc_major == 10 && plan->img4096 != nullptr && encode_tiled() != nullptr;
}

// Four row groups per CTA, 32-word constant chunks, one buffer per regrouping (measured fastest among the
// configurations that compile without spills; more groups did not help).
// hadamard: the fixed Walsh-Hadamard transform instead of the plan's butterfly.  y != nullptr: write the rotated
// rows in bf16 instead of INT4 codes + scales.
cudaError_t fwdq4096_launch(const bfq_plan* plan, const void* x, int64_t rows, int64_t ldx, bool hadamard,
                            uint8_t* codes, uint16_t* scales, void* y, int64_t ldy, cudaStream_t st) {
    CUtensorMap tmap;
    if (!encode_row_map(&tmap, x, rows, ldx)) return cudaErrorInvalidValue;
    using namespace f4k;
    if (!hadamard) {
        return y == nullptr ? launch_variant<4, 32, 2, kButterfly, kOutInt4>(plan, tmap, rows, codes, scales, y, ldy, st)
                            : launch_variant<4, 32, 2, kButterfly, kOutBf16>(plan, tmap, rows, codes, scales, y, ldy, st);
    }
    return y == nullptr ? launch_variant<4, 32, 2, kHadamard, kOutInt4>(plan, tmap, rows, codes, scales, y, ldy, st)
                        : launch_variant<4, 32, 2, kHadamard, kOutBf16>(plan, tmap, rows, codes, scales, y, ldy, st);
}

// INT2 / INT8 codes: same kernel, other packing in the epilogue
cudaError_t fwdq4096_launch_bits(const bfq_plan* plan, const void* x, int64_t rows, int64_t ldx, bool hadamard, int bits,
                                 uint8_t* codes, uint16_t* scales, cudaStream_t st) {
    CUtensorMap tmap;
    if (!encode_row_map(&tmap, x, rows, ldx)) return cudaErrorInvalidValue;
    using namespace f4k;
    if (hadamard) {
        return bits == 2 ? launch_variant<4, 32, 2, kHadamard, kOutInt2>(plan, tmap, rows, codes, scales, nullptr, 0, st)
                         : launch_variant<4, 32, 2, kHadamard, kOutInt8>(plan, tmap, rows, codes, scales, nullptr, 0, st);
    }
    return bits == 2 ? launch_variant<4, 32, 2, kButterfly, kOutInt2>(plan, tmap, rows, codes, scales, nullptr, 0, st)
                     : launch_variant<4, 32, 2, kButterfly, kOutInt8>(plan, tmap, rows, codes, scales, nullptr, 0, st);
}

// weight folding that keeps the rotated rows: codes + scales and W Q^T in bf16 (leading dimension ldy) from one pass
cudaError_t fwdq4096_launch_codes_rows(const bfq_plan* plan, const void* x, int64_t rows, int64_t ldx, int bits,
                                       uint8_t* codes, uint16_t* scales, void* y, int64_t ldy, cudaStream_t st) {
    CUtensorMap tmap;
    if (!encode_row_map(&tmap, x, rows, ldx)) return cudaErrorInvalidValue;
    using namespace f4k;
    if (bits == 4) return launch_variant<4, 32, 2, kButterfly, kOutInt4, true>(plan, tmap, rows, codes, scales, y, ldy, st);
    if (bits == 2) return launch_variant<4, 32, 2, kButterfly, kOutInt2, true>(plan, tmap, rows, codes, scales, y, ldy, st);
    return launch_variant<4, 32, 2, kButterfly, kOutInt8, true>(plan, tmap, rows, codes, scales, y, ldy, st);
}

// fp32 rows in: codes + scales (bits = 2, 4, 8), or the rotated rows in fp32 (bits = 0, y with leading dimension ldy)
cudaError_t fwdq4096_launch_f32(const bfq_plan* plan, const void* x, int64_t rows, int64_t ldx, int bits, uint8_t* codes,
                                uint16_t* scales, void* y, int64_t ldy, cudaStream_t st) {
    CUtensorMap tmap;
    if (!encode_row_map_f32(&tmap, x, rows, ldx)) return cudaErrorInvalidValue;
    using namespace f4k;
    if (bits == 0) return launch_variant<4, 32, 2, kButterfly, kOutF32, false, true>(plan, tmap, rows, codes, scales, y, ldy, st);
    if (bits == 4) return launch_variant<4, 32, 2, kButterfly, kOutInt4, false, true>(plan, tmap, rows, codes, scales, nullptr, 0, st);
    if (bits == 2) return launch_variant<4, 32, 2, kButterfly, kOutInt2, false, true>(plan, tmap, rows, codes, scales, nullptr, 0, st);
    return launch_variant<4, 32, 2, kButterfly, kOutInt8, false, true>(plan, tmap, rows, codes, scales, nullptr, 0, st);
}

// bfq_forward_quant_stats on the tuned path: codes + scales + row moments + code counts from one launch of k_fwdq4096
// (hist must have been zeroed on the same stream).
cudaError_t fwdq4096_launch_stats(const bfq_plan* plan, const void* x, int64_t rows, int64_t ldx, uint8_t* codes,
                                  uint16_t* scales, unsigned long long* hist, float* rowstats, cudaStream_t st) {
    CUtensorMap tmap;
    if (!encode_row_map(&tmap, x, rows, ldx)) return cudaErrorInvalidValue;
    using namespace f4k;
    return launch_variant<4, 32, 2, kButterfly, kOutInt4Stats>(plan, tmap, rows, codes, scales, rowstats, 0, st, hist);
}

}  // namespace bfq
