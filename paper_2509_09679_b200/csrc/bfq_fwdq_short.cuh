// Forward of rows of n = 4096 >> SUB elements, 2^SUB rows as one of 4096 (see SUB at the kernel); one source file per n.
#pragma once
#include <type_traits>

#include "bfq_fast.h"
#include "bfq_generic.cuh"
#include "bfq_n4096.cuh"
#include "bfq_fwdq4096.cuh"

namespace bfq {

template <int SUB>
static cudaError_t fwdq_short_launch(const bfq_plan* plan, const void* x, bool f32, int64_t rows, int64_t ldx, int bits, uint8_t* codes,
                                     uint16_t* scales, void* y, cudaStream_t st) {
    constexpr int n = f4k::kN >> SUB;
    CUtensorMap tmap;
    if (!(f32 ? encode_row_map_f32(&tmap, x, rows, ldx, n) : encode_row_map(&tmap, x, rows, ldx, n))) return cudaErrorInvalidValue;
    const int64_t elems = rows * n, joint = (elems + f4k::kN - 1) / f4k::kN;
    const int type = f32 ? kF32 : kBF16;
    const Again again{x, ldx, type, plan->tw, false, 12 - SUB, elems, bits, y, type, codes, scales};
    using namespace f4k;
    auto go = [&](auto out, auto in_f32) {
        return launch_variant<4, 32, 2, kButterfly, decltype(out)::value, false, decltype(in_f32)::value, SUB>(plan, tmap, joint, codes, scales, y,
                                                                                                    kN, st, nullptr, elems, again);
    };
    if (f32) {
        const std::true_type in{};
        if (bits == 0) return go(std::integral_constant<int, kOutF32>(), in);
        if (bits == 2) return go(std::integral_constant<int, kOutInt2>(), in);
        if (bits == 4) return go(std::integral_constant<int, kOutInt4>(), in);
        return go(std::integral_constant<int, kOutInt8>(), in);
    }
    const std::false_type in{};
    if (bits == 0) return go(std::integral_constant<int, kOutBf16>(), in);
    if (bits == 2) return go(std::integral_constant<int, kOutInt2>(), in);
    if (bits == 4) return go(std::integral_constant<int, kOutInt4>(), in);
    return go(std::integral_constant<int, kOutInt8>(), in);
}

}  // namespace bfq
