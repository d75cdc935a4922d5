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
                                     uint16_t* scales, void* y, int64_t ldy, cudaStream_t st) {
    constexpr int n = f4k::kN >> SUB;
    CUtensorMap tmap;
    if (!(f32 ? encode_row_map_f32(&tmap, x, rows, ldx, n) : encode_row_map(&tmap, x, rows, ldx, n))) return cudaErrorInvalidValue;
    const int64_t elems = rows * n, joint = (elems + f4k::kN - 1) / f4k::kN;
    using namespace f4k;
    auto go = [&](auto out, auto in_f32, auto rows_too, auto strided) {
        return launch_variant<4, 32, 2, kButterfly, decltype(out)::value, decltype(rows_too)::value, decltype(in_f32)::value, SUB, decltype(strided)::value>(
            plan, tmap, joint, codes, scales, y, ldy << SUB, st, nullptr, elems, RowSource{x, ldx, plan->tw});
    };
    auto of_type = [&](auto in_f32) {
        constexpr int kRowsOut = decltype(in_f32)::value ? kOutF32 : kOutBf16;
        const std::false_type no{};
        const std::true_type yes{};
        if (bits == 0)
            return ldy == n ? go(std::integral_constant<int, kRowsOut>(), in_f32, no, no) : go(std::integral_constant<int, kRowsOut>(), in_f32, no, yes);
        auto coded = [&](auto rows_too) {
            if (bits == 2) return go(std::integral_constant<int, kOutInt2>(), in_f32, rows_too, no);
            if (bits == 4) return go(std::integral_constant<int, kOutInt4>(), in_f32, rows_too, no);
            return go(std::integral_constant<int, kOutInt8>(), in_f32, rows_too, no);
        };
        return y != nullptr ? coded(yes) : coded(no);
    };
    return f32 ? of_type(std::true_type()) : of_type(std::false_type());
}

}  // namespace bfq
