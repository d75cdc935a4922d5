// Forward of rows of 2048 elements on the n = 4096 kernel.
#include "bfq_fwdq_short.cuh"

namespace bfq {

cudaError_t fwdq2048_launch(const bfq_plan* plan, const void* x, bool f32, int64_t rows, int64_t ldx, int bits, uint8_t* codes, uint16_t* scales,
                           void* y, int64_t ldy, cudaStream_t st) {
    return fwdq_short_launch<1>(plan, x, f32, rows, ldx, bits, codes, scales, y, ldy, st);
}

}  // namespace bfq
