// Entry points of the tuned kernels (host side), called by the C-ABI layer.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "bfq_plan.h"

namespace bfq {

// n = 4096, bf16 rows, INT4: tensor-memory-resident rotation constants
bool fwdq4096_available(const bfq_plan* plan);
size_t fwdq4096_image_bytes();
size_t fwdq4096_prep_bytes();
// builds the plan's (cos, sin) table and the tensor-memory image from the angles
cudaError_t fwdq4096_set_angles(const bfq_plan* plan, const float* theta, cudaStream_t st);
cudaError_t fwdq4096_launch(const bfq_plan* plan, const void* x, int64_t rows, int64_t ldx, bool hadamard,
                            uint8_t* codes, uint16_t* scales, void* y_bf16, int64_t ldy, cudaStream_t st);

// INT2 / INT8 codes from the same kernel (bits = 2 or 8)
cudaError_t fwdq4096_launch_bits(const bfq_plan* plan, const void* x, int64_t rows, int64_t ldx, bool hadamard, int bits,
                                 uint8_t* codes, uint16_t* scales, cudaStream_t st);
// codes + scales (bits = 2, 4, 8) and the rotated rows in bf16 from one pass
cudaError_t fwdq4096_launch_codes_rows(const bfq_plan* plan, const void* x, int64_t rows, int64_t ldx, int bits,
                                       uint8_t* codes, uint16_t* scales, void* y_bf16, int64_t ldy, cudaStream_t st);
// fp32 rows in: codes + scales (bits = 2, 4, 8) or, with bits = 0, the rotated rows in fp32
cudaError_t fwdq4096_launch_f32(const bfq_plan* plan, const void* x, int64_t rows, int64_t ldx, int bits, uint8_t* codes,
                                uint16_t* scales, void* y_f32, int64_t ldy, cudaStream_t st);
// the same with the statistics of bfq_forward_quant_stats (hist already zeroed on `st`)
cudaError_t fwdq4096_launch_stats(const bfq_plan* plan, const void* x, int64_t rows, int64_t ldx, uint8_t* codes,
                                  uint16_t* scales, unsigned long long* hist, float* rowstats, cudaStream_t st);

// a few rows of n = 4096, a row to a cluster; bits as in fwdq_short_launch
bool forward_few_available(const bfq_plan* plan, int64_t rows);
cudaError_t forward_few_launch(const bfq_plan* plan, const void* x, bool f32, int64_t rows, int64_t ldx, int bits, uint8_t* codes, uint16_t* scales, void* y,
                               int64_t ldy, cudaStream_t st);

cudaError_t fwdq4096_build_forward(const bfq_plan* plan, const float* theta, cudaStream_t st);
// rows of 128 .. 2048 elements: several as one of 4096 on the same kernel.  bits = 2, 4, 8: codes + scales, and
// the rows if y is not null; bits = 0: the rows alone.  Rows are in the type of x, ldy apart (beside codes: contiguous)
bool fwdq_short_available(const bfq_plan* plan);
cudaError_t fwdq_short_launch(const bfq_plan* plan, const void* x, bool f32, int64_t rows, int64_t ldx, int bits, uint8_t* codes,
                              uint16_t* scales, void* y, int64_t ldy, cudaStream_t st);
cudaError_t fwdq128_launch(const bfq_plan* plan, const void* x, bool f32, int64_t rows, int64_t ldx, int bits, uint8_t* codes, uint16_t* scales,
                           void* y, int64_t ldy, cudaStream_t st);
cudaError_t fwdq256_launch(const bfq_plan* plan, const void* x, bool f32, int64_t rows, int64_t ldx, int bits, uint8_t* codes, uint16_t* scales,
                           void* y, int64_t ldy, cudaStream_t st);
cudaError_t fwdq512_launch(const bfq_plan* plan, const void* x, bool f32, int64_t rows, int64_t ldx, int bits, uint8_t* codes, uint16_t* scales,
                           void* y, int64_t ldy, cudaStream_t st);
cudaError_t fwdq1024_launch(const bfq_plan* plan, const void* x, bool f32, int64_t rows, int64_t ldx, int bits, uint8_t* codes, uint16_t* scales,
                           void* y, int64_t ldy, cudaStream_t st);
cudaError_t fwdq2048_launch(const bfq_plan* plan, const void* x, bool f32, int64_t rows, int64_t ldx, int bits, uint8_t* codes, uint16_t* scales,
                           void* y, int64_t ldy, cudaStream_t st);
// the same rows inverse
bool inv_short_available(const bfq_plan* plan);
cudaError_t inv_short_launch(bfq_plan* plan, const void* y, bool y_f32, int64_t rows, int64_t ldy, void* x, bool x_bf16, int64_t ldx, cudaStream_t st);

// n = 8192, bf16 rows, INT2 (INT4 / INT8 through another epilogue): two-CTA clusters, one 4096-point half per CTA
size_t fwdq8192_image_bytes();
size_t fwdq8192_prep_bytes();
bool fwdq8192_available(const bfq_plan* plan);
cudaError_t fwdq8192_set_angles(const bfq_plan* plan, const float* theta, cudaStream_t st);
cudaError_t fwdq8192_launch(const bfq_plan* plan, const void* x, int64_t rows, int64_t ldx, int bits, uint8_t* codes,
                            uint16_t* scales, cudaStream_t st);
cudaError_t fwdq8192_launch_codes_rows(const bfq_plan* plan, const void* x, int64_t rows, int64_t ldx, int bits,
                                       uint8_t* codes, uint16_t* scales, void* y_bf16, int64_t ldy, cudaStream_t st);
cudaError_t fwdq8192_launch_f32(const bfq_plan* plan, const void* x, int64_t rows, int64_t ldx, int bits, uint8_t* codes,
                                uint16_t* scales, void* y_f32, int64_t ldy, cudaStream_t st);
cudaError_t fwdq8192_launch_hadamard(const bfq_plan* plan, const void* x, int64_t rows, int64_t ldx, int bits, uint8_t* codes,
                                     uint16_t* scales, void* y_bf16, int64_t ldy, cudaStream_t st);
cudaError_t fwdq8192_launch_bf16(const bfq_plan* plan, const void* x, int64_t rows, int64_t ldx, void* y, int64_t ldy,
                                 cudaStream_t st);

// rows of 128 .. 4096 elements (below 4096: contiguous, several as one row), x, g and dx all bf16 or all fp32: backward with
// tensor-memory constants and accumulators, from the tables of the forward kernel.  takes_short_backward: whether bfq_backward
// (and bfq_backward_noalloc, whose dx are the same bits) hands a call with n < 4096 to grad4096_launch
bool takes_short_backward(int n, int xt, int gt, bool want_dx, int dxt, int64_t rows, int64_t ld);
size_t grad4096_weight_bytes();
size_t grad4096_partial_floats(int ctas);
bool grad4096_available(const bfq_plan* plan);
cudaError_t grad4096_prepare(int device);
cudaError_t grad4096_launch(bfq_plan* plan, const void* x, const void* g, int64_t rows, int64_t ld, void* dx, float* dtheta, bool f32, cudaStream_t st);

// tables of the inverse, and (dsign) of the backward of the halves of n = 8192
size_t bwd4096_image_bytes();
size_t inv4096_image_bytes();
size_t bwd4096_dsign_bytes();
size_t bwd4096_gsign_bytes();
bool bwd4096_available(const bfq_plan* plan);
// n = 8192 bf16 rows: the n = 4096 backward kernel on the two halves of the elements (one launch, even CTAs on the lower half, odd CTAs on the upper); the
// stage that joins the halves is folded into the read of g and its sums are taken there too
size_t bwd8192_prep_bytes();
size_t bwd8192_partial_floats(int sm_count);
bool bwd8192_available(const bfq_plan* plan);
cudaError_t bwd8192_build_tables(const bfq_plan* plan, cudaStream_t st);
cudaError_t inv8192_launch(bfq_plan* plan, const void* y, int64_t rows, int64_t ldy, void* x, bool x_bf16, int64_t ldx,
                           cudaStream_t st);
cudaError_t bwd8192_launch_halves(bfq_plan* plan, const void* x, const void* g, int64_t rows, int64_t ld, void* dx,
                                  float* dtheta, cudaStream_t st);
cudaError_t bwd4096_build_tables(const bfq_plan* plan, cudaStream_t st, bool forward_too = false);  // forward_too: img4096 as well

// n = 4096, bf16 y -> bf16 / fp32 x: inverse (uses the backward tables)
cudaError_t inv4096_launch_f32(bfq_plan* plan, const void* y, int64_t rows, int64_t ldy, void* x, int64_t ldx,
                               cudaStream_t st);
cudaError_t inv4096_launch(bfq_plan* plan, const void* y, int64_t rows, int64_t ldy, void* x, bool x_bf16, int64_t ldx,
                           cudaStream_t st);

// composite transform Q1 (x) Q2 (n1 <= 64, n2 = the plan's n): whole tokens in shared memory (n2 = 128 .. 1024, forward), Cayley
// solve and the kernels for every shape
bool composite_forward_available(const bfq_plan* plan, int n1);
cudaError_t composite_forward_launch(const bfq_plan* plan, const float* q1, int n1, const void* x, int xt, int64_t rows, int64_t ldx, void* y, int yt,
                                     int64_t ldy, int bits, uint8_t* codes, uint16_t* scales, cudaStream_t st);
cudaError_t cayley_launch(const bfq_plan* plan, const float* params, int n1, float* q1, cudaStream_t st);
cudaError_t cayley_backward_launch(const bfq_plan* plan, const float* params, int n1, const float* q1, const float* dq1, float* dparams, cudaStream_t st);
// dx (may be null, type of x), dtheta of Q2 and dQ1 for upstream rows g; ld: row stride of x, g and dx
bool composite_backward_available(const bfq_plan* plan, int n1);
cudaError_t composite_backward_launch(bfq_plan* plan, const float* q1, int n1, const void* x, int xt, const void* g, int gt, int64_t rows,
                                      int64_t ld, void* dx, float* dtheta, float* dq1, cudaStream_t st);
cudaError_t composite_generic_launch(const bfq_plan* plan, const float* q1, int n1, const void* x, int xt, int64_t rows,
                                     int64_t ldx, void* y, int yt, int64_t ldy, int bits, uint8_t* codes,
                                     uint16_t* scales, bool inverse, cudaStream_t st);


// composite 40 x 128 on bf16 rows: butterfly with kernel-parameter constants + tcgen05 TF32 dense factor
bool comp5120_available(const bfq_plan* plan);
size_t comp5120_param_bytes();
cudaError_t comp5120_launch(bfq_plan* plan, const float* q1, const void* x, int64_t rows, int64_t ldx, uint8_t* codes,
                            uint16_t* scales, void* y_bf16, int64_t ldy, cudaStream_t st);


// composite 40 x 128 on bf16 rows with both factors on the tensor cores (Q2 merged into a dense 128 x 128 block)
size_t comp5120d_image_bytes();
bool comp5120d_available(const bfq_plan* plan);
cudaError_t comp5120d_set_angles(const bfq_plan* plan, cudaStream_t st);
cudaError_t comp5120d_launch(bfq_plan* plan, const float* q1, const void* x, int64_t rows, int64_t ldx, int bits,
                             uint8_t* codes, uint16_t* scales, void* y_bf16, int64_t ldy, bool inverse, cudaStream_t st);

}  // namespace bfq
