// Short rows (128 .. 2048 elements) a second time, as the kernels for every n compute them.  The kernels that take several
// short rows as one of 4096 keep each value divided by a product of cosines (down to 2^-64), so a row with values from 2^56
// on may overflow there although its result does not; and what they make of infinities and NaN is not what the rotation by
// cos and sin makes of them.  Either shows as a result that is not finite.  A thread that meets one raises its group's flag;
// a group whose flag is up looks through its rows once all are written and does the ones in question again from their input,
// one stage at a time in shared memory (a few microseconds a row: not meant to be met often).  Whether a row is done again
// depends on the row alone.
#pragma once

#include "bfq_generic.cuh"
#include "bfq_n4096.cuh"

namespace bfq {

// the call's input rows, row stride ld, and the plan's (cos, sin): what the kernels do not have anyway
struct RowSource {
    const void* x;
    int64_t ld;
    const float2* tw;
};
struct Never {};  // in the place of Again: kernels that never do a row again

struct Again {
    RowSource from;
    int xtype;
    bool inverse;
    int levels;     // log2 of the row length
    int64_t elems;  // elements of all rows
    int bits;       // 0: rows out only; else codes and scales
    void* y;        // rows of ytype out, row stride ldy, or null
    int64_t ldy;
    int ytype;
    uint8_t* codes;
    uint16_t* scales;
};

namespace f4k {

// magnitudes from this bit pattern on are no finite result: infinity and NaN, or what rounds to infinity in bf16
__host__ __device__ constexpr uint32_t not_finite(bool bf16) { return bf16 ? 0x7F7F8000u : 0x7F800000u; }

// max of |a|, |b| and m >= 0; NaN if one of them is
__device__ __forceinline__ float max_abs_nan(float m, float a, float b) {
    float r;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(m), "f"(a), "f"(b));
    return r;
}

// The largest magnitude among the thread's elements in registers m with (m & SKIP) == 0, NaN if there is one.  The inverse's last
// stage multiplies the factors out, so that an infinity or NaN in either element of a pair is in both results: it looks at one of
// them.  The forward's last stage may overflow in one element alone.
template <int SKIP>
__device__ __forceinline__ float largest(const u64 (&P)[16]) {
    float r[2] = {0.f, 0.f};
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        if ((m & SKIP) != 0) continue;
        float a, b;
        unpack2(P[m], a, b);
        float& chain = r[((m / 2 + m / 4) ^ m) & 1];
        chain = max_abs_nan(chain, a, b);
    }
    return max_abs_nan(r[0], r[1], 0.f);
}

// whether `yes` holds for any of the group's threads
__device__ __forceinline__ bool group_any(int bar, bool yes) {
    uint32_t r;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, %2, %3, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                 : "=r"(r)
                 : "r"(static_cast<uint32_t>(yes)), "r"(bar), "n"(kGroupThreads)
                 : "memory");
    return r != 0u;
}

// Row `row` by the 128 threads t of a group with named barrier `bar`; `buf`: the group's own shared memory, four floats more
// than a row.  What the group has stored for the row before is overwritten.
__device__ __forceinline__ void row_again(const Again& p, int64_t row, uint32_t buf, int bar, int t) {
    const int n = 1 << p.levels, half = n >> 1;
    bar_sync(bar, kGroupThreads);  // nobody uses the buffer any more
    for (int e = t; e < n; e += kGroupThreads) {
        const int64_t at = row * p.from.ld + e;
        const float v = p.xtype == kF32 ? static_cast<const float*>(p.from.x)[at] : __bfloat162float(static_cast<const __nv_bfloat16*>(p.from.x)[at]);
        sts32(buf + 4 * e, __float_as_uint(v));
    }
    bar_sync(bar, kGroupThreads);
    for (int i = 0; i < p.levels; ++i) {
        const int s = p.inverse ? p.levels - 1 - i : i;
        for (int j = t; j < half; j += kGroupThreads) {
            const uint32_t lo = buf + 4 * (((j >> s) << (s + 1)) | (j & ((1 << s) - 1))), hi = lo + (4u << s);
            const float2 cs = load_plain(p.from.tw + s * half + j);
            const float a = __uint_as_float(lds32(lo)), b = __uint_as_float(lds32(hi));
            sts32(lo, __float_as_uint(p.inverse ? cs.x * a + cs.y * b : cs.x * a - cs.y * b));
            sts32(hi, __float_as_uint(p.inverse ? cs.x * b - cs.y * a : cs.y * a + cs.x * b));
        }
        bar_sync(bar, kGroupThreads);
    }
    auto value = [&](int e) { return __uint_as_float(lds32(buf + 4 * e)); };
    if (p.y != nullptr) {
        for (int e = t; e < n; e += kGroupThreads) {
            if (p.ytype == kF32) static_cast<float*>(p.y)[row * p.ldy + e] = value(e);
            else static_cast<__nv_bfloat16*>(p.y)[row * p.ldy + e] = __float2bfloat16_rn(value(e));
        }
    }
    if (p.bits == 0) return;
    float m = 0.f;
    for (int e = t; e < n; e += kGroupThreads) m = fmaxf(m, fabsf(value(e)));  // drops NaN
    const uint32_t wmax = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(m));
    if ((t & 31) == 0) sts32(buf + 4 * (n + (t >> 5)), wmax);
    bar_sync(bar, kGroupThreads);
    const uint4 o = lds128(buf + 4 * n);
    const int qmax = (1 << (p.bits - 1)) - 1, per = 8 / p.bits;
    float inv;
    const uint16_t s16 = row_scale(__uint_as_float(max(max(o.x, o.y), max(o.z, o.w))), qmax, &inv);
    if (t == 0) p.scales[row] = s16;
    for (int b = t; b < n / per; b += kGroupThreads) {
        uint32_t byte = 0;
        for (int e = 0; e < per; ++e) byte |= (static_cast<uint32_t>(quant1(value(b * per + e), inv, -qmax - 1, qmax)) & ((1u << p.bits) - 1u)) << (p.bits * e);
        p.codes[row * (n / per) + b] = static_cast<uint8_t>(byte);
    }
}

// The group's joint rows first, first + stride, ...: those of their rows that are not finite (in the elements that `largest`
// looks at: in the inverse the lower ones of the last stage's pairs).  A quantized row of that kind has a NaN for its scale
// (row_scale_fast of an infinite or NaN maximum; no finite row has).
static __device__ __noinline__ void rows_again(const Again& p, int first, int stride, int count, uint32_t buf, int bar, int t) {
    const int n = 1 << p.levels, upper = p.inverse ? 1 : 0;
    for (int k = 0; k < count; ++k) {
        int64_t row = (static_cast<int64_t>(first) + static_cast<int64_t>(k) * stride) << (12 - p.levels);
        for (const int64_t end = row + (4096 >> p.levels); row < end && (row << p.levels) < p.elems; ++row) {
            bool bad = false;
            if (p.bits != 0) {
                bad = *reinterpret_cast<volatile const uint16_t*>(p.scales + row) > 0x7C00u;
            } else {
                for (int e = t; e < n; e += kGroupThreads) {
                    if ((e & upper) != 0) continue;
                    if (p.ytype == kF32) bad |= (*reinterpret_cast<volatile const uint32_t*>(static_cast<float*>(p.y) + row * p.ldy + e) & 0x7F800000u) == 0x7F800000u;
                    else bad |= (*reinterpret_cast<volatile const uint16_t*>(static_cast<__nv_bfloat16*>(p.y) + row * p.ldy + e) & 0x7F80u) == 0x7F80u;
                }
            }
            if (group_any(bar, bad)) row_again(p, row, buf, bar, t);
        }
    }
}

}  // namespace f4k
}  // namespace bfq
