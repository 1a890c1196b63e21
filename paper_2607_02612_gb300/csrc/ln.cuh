// LayerNorm pieces of the exit kernels (Sec. III-D, Eq. 6: the exit head's LayerNorm of the
// CLS row): compensated sums and the output element rounded once to the head's input type.
#pragma once

#include "common.cuh"

namespace fz {

// Neumaier-compensated accumulation: (s, c) carries the sum of every term added
// with an error of a few units in the last place of the result.
__device__ __forceinline__ void neu_add(float &s, float &c, float x) {
    const float t = __fadd_rn(s, x);
    c = __fadd_rn(c, fabsf(s) >= fabsf(x) ? __fadd_rn(__fsub_rn(s, t), x) : __fadd_rn(__fsub_rn(x, t), s));
    s = t;
}

// Packed pairs of float32 (one issue slot each on sm_100 and later), every lane rounded as the scalar form.
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 a, b, r;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tadd.rn.f32x2 r, a, b;\n\t"
        "mov.b64 {%0, %1}, r;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 a, b, r;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmul.rn.f32x2 r, a, b;\n\t"
        "mov.b64 {%0, %1}, r;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 r;
    asm("{\n\t.reg .b64 a, b, c, r;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
        "fma.rn.f32x2 r, a, b, c;\n\tmov.b64 {%0, %1}, r;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return fma2(b, make_float2(-1.0f, -1.0f), a); }
// (s, c) += x in both lanes: the error of every sum by the branch-free two-sum (exact, as neu_add's).
__device__ __forceinline__ void comp_add2(float2 &s, float2 &c, float2 x) {
    const float2 t = add2(s, x), xx = sub2(t, s);
    c = add2(c, add2(sub2(s, sub2(t, xx)), sub2(x, xx)));
    s = t;
}

// u = (x - mean) * rstd * gamma + beta for one element, rounded once to the head's
// input type.  A float32 evaluation is exact enough unless it lands within a few
// float32 ulps of a bf16 rounding midpoint (or beta cancels most of it); then the
// float-float evaluation decides.
__device__ __forceinline__ uint16_t ln_out_bf16(float x, F2 mean, F2 rstd, float g, float b) {
    const float d = __fsub_rn(__fsub_rn(x, mean.hi), mean.lo);
    const float v = __fmul_rn(__fmul_rn(d, rstd.hi), g);
    const float u = __fadd_rn(v, b);
    const uint32_t low = __float_as_uint(u) & 0xFFFFu;
    const uint32_t dist = low > 0x8000u ? low - 0x8000u : 0x8000u - low;
    if (dist > 24u && fabsf(u) >= 0.5f * fabsf(v)) {
        const uint32_t bits = __float_as_uint(u);
        if ((bits & 0x7F800000u) == 0x7F800000u) return (uint16_t)((bits >> 16) | ((bits & 0x7FFFFFu) ? 0x40u : 0u));
        return (uint16_t)((bits + (low > 0x8000u ? 0x8000u : 0u)) >> 16);   // not near a tie: plain rounding
    }
    F2 dd = two_sum(x, -mean.hi);
    dd.lo = __fsub_rn(dd.lo, mean.lo);
    F2 t = f2_mul(quick_two_sum(dd.hi, dd.lo), rstd);
    t = f2_mul(t, {g, 0.0f});
    return f2_to_bf16_bits(f2_add_f(t, b));
}
// A chunk of 8 elements at x (gamma at g, beta at b): the float32 evaluation on packed pairs, rounded by the
// conversion instruction; the elements it does not settle are evaluated in float-float afterwards, in
// one loop per chunk.  Its error is at most 5 ulps of v and half an ulp of u, so 24 ulps of u from a rounding
// midpoint settle it while |u| >= |v| / 2, and 200 while |u| >= |v| / 16: beta cancels half of v in about
// one element of 20, which made nearly every warp go through the float-float form for every element.
__device__ __forceinline__ uint4 ln_chunk_bf16(const __nv_bfloat16 *x, const __nv_bfloat16 *g, const __nv_bfloat16 *b, F2 mean,
                                               F2 rstd) {
    float f[8], gf[8], bf[8];
    chunk_to_f(*reinterpret_cast<const uint4 *>(x), f);
    chunk_to_f(*reinterpret_cast<const uint4 *>(g), gf);
    chunk_to_f(*reinterpret_cast<const uint4 *>(b), bf);
    uint32_t w4[4];
    unsigned left = 0u;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float2 d = sub2(sub2(make_float2(f[2 * q], f[2 * q + 1]), make_float2(mean.hi, mean.hi)), make_float2(mean.lo, mean.lo));
        const float2 v = mul2(mul2(d, make_float2(rstd.hi, rstd.hi)), make_float2(gf[2 * q], gf[2 * q + 1]));
        const float2 u = add2(v, make_float2(bf[2 * q], bf[2 * q + 1]));
        auto open = [](float uu, float vv) {   // (a NaN is not settled)
            const uint32_t low = __float_as_uint(uu) & 0xFFFFu;
            const bool half = fabsf(uu) >= 0.5f * fabsf(vv);
            const uint32_t near = half ? 24u : 200u;
            return low - (0x8000u - near) <= 2u * near || !(fabsf(uu) >= 0.0625f * fabsf(vv));
        };
        left |= (open(u.x, v.x) ? 1u : 0u) << (2 * q) | (open(u.y, v.y) ? 2u : 0u) << (2 * q);
        const __nv_bfloat162 r = __floats2bfloat162_rn(u.x, u.y);
        w4[q] = *reinterpret_cast<const uint32_t *>(&r);
    }
#pragma unroll 1
    while (left) {
        const int e = __ffs(left) - 1;
        left &= left - 1u;
        F2 dd = two_sum(__bfloat162float(x[e]), -mean.hi);
        dd.lo = __fsub_rn(dd.lo, mean.lo);
        F2 t = f2_mul(quick_two_sum(dd.hi, dd.lo), rstd);
        t = f2_mul(t, {__bfloat162float(g[e]), 0.0f});
        const uint32_t r = f2_to_bf16_bits(f2_add_f(t, __bfloat162float(b[e])));
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (q == e >> 1) w4[q] = (e & 1) ? (w4[q] & 0xFFFFu) | r << 16 : (w4[q] & 0xFFFF0000u) | r;
    }
    return make_uint4(w4[0], w4[1], w4[2], w4[3]);
}
__device__ __forceinline__ float ln_out_f32(float x, F2 mean, F2 rstd, float g, float b) {
    const float d = __fsub_rn(__fsub_rn(x, mean.hi), mean.lo);
    return __fmaf_rn(__fmul_rn(d, rstd.hi), g, b);
}

// ln_out_bf16 / ln_out_f32 for a float-float input element x + xlo (|xlo| <= ulp(x) / 2).
__device__ __forceinline__ uint16_t ln_out_bf16_lo(float x, float xlo, F2 mean, F2 rstd, float g, float b) {
    const float d = __fadd_rn(__fsub_rn(__fsub_rn(x, mean.hi), mean.lo), xlo);
    const float v = __fmul_rn(__fmul_rn(d, rstd.hi), g);
    const float u = __fadd_rn(v, b);
    const uint32_t low = __float_as_uint(u) & 0xFFFFu;
    const uint32_t dist = low > 0x8000u ? low - 0x8000u : 0x8000u - low;
    if (dist > 24u && fabsf(u) >= 0.5f * fabsf(v)) {
        const uint32_t bits = __float_as_uint(u);
        if ((bits & 0x7F800000u) == 0x7F800000u) return (uint16_t)((bits >> 16) | ((bits & 0x7FFFFFu) ? 0x40u : 0u));
        return (uint16_t)((bits + (low > 0x8000u ? 0x8000u : 0u)) >> 16);
    }
    F2 dd = two_sum(x, -mean.hi);
    dd.lo = __fadd_rn(__fsub_rn(dd.lo, mean.lo), xlo);
    F2 t = f2_mul(quick_two_sum(dd.hi, dd.lo), rstd);
    t = f2_mul(t, {g, 0.0f});
    return f2_to_bf16_bits(f2_add_f(t, b));
}
__device__ __forceinline__ float ln_out_f32_lo(float x, float xlo, F2 mean, F2 rstd, float g, float b) {
    const float d = __fadd_rn(__fsub_rn(__fsub_rn(x, mean.hi), mean.lo), xlo);
    return __fmaf_rn(__fmul_rn(d, rstd.hi), g, b);
}

}  // namespace fz
