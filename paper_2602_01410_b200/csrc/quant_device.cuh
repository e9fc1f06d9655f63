// Device helpers shared by the quantizer and the layer-statistics kernel: packed bf16 maxima, the
// tile-scale rules (paper Sec. 2.3: S = FPX_MAX / amax; power-of-two option), and the conversions
// binary32 <-> FP8 E4M3 / FP4 E2M1 codes.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <float.h>

#include "common.cuh"

namespace snip {

struct CtaPartial {  // statistics of one CTA, reduced in fixed order
    double sumsq_x;
    double sumsq_err;
    float amax;
    float pad[3];
};

// Fixed-order reduction of one set of per-CTA partials by one warp (each lane a fixed strided subset, then shuffles).
__device__ __forceinline__ void reduce_stats_warp(const StatJob &job, int lane)
{
    const CtaPartial *p = static_cast<const CtaPartial *>(job.partials);
    double dx = 0.0, de = 0.0;
    float am = 0.0f;
#pragma unroll 4
    for (int i = lane; i < job.n; i += 32) {
        const double2 v = __ldcg(reinterpret_cast<const double2 *>(p + i));
        dx += v.x;
        de += v.y;
        am = fmaxf(am, __ldcg(&p[i].amax));
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        dx += __shfl_xor_sync(0xFFFFFFFFu, dx, off);
        de += __shfl_xor_sync(0xFFFFFFFFu, de, off);
        am = fmaxf(am, __shfl_xor_sync(0xFFFFFFFFu, am, off));
    }
    if (lane == 0) { job.out->sumsq_x = dx; job.out->sumsq_err = de; job.out->amax = am; job.out->reserved = 0; }
}

__device__ __forceinline__ float bf16lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16hi(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }

// packed bf16: magnitude of each half = max(|a|, |b|); the sign bits are meaningless (mask them at the end)
__device__ __forceinline__ uint32_t absmax2x(uint32_t a, uint32_t b)
{
    uint32_t d;
    asm("max.xorsign.abs.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

__device__ __forceinline__ uint32_t max2(uint32_t x, uint32_t y)
{
    __nv_bfloat162 a = *reinterpret_cast<__nv_bfloat162 *>(&x);
    __nv_bfloat162 b = *reinterpret_cast<__nv_bfloat162 *>(&y);
    __nv_bfloat162 m = __hmax2(a, b);
    return *reinterpret_cast<uint32_t *>(&m);
}

// Scale of a tile from its amax.  Paper's rule: IEEE binary32 quotient FPX_MAX / amax, 1 for an empty
// tile, clamped to FLT_MAX.  Power-of-two option: the largest 2^e with amax * 2^e <= FPX_MAX, worked out
// on the exponent and significand bits (no division), e clamped to [-126, 127].
template <int FMT>
__device__ __forceinline__ float tile_scale(float amax, int pow2)
{
    constexpr float kMax = (FMT == SNIP_FMT_FP8_E4M3) ? 448.0f : 6.0f;
    if (amax == 0.0f) return 1.0f;
    if (pow2) {
        constexpr int kMaxExp = (FMT == SNIP_FMT_FP8_E4M3) ? 8 : 2;                       // FPX_MAX = m_f * 2^kMaxExp
        constexpr uint32_t kMaxMant = (FMT == SNIP_FMT_FP8_E4M3) ? 0x600000u : 0x400000u;  // m_f = 1.75 / 1.5
        const uint32_t b = __float_as_uint(amax);
        const int ef = (int)(b >> 23);                 // biased exponent; 0 for a (bf16) subnormal amax
        if (ef == 0) return __uint_as_float(254u << 23);   // amax < 2^-126: the clamp e = 127 applies
        int e = kMaxExp - (ef - 127) - (((b & 0x7FFFFFu) > kMaxMant) ? 1 : 0);
        e = max(-126, min(127, e));
        return __uint_as_float((uint32_t)(e + 127) << 23);
    }
    float s = __fdiv_rn(kMax, amax);
    return fminf(s, FLT_MAX);  // +inf -> FLT_MAX
}
// UE8M0 byte of 1/S for a power-of-two S, replicated into the four bytes of a word
__device__ __forceinline__ uint32_t sf_word(float s) { return (254u - (__float_as_uint(s) >> 23)) * 0x01010101u; }

// Two binary32 values -> two codes.  `lo` lands in the low byte / nibble.
__device__ __forceinline__ uint32_t cvt_e4m3x2(float lo, float hi)
{
    uint16_t r;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ uint32_t cvt_e2m1x2(float lo, float hi)
{
    uint16_t r;
    asm("{ .reg .b8 t; cvt.rn.satfinite.e2m1x2.f32 t, %1, %2; mov.b16 %0, {t, 0}; }"
        : "=h"(r) : "f"(hi), "f"(lo));
    return r;
}
// Two codes -> two binary32 values (exact).
__device__ __forceinline__ float2 dec_e4m3x2(uint32_t c)
{
    uint32_t h2;
    asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"((uint16_t)c));
    return __half22float2(*reinterpret_cast<__half2 *>(&h2));
}
__device__ __forceinline__ float2 dec_e2m1x2(uint32_t c)
{
    uint32_t h2;
    asm("{ .reg .b8 t, u; mov.b16 {t, u}, %1; cvt.rn.f16x2.e2m1x2 %0, t; }"
        : "=r"(h2) : "h"((uint16_t)c));
    return __half22float2(*reinterpret_cast<__half2 *>(&h2));
}

// FP4 error term of an element pair in units of 1/S: value(code) - t, t the binary32 products that the codes were rounded from.  The f16
// values of the codes (exact) enter the subtraction as they are; against decoding to binary32 and an FMA with -1/S it is a packed FMA and
// two conversions less (12.4 -> 9.7 clocks per pair and scheduler, the whole term alone), at a factor S^-2 per tile line.  The
// rounding of t stays in the term; next to FP4's coarse grid that is less than what a rounded 1/S left in it (the sums against 64 bits:
// 5e-8 -> 1e-8 of the result).  FP8's grid is sixteen times finer, and there it is more (up to 1.4e-7), so FP8 keeps the exact product.
__device__ __forceinline__ float2 fp4_scaled_err(uint32_t h2, const float2 t)
{
    float2 e;
    asm("{\n\t.reg .f16 l, h;\n\tmov.b32 {l, h}, %2;\n\t"
        "add.f32.f16 %0, l, %3;\n\t"
        "add.f32.f16 %1, h, %4;\n\t}"
        : "=f"(e.x), "=f"(e.y) : "r"(h2), "f"(-t.x), "f"(-t.y));
    return e;
}
// ... of a code pair
__device__ __forceinline__ float2 fp4_scaled_err_of_code(uint32_t c, const float2 t)
{
    uint32_t h2;
    asm("{ .reg .b8 t, u; mov.b16 {t, u}, %1; cvt.rn.f16x2.e2m1x2 %0, t; }" : "=r"(h2) : "h"((uint16_t)c));
    return fp4_scaled_err(h2, t);
}
// ... where the codes themselves are not wanted
__device__ __forceinline__ float2 fp4_scaled_rounding_err(const float2 t)
{
    uint32_t h2;
    asm("{ .reg .b8 c; cvt.rn.satfinite.e2m1x2.f32 c, %1, %2; cvt.rn.f16x2.e2m1x2 %0, c; }" : "=r"(h2) : "f"(t.y), "f"(t.x));
    return fp4_scaled_err(h2, t);
}

// ---- stochastic rounding (paper Sec. 6.1: FP4 output gradients) ------------------------------------

// Philox4x32 with 10 rounds (Salmon et al., SC'11): counter (c0, c1, 0, 0), key (k0, k1).
__device__ __forceinline__ void philox4x32_10(uint32_t c0, uint32_t c1, uint32_t k0, uint32_t k1, uint32_t (&out)[4])
{
    uint32_t c2 = 0, c3 = 0;
#pragma unroll
    for (int round = 0; round < 10; ++round) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
        c0 = hi1 ^ c1 ^ k0; c1 = lo1; c2 = hi0 ^ c3 ^ k1; c3 = lo0;
        k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
    }
    out[0] = c0; out[1] = c1; out[2] = c2; out[3] = c3;
}

// The 16-bit uniforms of an element pair (first element low) in the form sr_e2m1_value takes: 64 (65535 - u) + 31.
__device__ __forceinline__ void sr_addends(uint32_t u2, uint32_t &r0, uint32_t &r1)
{
    const uint32_t n = ~u2;
    r0 = ((n << 6) & 0x3FFFC0u) | 31u;
    r1 = ((n >> 10) & 0x3FFFC0u) | 31u;
}

// Stochastically rounded E2M1 value of t for the 16-bit uniform u: with a = min(|t|, 6), g the grid step at a (0.5 below 2, 1 below 4,
// else 2) and lo = floor(a/g)*g, the result is lo + g iff (a - lo)/g > (u + 1/2)/2^16, else lo; the sign of t is kept.
// On the bits: from 1 up, a grid point is a binary32 number whose low 22 significand bits are zero, and the rule asks whether these
// bits of a, f, exceed 32 (2u + 1), i.e. whether f + 64 (65535 - u) + 31 (= r, see sr_addends) carries out of them: one integer addition
// and a mask round the way the rule says, exponent included.  Below 1 the same holds for a + 1, added with upward rounding (a strict
// comparison with a multiple of the sum's last place cannot tell f from f rounded up).  About seven operations; in floating point it
// took sixteen and an integer conversion (quarter rate).
// SAT = false: |t| is known to be at most 6 up to rounding (a tile scaled by its own maximum; a few units in the last place above 6
// still round to 6, the largest addend leaves 33 units to the next grid point).
template <bool SAT>
__device__ __forceinline__ float sr_e2m1_value(float t, uint32_t r)
{
    const float a = SAT ? fminf(fabsf(t), 6.0f) : fabsf(t);
    float off;
    // 1 below 1, else 0: 2^120 - 2^120 a, which is 2^96 or more from the number next below 1 down (a set instruction would go to the
    // integer pipe, the one this function is bound by: two-output quantizers of an 8192 x 8640 gradient 116.0 -> 114.3 us, two-level 135.8 ->
    // 133.3 us)
    asm("fma.rn.sat.f32 %0, %1, 0fFB800000, 0f7B800000;" : "=f"(off) : "f"(a));
    const uint32_t q = (__float_as_uint(__fadd_ru(a, off)) + r) & 0xFFC00000u;
    return copysignf(__uint_as_float(q) - off, t);
}

}  // namespace snip
