#pragma once
// Single-precision Box-Muller (the single-precision sampler's normals) for the
// 24-bit uniforms u1 = fl(a + 1/2) 2^-24, u2 = fl(b + 1/2) 2^-24 (a, b the top
// 24 bits of two Philox words), in float, from the hardware approximations:
//  * -2 ln u1 = -2 ln 2 log2(u1) with lg2.approx.f32 (absolute error about
//    2^-22.6), except for u1 > 15/16, where that absolute error would be large
//    against ln u1 itself: there -ln(1 - t) = t (1 + t/2 + .. + t^6/7) with
//    t = 1 - u1 exact (truncation t^7/8 < 2^-31 relative);
//  * R = sqrt(v) by sqrt.approx.f32 (0 where u1 rounds to 1);
//  * cos/sin(2 pi u2) = -(cos, sin)(2 pi (u2 - 1/2)) by __sincosf on an
//    argument in (-pi, pi) (u2 - 1/2 is exact; absolute error about 2^-21).
// Largest error: about 5e-7 R from the sine and cosine, at most 3e-7 from
// the logarithm (at u1 = 15/16, where R = 0.36); the GPU tests hold the
// normals to 1e-6 (1 + R) of the oracle's double-precision Box-Muller on the
// same uniforms.  Earlier, table-driven forms
// (a 49-node logarithm, quadrant-reduced 33-node sin/cos), were a few units
// in the last place accurate but cost about 55 instructions per pair, the
// largest item of the issue-bound single-precision sampler after the W_p
// Horner; this one costs about 25, and with two pairs side by side in packed
// operations about 18 (the anharmonic oscillator's 48 x 48 amplitude matrix at p = 10, 54.0 ->
// 52.2 ms; the anharmonic oscillator at p = 18, N = 1024, 17.5 -> 17.2 ms).
#include <cstdint>

namespace su {
namespace bm32 {

// z[0], z[1] = R cos(2 pi u2), R sin(2 pi u2), R = sqrt(-2 ln u1), of the words
// w.x, w.y, and z[2], z[3] of w.z, w.w.  Both pairs at once: a packed operation
// occupies the two FMA pipes of a scheduler for as long as a single one holds up
// the packed Horner of W_p beside it.  The approximations in their ftz forms, with
// no code for subnormal arguments (u1 >= 2^-25, v = 0 or >= 2^-24).
__device__ __forceinline__ void quad(uint4 w, float (&z)[4]) {
    auto both = [](float c) { return make_float2(c, c); };
    // ((w >> 8) + 1/2) 2^-24 in one rounding: the scaling is exact
    const float2 u1 = __ffma2_rn(make_float2((float)(w.x >> 8), (float)(w.z >> 8)), both(0x1p-24f), both(0x1p-25f));
    const float2 u2 = __ffma2_rn(make_float2((float)(w.y >> 8), (float)(w.w >> 8)), both(0x1p-24f), both(0x1p-25f));

    // ---- v = -2 ln u1; the series with its coefficients doubled
    const float2 t = __ffma2_rn(u1, both(-1.0f), both(1.0f));
    float2 ser = __ffma2_rn(t, both(2.0f / 7.0f), both(2.0f / 6.0f));
    ser = __ffma2_rn(t, ser, both(0.4f));
    ser = __ffma2_rn(t, ser, both(0.5f));
    ser = __ffma2_rn(t, ser, both(2.0f * 0.333333343f));
    ser = __ffma2_rn(t, ser, both(1.0f));
    ser = __ffma2_rn(t, ser, both(2.0f));
    const float2 near = __fmul2_rn(t, ser);
    float2 lg;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(lg.x) : "f"(u1.x));
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(lg.y) : "f"(u1.y));
    const float2 far = __fmul2_rn(lg, both(-1.38629436f));   // -2 ln 2
    const float va = t.x < 0.0625f ? near.x : far.x, vb = t.y < 0.0625f ? near.y : far.y;

    // ---- R = sqrt(v), v in {0} u [2^-24, 35]
    float Ra, Rb;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(Ra) : "f"(va));
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(Rb) : "f"(vb));

    // ---- cos, sin of 2 pi u2
    const float2 x = __fmul2_rn(__fadd2_rn(u2, both(-0.5f)), both(6.28318530718f));
    float2 ca, cb;   // (cos, sin)
    __sincosf(x.x, &ca.y, &ca.x);
    __sincosf(x.y, &cb.y, &cb.x);
    const float2 za = __fmul2_rn(ca, both(-Ra)), zb = __fmul2_rn(cb, both(-Rb));
    z[0] = za.x;
    z[1] = za.y;
    z[2] = zb.x;
    z[3] = zb.y;
}

}  // namespace bm32
}  // namespace su
