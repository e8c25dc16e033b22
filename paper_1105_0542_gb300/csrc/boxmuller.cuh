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
// Horner; this one costs about 25.
#include <cstdint>

namespace su {
namespace bm32 {

// z0 = R cos(2 pi u2), z1 = R sin(2 pi u2), R = sqrt(-2 ln u1)
__device__ __forceinline__ void pair(uint32_t a, uint32_t b, float &z0, float &z1) {
    // ((w >> 8) + 1/2) 2^-24 in one rounding: the scaling is exact
    const float u1 = fmaf((float)(a >> 8), 0x1p-24f, 0x1p-25f);
    const float u2 = fmaf((float)(b >> 8), 0x1p-24f, 0x1p-25f);

    // ---- v = -2 ln u1
    const float t = 1.0f - u1;
    float lg;
    asm("lg2.approx.f32 %0, %1;" : "=f"(lg) : "f"(u1));
    float ser = fmaf(t, 1.0f / 7.0f, 1.0f / 6.0f);
    ser = fmaf(t, ser, 0.2f);
    ser = fmaf(t, ser, 0.25f);
    ser = fmaf(t, ser, 0.333333343f);
    ser = fmaf(t, ser, 0.5f);
    ser = fmaf(t, ser, 1.0f);
    const float v = t < 0.0625f ? 2.0f * t * ser : -1.38629436f * lg;   // -2 ln 2 = -1.38629436

    // ---- R = sqrt(v), v in {0} u [2^-24, 35]
    float R;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(R) : "f"(v));

    // ---- cos, sin of 2 pi u2
    float sn, cs;
    __sincosf(6.28318530718f * (u2 - 0.5f), &sn, &cs);
    z0 = -R * cs;
    z1 = -R * sn;
}

}  // namespace bm32
}  // namespace su
