// Sine and cosine of an angle given in turns, for the w-phases (FP32).
#pragma once

#include <cuda_runtime.h>

namespace rimo {

// (cos, sin) of 2 pi r for |r| <= 1/2 (a little more does no harm): the nearest quarter turn q is
// split off by a rounding shift (1.5 x 2^23 gives 4 r + it unit spacing), and the remainder
// |f| <= 1/8 goes through the Taylor series of sin and cos in x = 2 pi f, |x| <= pi / 4, to x^9
// and x^10 (first omitted terms 2e-9 and 1e-10; against 64 bits over a turn: at most 8.7e-8,
// 1.9e-8 rms, where rounding alone is 1.5e-8).  About 25 instructions, none on the special
// function unit, where sincospif took about 45 with four there (row
// passes 2 to 6 % faster: forward rows of 4096^2 / 32 bins 5.33 -> 5.21 ms)
__device__ __forceinline__ float2 cis_turn(float r) {
    const float t = __fadd_rn(4.f * r, 12582912.f);
    const int q = __float_as_int(t);
    const float f = fmaf(__fsub_rn(t, 12582912.f), -0.25f, r);
    const float g = f * f;
    // sin: f (2 pi - (2 pi)^3 / 3! g + ...), cos: 1 - (2 pi)^2 / 2! g + ...
    const float s = f * fmaf(g, fmaf(g, fmaf(g, fmaf(g, 42.0586939448f, -76.7058597531f), 81.6052492761f), -41.3417022404f),
                             6.2831853072f);
    const float c = fmaf(g, fmaf(g, fmaf(g, fmaf(g, fmaf(g, -26.4262567834f, 60.2446413719f), -85.4568172066f), 64.9393940227f),
                                 -19.7392088022f),
                         1.f);
    const float cq = (q & 1) ? s : c, sq = (q & 1) ? c : s;  // up to sign
    return make_float2(__int_as_float(__float_as_int(cq) ^ (((q + 1) & 2) << 30)),
                       __int_as_float(__float_as_int(sq) ^ ((q & 2) << 30)));
}

}  // namespace rimo
