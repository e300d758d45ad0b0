// Sine and cosine of an angle given in turns, for the w-phases (FP32).
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

namespace rimo {

__host__ __device__ __forceinline__ int cis_bits(float v) {
#ifdef __CUDA_ARCH__
    return __float_as_int(v);
#else
    int i;
    memcpy(&i, &v, sizeof(i));
    return i;
#endif
}
__host__ __device__ __forceinline__ float cis_float(int i) {
#ifdef __CUDA_ARCH__
    return __int_as_float(i);
#else
    float v;
    memcpy(&v, &i, sizeof(v));
    return v;
#endif
}

// an addition that is not fused with the product before it
__host__ __device__ __forceinline__ float cis_add(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fadd_rn(a, b);
#else
    return a + b;
#endif
}

// (cos, sin) of 2 pi r for |r| <= 1/2 (a little more does no harm): the nearest quarter turn q is
// split off by a rounding shift (1.5 x 2^23 gives 4 r + it unit spacing), and the remainder
// |f| <= 1/8 goes through the Taylor series of sin and cos in x = 2 pi f, |x| <= pi / 4, to x^9
// and x^10 (first omitted terms 2e-9 and 1e-10).  2 pi is 6.28125 (exact in FP32 with 9 bits) and the
// rest, so that the product with the leading term is rounded once, and the coefficient of f^4 in cos
// is 3.8e-5 below (2 pi)^4 / 4!, which takes up at |f| = 1/8 what rounding to FP32 takes from that of
// f^2.  Against 64 bits, over a turn: at most 5.3e-8, 0.89 ulp, 1.50e-8 rms; sincospif 5.3e-8, 0.97
// ulp, 1.51e-8 (with 2 pi in one FP32 number and the series' own coefficients 8.8e-8, 1.7 ulp,
// 1.9e-8).  About 26 instructions, none on the special function unit, where sincospif took about 45
// with four there (row passes 2 to 6 % faster: forward rows of 4096^2 / 32 bins 5.33 -> 5.21 ms).
// Minimax polynomials with a term less in each are as accurate and slower in the inverse row passes,
// whose loads are then scheduled later: 2048^2 0.549 -> 0.576 ms, 4096^2 3.97 -> 4.07.
__host__ __device__ __forceinline__ float2 cis_turn(float r) {
    const float t = cis_add(4.f * r, 12582912.f);
    const int q = cis_bits(t);
    const float f = fmaf(cis_add(t, -12582912.f), -0.25f, r);
    const float g = f * f;
    // sin: 2 pi f - (2 pi)^3 / 3! f^3 + ..., cos: 1 - (2 pi)^2 / 2! f^2 + ...
    const float p = fmaf(g, fmaf(g, fmaf(g, fmaf(g, 42.0586939448f, -76.7058597531f), 81.6052492761f), -41.3417022404f),
                         1.9353071796e-3f);
    const float s = fmaf(f, 6.28125f, f * p);
    const float c = fmaf(g, fmaf(g, fmaf(g, fmaf(g, fmaf(g, -26.4262567834f, 60.2446413719f), -85.4568172066f), 64.9393561f),
                                 -19.7392088022f),
                         1.f);
    const float cq = (q & 1) ? s : c, sq = (q & 1) ? c : s;  // up to sign
    return make_float2(cis_float(cis_bits(cq) ^ (((q + 1) & 2) << 30)), cis_float(cis_bits(sq) ^ ((q & 2) << 30)));
}

}  // namespace rimo
