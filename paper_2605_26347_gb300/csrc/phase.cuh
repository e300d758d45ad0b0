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

// (cos, sin) of 2 pi r for |r| <= 1/2 (a little more does no harm): the nearest quarter turn q is
// split off by a rounding shift (1.5 x 2^23 gives 4 r + it unit spacing), and the remainder
// |f| <= 1/8 goes through polynomials in g = f^2, sin(2 pi f) = f (6.28125 + p(g)) (6.28125 is exact in
// FP32, so that the product with the leading term is rounded once) and cos(2 pi f) = 1 + g (...).  Their
// coefficients are minimax fits (linear programme over [0, 1/64]; relative error 3.6e-9 of the sine,
// 4e-10 of the cosine), each rounded to FP32 before the next ones are fitted.  Against 64 bits, over
// a turn: at most 5.2e-8, 0.86 ulp, 1.50e-8 rms; sincospif 5.3e-8, 0.97 ulp, 1.51e-8 (the Taylor
// series with 2 pi in one FP32 number, two terms more: 8.8e-8, 1.7 ulp, 1.9e-8).  About 24
// instructions, none on the special function unit, where sincospif took about 45 with four there
// (row passes 2 to 6 % faster: forward rows of 4096^2 / 32 bins 5.33 -> 5.21 ms).
__host__ __device__ __forceinline__ float2 cis_turn(float r) {
    const float t = 4.f * r + 12582912.f;  // (4 r is exact: the same with or without a fused multiply-add)
    const int q = cis_bits(t);
    const float f = fmaf(t - 12582912.f, -0.25f, r);
    const float g = f * f;
    const float p = fmaf(g, fmaf(g, fmaf(g, -75.3683167f, 81.5918808f), -41.3416595f), 1.9352868e-3f);
    const float s = fmaf(f, 6.28125f, f * p);
    const float c = fmaf(g, fmaf(g, fmaf(g, fmaf(g, 58.5611687f, -85.4231186f), 64.9391403f), -19.7392082f), 1.f);
    const float cq = (q & 1) ? s : c, sq = (q & 1) ? c : s;  // up to sign
    return make_float2(cis_float(cis_bits(cq) ^ (((q + 1) & 2) << 30)), cis_float(cis_bits(sq) ^ ((q & 2) << 30)));
}

}  // namespace rimo
