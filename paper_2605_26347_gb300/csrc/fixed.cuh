// Fixed-point accumulation in shared memory, shared by the grid step and the holographic apply:
// packed FP32 arithmetic, the split of a scaled contribution into two integer words, and the
// accumulator planes' row pitch.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace rimo {

// Row pitch of the accumulator planes for patches of side PW and tiles of side max_S: the rows
// one instruction adds to (32 / CW rows of CW lanes, see vis_tile) fall in different banks.
__host__ __device__ constexpr int pitch_of(int PW, int max_S = 15) {
    return max_S <= 8 ? PW + (40 - PW % 16) % 16      // 8 modulo 16: four rows of 8 lanes
         : max_S <= 16 ? PW + (48 - PW % 32) % 32     // 16 modulo 32: two rows of 16
                       : PW;
}

// Two FP32 numbers in one 64-bit register pair (packed arithmetic: the same roundings as two
// scalar instructions in one issue slot).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pk(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 upk(f32x2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// rint by the 1.5 x 2^23 shift: for |d| < 2^22, d + FX_MAGIC has unit spacing, so its bits
// minus those of FX_MAGIC are rint(d) (round to nearest even)
constexpr float FX_MAGIC = 12582912.0f;
constexpr int FX_MAGIC_BITS = 0x4B400000;

// The scaled contribution d (|d.x|, |d.y| <= 2^21) to cell a of the accumulator planes [hi re, hi
// im, lo re, lo im], split into rint(d) and 2^16 x the residual.
__device__ __forceinline__ void fx_add2(int* a, int plane, f32x2 d) {
    const f32x2 M = pk(FX_MAGIC, FX_MAGIC);
    const f32x2 h = add2(d, M);
    const f32x2 rf = fma2(add2(h, pk(-FX_MAGIC, -FX_MAGIC)), pk(-1.f, -1.f), d);
    const float2 hs = upk(h), ls = upk(fma2(rf, pk(65536.f, 65536.f), M));
    atomicAdd(a, __float_as_int(hs.x) - FX_MAGIC_BITS);
    atomicAdd(a + plane, __float_as_int(hs.y) - FX_MAGIC_BITS);
    atomicAdd(a + 2 * plane, __float_as_int(ls.x) - FX_MAGIC_BITS);
    atomicAdd(a + 3 * plane, __float_as_int(ls.y) - FX_MAGIC_BITS);
}

}  // namespace rimo
