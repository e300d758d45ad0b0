// The oversampled 2-D DFT F of Eq. 6 and its adjoint, as four row passes.
//
// Forward, for w-bin p (F Z_p of Eq. 6):
//   rows pass  : image row i (n_x pixels) -> z = x * Z_p (grid correction and the w-layer
//                chirp, Section 3.2) -> zero-padded 2n_x-point DFT along l, written
//                transposed as A^T[u][i]  (2 n_x rows of n_y).
//   cols pass  : row u of A^T -> zero-padded 2n_y-point DFT along m -> X[u][v].
// Adjoint (Z_p^dagger F^dagger of Eq. 8):
//   cols pass  : row u of Xh (2 n_y cells) -> 2n_y-point inverse DFT cropped to the n_y
//                image rows -> B[i][u], transposed.
//   rows pass  : row i of B (2 n_x cells) -> cropped inverse DFT along u -> * conj(Z_p),
//                accumulated into the output image.
//
// Each pass is one 2N-point Stockham radix-16 FFT per row held in registers (16 points per
// thread, 2N/16 threads per row), exchanging through shared memory between stages; at
// 2N = 8192 the two column passes hold 32 points per thread instead (256 threads per row,
// radix 32 x 16 x 16: two exchanges and barriers instead of three; measured per 4096^2/50M
// apply when it was introduced, forward cols 4.28 -> 3.81 ms and inverse cols + fold 7.56 ->
// 6.90 ms, while the row passes, which also evaluate Z_p per point, were slower so: 5.32 -> 5.55
// and 4.30 -> 4.61 ms).  What bounds the passes at 4096^2 (32 bins, 24M visibilities, per apply):
// forward cols 2.91 ms, issue and the FMA pipe (63 and 62 %) and latency; fold + inverse cols 5.25
// ms, memory latency and the clusters' barriers; forward rows 5.12 ms, barriers (block and cluster), the exchange and the
// 32-byte pieces of the transposed store (69 % of the load/store pipe); inverse rows 3.95 ms,
// memory latency at 4.3 TB/s with two 512-thread rows per SM (with the 8192 points as two halves of
// 4096, two exchanges instead of three, they took the same 5.18 and 4.09 ms).  The
// zero padding and the crop are exploited where they cost nothing: forward passes never
// load the zero half of their input (those points enter the first butterflies as
// constants), inverse passes store only the kept half of their output, and the
// column passes touch only the grid rows and tiles the bin's footprints reach.
#include <cstring>
#include <cstdio>

#include <type_traits>

#include "internal.h"
#include "phase.cuh"

namespace rimo {

// Complex additions of the butterflies: packed (both halves in one issue slot, with the roundings of
// two scalar additions) or, with PK = false, scalar (see fft_n).
template <bool PK = true>
__device__ __forceinline__ float2 cadd(float2 a, float2 b) {
    return PK ? __fadd2_rn(a, b) : make_float2(a.x + b.x, a.y + b.y);
}
template <bool PK = true>
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
    return PK ? __ffma2_rn(b, make_float2(-1.f, -1.f), a) : make_float2(a.x - b.x, a.y - b.y);
}
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {  // a * conj(b)
    return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.y, b.x, -a.x * b.y));
}

template <bool PK>
__device__ __forceinline__ void dft2(float2& a, float2& b) {
    float2 t = a;
    a = cadd<PK>(t, b);
    b = csub<PK>(t, b);
}

template <bool INV, bool PK>
__device__ __forceinline__ void dft4(float2& x0, float2& x1, float2& x2, float2& x3) {
    const float2 a0 = cadd<PK>(x0, x2), a1 = csub<PK>(x0, x2), a2 = cadd<PK>(x1, x3), d = csub<PK>(x1, x3);
    x0 = cadd<PK>(a0, a2);
    x2 = csub<PK>(a0, a2);
    // a1 -+ i d: the halves swap, so these additions are scalar
    const float2 p = make_float2(a1.x + d.y, a1.y - d.x), q = make_float2(a1.x - d.y, a1.y + d.x);
    x1 = INV ? q : p;
    x3 = INV ? p : q;
}

#define RS2 0.70710678118654752440f
#define C16 0.92387953251128675613f
#define S16 0.38268343236508977173f

// W_N^k for the small radices: forward e^{-2 pi i k / N}, inverse its conjugate
template <bool INV>
__device__ __forceinline__ float2 w8(int k) {
    const float c[4] = {1.f, RS2, 0.f, -RS2};
    const float s[4] = {0.f, RS2, 1.f, RS2};
    return make_float2(c[k], INV ? s[k] : -s[k]);
}

template <bool INV, bool PK = true>
__device__ __forceinline__ void dft8(float2* v) {
    dft4<INV, PK>(v[0], v[2], v[4], v[6]);
    dft4<INV, PK>(v[1], v[3], v[5], v[7]);
    float2 o1 = cmul(v[3], w8<INV>(1)), o2 = cmul(v[5], w8<INV>(2)), o3 = cmul(v[7], w8<INV>(3));
    float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1];
    v[0] = cadd<PK>(e0, o0);
    v[4] = csub<PK>(e0, o0);
    v[1] = cadd<PK>(e1, o1);
    v[5] = csub<PK>(e1, o1);
    v[2] = cadd<PK>(e2, o2);
    v[6] = csub<PK>(e2, o2);
    v[3] = cadd<PK>(e3, o3);
    v[7] = csub<PK>(e3, o3);
}

template <bool INV>
__device__ __forceinline__ float2 w16(int k) {  // k in [0, 9]
    const float c[10] = {1.f, C16, RS2, S16, 0.f, -S16, -RS2, -C16, -1.f, -C16};
    const float s[10] = {0.f, S16, RS2, C16, 1.f, C16, RS2, S16, 0.f, -S16};
    return make_float2(c[k], INV ? s[k] : -s[k]);
}

// 16-point DFT as 4 x 4: inner DFT_4 over n1 (stride 4), twiddle W16^{n2 k1}, outer DFT_4.
template <bool INV, bool PK = true>
__device__ __forceinline__ void dft16(float2* v) {
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) dft4<INV, PK>(v[n2], v[n2 + 4], v[n2 + 8], v[n2 + 12]);
    // now v[n2 + 4 k1] = A[n2][k1]
#pragma unroll
    for (int n2 = 1; n2 < 4; ++n2)
#pragma unroll
        for (int k1 = 1; k1 < 4; ++k1) v[n2 + 4 * k1] = cmul(v[n2 + 4 * k1], w16<INV>(n2 * k1));
    float2 t[16];
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
        float2 a = v[0 + 4 * k1], b = v[1 + 4 * k1], c = v[2 + 4 * k1], d = v[3 + 4 * k1];
        dft4<INV, PK>(a, b, c, d);
        t[k1 + 0] = a;
        t[k1 + 4] = b;
        t[k1 + 8] = c;
        t[k1 + 12] = d;
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = t[k];
}

// dft16 of an input whose points 4 .. 11 are zero (the first stage of a forward pass, whose
// row holds its samples in the centred half): the first layer of 4-point DFTs reduces to
// sums and differences of x_n2 and x_n2+12 (written out, since the compiler may not drop an
// addition of +0, which would turn -0 into +0)
template <bool INV, bool PK = true>
__device__ __forceinline__ void dft16_hz(float2* v) {
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) {
        const float2 a = v[n2], d = v[n2 + 12];
        v[n2] = cadd<PK>(a, d);
        v[n2 + 8] = csub<PK>(a, d);
        const float2 p = make_float2(a.x + d.y, a.y - d.x), q = make_float2(a.x - d.y, a.y + d.x);
        v[n2 + 4] = INV ? p : q;
        v[n2 + 12] = INV ? q : p;
    }
#pragma unroll
    for (int n2 = 1; n2 < 4; ++n2)
#pragma unroll
        for (int k1 = 1; k1 < 4; ++k1) v[n2 + 4 * k1] = cmul(v[n2 + 4 * k1], w16<INV>(n2 * k1));
    float2 t[16];
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
        float2 a = v[0 + 4 * k1], b = v[1 + 4 * k1], c = v[2 + 4 * k1], d = v[3 + 4 * k1];
        dft4<INV, PK>(a, b, c, d);
        t[k1 + 0] = a;
        t[k1 + 4] = b;
        t[k1 + 8] = c;
        t[k1 + 12] = d;
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = t[k];
}

template <int R, bool INV, bool PK>
__device__ __forceinline__ void dft_r(float2* v) {
    if constexpr (R == 2) dft2<PK>(v[0], v[1]);
    else if constexpr (R == 4) dft4<INV, PK>(v[0], v[1], v[2], v[3]);
    else if constexpr (R == 8) dft8<INV, PK>(v);
    else dft16<INV, PK>(v);
}

// Exchange buffers are padded: element i at i + i / 16.  A stage's addresses are one base per
// thread and compile-time offsets (a multiple of 16 moves by padded16): the index arithmetic,
// spelled out per element, was 15 to 20 % of the passes' instructions (see the stages below).
__device__ __forceinline__ int pidx(int i) { return i + (i >> 4); }
__host__ __device__ constexpr int padded16(int i) { return i + i / 16; }

// One Stockham stage of radix R after NS points have been combined (NS * R <= N).
// Thread t owns butterflies j = t + q T (q < 16/R, T = N/16); butterfly j reads
// a[j + r N/R] and writes a'[(j / NS) NS R + j % NS + r NS].  Its twiddles
// W_{NS R}^{r (j mod NS)} come from the stage table tws[r NS + j mod NS], laid out so that
// consecutive threads read consecutive entries.
// HZ: a first stage whose inputs m = 4 .. 11 are zero (forward passes)
template <int N, int R, int NS, bool INV, bool FIRST, bool LAST, bool HZ = false, bool PK = true>
__device__ __forceinline__ void fft_stage(float2 (&v)[16], float2* sm, int t, const float2* __restrict__ tws) {
    constexpr int T = N / 16;
    constexpr int Q = 16 / R;
    if (!FIRST) {
        const float2* rd = sm + pidx(t);
#pragma unroll
        for (int q = 0; q < Q; ++q)
#pragma unroll
            // element t + q T + r N / R: T and N / R are multiples of 16, or T = 8 and q < 2
            for (int r = 0; r < R; ++r) v[q * R + r] = rd[padded16(q * T) + padded16(r * (N / R))];
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        if (NS > 1) {
            const int jm = (t + q * T) & (NS - 1);
            if constexpr (R == 16) {
                // W^r for r = 1 .. 15 from two table entries (W and W^4), at most three
                // products deep: two loads instead of fifteen (fifteen loads from the table
                // were slower: 49.0 against 48.4 ms per 4096^2/50M apply)
                float2 w[16];
                w[1] = __ldg(&tws[NS + jm]);
                w[4] = __ldg(&tws[4 * NS + jm]);
                w[2] = cmul(w[1], w[1]);
                w[3] = cmul(w[2], w[1]);
                w[8] = cmul(w[4], w[4]);
#pragma unroll
                for (int r = 5; r < 8; ++r) w[r] = cmul(w[4], w[r - 4]);
#pragma unroll
                for (int r = 9; r < 16; ++r) w[r] = cmul(w[8], w[r - 8]);
#pragma unroll
                for (int r = 1; r < 16; ++r) v[q * R + r] = INV ? cmulc(v[q * R + r], w[r]) : cmul(v[q * R + r], w[r]);
            } else {
#pragma unroll
                for (int r = 1; r < R; ++r) {
                    float2 w = __ldg(&tws[r * NS + jm]);
                    v[q * R + r] = INV ? cmulc(v[q * R + r], w) : cmul(v[q * R + r], w);
                }
            }
        }
        if constexpr (HZ && R == 16) dft16_hz<INV, PK>(&v[q * R]);
        else dft_r<R, INV, PK>(&v[q * R]);
    }
    if constexpr (!LAST) {
        // butterfly j = t (R = 16, Q = 1): element (j / NS) 16 NS + j mod NS + r NS
        static_assert(R == 16, "only a last stage has a smaller radix");
        float2* wr = sm + padded16((t / NS) * NS * 16) + (NS == 1 ? 0 : pidx(t & (NS - 1)));
#pragma unroll
        for (int r = 0; r < R; ++r) wr[NS == 1 ? r : padded16(r * NS)] = v[r];
        __syncthreads();
    }
}

// Radix plan of an L-point transform: 16, then 16s, then the remainder; L <= 256: two
// stages (16, L/16), L <= 4096: three (16, 16, L/256), L = 8192: four (16, 16, 16, 2).
// ----------------------------------------------------------------------------- 32 points per thread
// The 8192-point transform with 256 threads of 32 points (radix 32, 16, 16): two
// shared-memory exchanges instead of three.  Exchange buffer index i + i / 32 (the stride-32
// writes of the first stage spread over the banks).
__device__ __forceinline__ int pidx32(int i) { return i + (i >> 5); }

#define C32_1 0.98078528040323044913f
#define S32_1 0.19509032201612826785f
#define C32_3 0.83146961230254523708f
#define S32_3 0.55557023301960222474f

// W_32^k, k in [0, 16): forward e^{-2 pi i k / 32}, inverse its conjugate
template <bool INV>
__device__ __forceinline__ float2 w32(int k) {
    const float c[16] = {1.f, C32_1, C16, C32_3, RS2, S32_3, S16, S32_1, 0.f, -S32_1, -S16, -S32_3, -RS2, -C32_3, -C16, -C32_1};
    const float s[16] = {0.f, S32_1, S16, S32_3, RS2, C32_3, C16, C32_1, 1.f, C32_1, C16, C32_3, RS2, S32_3, S16, S32_1};
    return make_float2(c[k], INV ? s[k] : -s[k]);
}

// 32-point DFT in place: v[r] in natural order in and out (even / odd halves by dft16, then
// one radix-2 layer with W_32^k).  HZ: inputs 8 .. 23 are zero.
template <bool INV, bool HZ>
__device__ __forceinline__ void dft32(float2* v) {
    float2 e[16], o[16];
#pragma unroll
    for (int n = 0; n < 16; ++n) {
        e[n] = v[2 * n];
        o[n] = v[2 * n + 1];
    }
    if constexpr (HZ) {
        // e[n] = x[2n], o[n] = x[2n + 1]: zero for 2n (+1) in [8, 24), i.e. n in [4, 12)
        dft16_hz<INV>(e);
        dft16_hz<INV>(o);
    } else {
        dft16<INV>(e);
        dft16<INV>(o);
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const float2 t = k == 0 ? o[0] : cmul(o[k], w32<INV>(k));
        v[k] = cadd(e[k], t);
        v[k + 16] = csub(e[k], t);
    }
}

// tws32 layout as in DevTables.  In: v[m] = element t + 256 m.  Out: v[s] is element
// out_k32(t, s).  All 256 threads of the row must call it.
template <bool INV, bool HZ>
__device__ __forceinline__ void fft8192_32(float2 (&v)[32], float2* sm, int t, const float2* __restrict__ tw) {
    // every address is one base per thread and a compile-time offset (multiples of 32 move by
    // 33 / 32): 9 % of the pass was index arithmetic without that
    dft32<INV, HZ>(v);  // stage 1: butterfly j = t, outputs at 32 t + r
    float2* w1 = sm + 33 * t;
#pragma unroll
    for (int r = 0; r < 32; ++r) w1[r] = v[r];
    __syncthreads();
    // stage 2: NS = 32, R = 16, butterflies j = t + 256 q, reads j + 512 r
    const float2* rd = sm + pidx32(t);
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int r = 0; r < 16; ++r) v[16 * q + r] = rd[264 * q + 528 * r];
    __syncthreads();
    float2* w2 = sm + (t >> 5) * 528 + (t & 31);  // outputs at (j / 32) 512 + j mod 32 + 32 r
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int j = t + 256 * q, jm = j & 31;
        float2 w[16];
        w[1] = __ldg(&tw[32 + jm]);
        w[4] = __ldg(&tw[4 * 32 + jm]);
        w[2] = cmul(w[1], w[1]);
        w[3] = cmul(w[2], w[1]);
        w[8] = cmul(w[4], w[4]);
#pragma unroll
        for (int r = 5; r < 8; ++r) w[r] = cmul(w[4], w[r - 4]);
#pragma unroll
        for (int r = 9; r < 16; ++r) w[r] = cmul(w[8], w[r - 8]);
#pragma unroll
        for (int r = 1; r < 16; ++r) v[16 * q + r] = INV ? cmulc(v[16 * q + r], w[r]) : cmul(v[16 * q + r], w[r]);
        dft16<INV>(&v[16 * q]);
#pragma unroll
        for (int r = 0; r < 16; ++r) w2[8 * 528 * q + 33 * r] = v[16 * q + r];
    }
    __syncthreads();
    // stage 3: NS = 512, R = 16, butterflies j = t + 256 q (< 512), reads j + 512 r
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int r = 0; r < 16; ++r) v[16 * q + r] = rd[264 * q + 528 * r];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int jm = t + 256 * q;
        const float2* __restrict__ tw3 = tw + 512;
        float2 w[16];
        w[1] = __ldg(&tw3[512 + jm]);
        w[4] = __ldg(&tw3[4 * 512 + jm]);
        w[2] = cmul(w[1], w[1]);
        w[3] = cmul(w[2], w[1]);
        w[8] = cmul(w[4], w[4]);
#pragma unroll
        for (int r = 5; r < 8; ++r) w[r] = cmul(w[4], w[r - 4]);
#pragma unroll
        for (int r = 9; r < 16; ++r) w[r] = cmul(w[8], w[r - 8]);
#pragma unroll
        for (int r = 1; r < 16; ++r) v[16 * q + r] = INV ? cmulc(v[16 * q + r], w[r]) : cmul(v[16 * q + r], w[r]);
        dft16<INV>(&v[16 * q]);
    }
}
// output index of v[s] after fft8192_32 in thread t: j = t + 256 (s / 16), k = j + 512 (s mod 16)
__device__ __forceinline__ int out_k32(int t, int s) { return t + 256 * (s >> 4) + 512 * (s & 15); }

template <int N>
struct Plan16 {
    static constexpr int STAGES = N <= 256 ? 2 : (N <= 4096 ? 3 : 4);
    static constexpr int R_LAST = N <= 256 ? N / 16 : (N <= 4096 ? N / 256 : N / 4096);
};

// In: v[m] = element t + T m of the input.  Out: element t + T m of the output is
// v[out_slot<N>(m)].  All threads of the block must call it (block-wide barriers).
// tws: the stage twiddle tables of length N (see stage_twiddles on the host): the second
// stage's W_{16 R}^{r j} at [0, 16 R), the third stage's W_{256 R}^{r j} at [256, 256 + 256 R),
// a fourth stage's W_{4096 R}^{r j} at [4352, 4352 + 4096 R).
// PK: packed additions.  Off for the 8192-point row passes and for inv_rows_bins_kernel, which hold
// every register: the moves and spills that register pairs cost are more than the issue slots they
// save.  Per 4096^2/24M apply, scalar and packed: forward rows 5.18 and 5.29 ms, inverse rows 4.04
// and 4.12; 512^2 in one bin, inverse rows 15.9 and 18.5 us.  The other passes gain: forward cols at
// 4096^2 3.53 -> 3.19 ms, inverse cols 5.65 -> 5.55, 2048^2 inverse rows 0.612 -> 0.561.
template <int N, bool INV, bool HZ = false, bool PK = N <= 4096>
__device__ __forceinline__ void fft_n(float2 (&v)[16], float2* sm, int t, const float2* __restrict__ tws) {
    constexpr int RL = Plan16<N>::R_LAST;
    fft_stage<N, 16, 1, INV, true, false, HZ, PK>(v, sm, t, tws);
    if constexpr (Plan16<N>::STAGES == 2) {
        fft_stage<N, RL, 16, INV, false, true, false, PK>(v, sm, t, tws);
    } else {
        fft_stage<N, 16, 16, INV, false, false, false, PK>(v, sm, t, tws);
        if constexpr (Plan16<N>::STAGES == 3) {
            fft_stage<N, RL, 256, INV, false, true, false, PK>(v, sm, t, tws + 256);
        } else {
            fft_stage<N, 16, 256, INV, false, false, false, PK>(v, sm, t, tws + 256);
            fft_stage<N, RL, 4096, INV, false, true, false, PK>(v, sm, t, tws + 256 + 4096);
        }
    }
}

template <int N>
__device__ __forceinline__ int out_slot(int m) {
    constexpr int RL = Plan16<N>::R_LAST;
    constexpr int Q = 16 / RL;
    return (m % Q) * RL + m / Q;
}

// e^{-2 pi i w dn} from the double-float phase w * dn, reduced modulo 1 before sincos.
// The product and reduction keep ~48 significant bits (error-free FMA product), which is
// the FP64-accurate w-phase argument; only the final sine and cosine are single precision.
__device__ __forceinline__ float2 wphase(float w_hi, float w_lo, float2 d) {
    float p = w_hi * d.x;
    float e = fmaf(w_hi, d.x, -p);
    e = fmaf(w_hi, d.y, e);
    e = fmaf(w_lo, d.x, e);
    float k = rintf(p);
    const float2 cs = cis_turn((p - k) + e);
    return make_float2(cs.x, -cs.y);
}

struct ZArgs {
    const float4* zq;   // quarter table [|i_c|][|j_c|]: (n - 1) as a float pair, |Z_p|
    int zq_ld;
    float w_hi, w_lo;
};

// Z_p(i, j) = gc_x gc_y [/ n] e^{-2 pi i w (n - 1)} at (l_j, m_i): one table load (the grid
// correction and the w-term depend on |i_c|, |j_c| only)
__device__ __forceinline__ float2 z_factor(const ZArgs& z, int i, int j, int ic, int jc) {
    (void)i;
    (void)j;
    const float4 q = __ldg(&z.zq[abs(ic) * z.zq_ld + abs(jc)]);
    const float2 ph = wphase(z.w_hi, z.w_lo, make_float2(q.x, q.y));
    return make_float2(ph.x * q.z, ph.y * q.z);
}

// ----------------------------------------------------------------------------- bound
// Bound on the grid-step contributions of Phi^dagger Phi x.  Every forward-grid value of
// every w-bin is a sum of Z_p x over the pixels with unit-modulus twiddles, and the
// w-phase has unit modulus, so |X| <= B_x = sum_l (|x_l.re| + |x_l.im|) |Z_l|; a
// de-gridded y_k then has |y_k.x| + |y_k.y| <= sqrt(2) T1 B_x (T1 = max tap sum), and a
// contribution component at most tmax times that.  2 tmax T1 B_x goes to
// d_fx[FX_MAXTERM].  Per-block partial sums are added by the last block in block order
// (the bound, hence the scales, do not depend on timing).  Non-finite x sets status 3.
__global__ void __launch_bounds__(256) image_bound_kernel(const float2* __restrict__ x, int nx, int ny, ZArgs z,
                                                          uint32_t* fx, int* status) {
    __shared__ float red[256];
    __shared__ bool last;
    float acc = 0.f;
    bool bad = false;
    const int n = nx * ny;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        const int i = e / nx, j = e - i * nx;
        const float g = __ldg(&z.zq[abs(i - ny / 2) * z.zq_ld + abs(j - nx / 2)]).z;  // |Z_p|
        const float2 v = x[e];
        const float m = fabsf(v.x) + fabsf(v.y);
        bad |= !(m <= 3.4028234e38f);
        acc = fmaf(m, fabsf(g), acc);
    }
    if (bad) atomicExch(status, 3);
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        reinterpret_cast<float*>(fx + FX_PART)[blockIdx.x] = red[0];
        __threadfence();
        last = atomicAdd(fx + FX_COUNT, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    float t = 0.f;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) t += __ldcg(reinterpret_cast<const float*>(fx + FX_PART) + b);
    red[threadIdx.x] = t;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const float mt = 2.f * __uint_as_float(__ldcg(fx + FX_TMAX)) * __uint_as_float(__ldcg(fx + FX_T1)) * red[0];
        if (!(mt <= 3.4028234e38f)) atomicExch(status, 3);
        fx[FX_MAXTERM] = __float_as_uint(mt);
        fx[FX_BX] = __float_as_uint(red[0]);
        fx[FX_COUNT] = 0u;
    }
}

// ----------------------------------------------------------------------------- clusters
// Transposed stores are made cluster-wide: the C CTAs of a thread-block cluster hold C x RB
// consecutive rows (or columns) in their shared memory; after a cluster barrier each CTA
// writes 1/C of the outputs for all C x RB of them, reading its partners' rows through
// distributed shared memory, so that every global write is C x RB x 8 contiguous bytes
// (32 bytes, one whole sector, for C x RB = 4) instead of RB x 8.
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// a barrier that orders no memory: all its arrivals' remote reads have returned already
__device__ __forceinline__ void cluster_sync_relaxed() {
    asm volatile("barrier.cluster.arrive.relaxed.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t dsmem_map(const void* ptr, uint32_t rank) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(ptr);
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ float2 dsmem_ld2(uint32_t addr) {
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
    return v;
}

// The oversampled transforms: one L = 2N point transform per row (16 values per thread,
// T = L/16 = N/8 threads).  Forward: the centred N samples (c = j - N/2 in [-N/2, N/2)) sit
// at positions c mod L of the zero-padded input, i.e. thread slots m < 4 (c = t + T m) and
// m >= 12 (c = t + T m - L); the other slots are zero.  Inverse: of the L outputs only
// c mod L with c in [-N/2, N/2) (the crop) are kept.

// The thread slots m of the kept (or non-zero) half: m = 0 .. 3 and 12 .. 15, known at compile
// time, so that a pruned last stage and the staging skip the others.
__host__ __device__ constexpr int kept_slot(int q) { return q < 4 ? q : q + 8; }

// Which steps of a transposed store a warp takes part in: its values of one step share a uv-tile
// (at most 16 in a row, aligned), so lane i asks for step i and a ballot tells every lane.
struct KeepAll {
    __device__ bool operator()(int) const { return true; }
};
template <int IT, class Keep, class At>
__device__ __forceinline__ uint32_t kept_steps(Keep keep, At at) {
    static_assert(IT <= 32, "one lane per step");
    if constexpr (std::is_same<Keep, KeepAll>::value) {
        return 0xffffffffu;
    } else {
        const int lane = threadIdx.x & 31;
        return __ballot_sync(0xffffffffu, lane < IT && keep(at(lane)));
    }
}

// Transposed store of a CTA's (C = 1) or a cluster's (C > 1) rows: output row dst(kk) of
// `out` (leading dimension ld) gets, at columns [r0, r0 + C RB), value src(kk) of each of
// the C RB rows, for the nk kept values kk with keep(kk) (the others are not written).  With C > 1, after a cluster barrier each CTA
// writes nk / C of them for all the cluster's rows, reading partners' rows through
// distributed shared memory (32-byte writes for C RB = 4).
template <int RB, int C, int SR, int NK, int THREADS, class Src, class Dst, class Keep>
__device__ __forceinline__ void transposed_store(float2* smem, Src src, Dst dst, Keep keep, float2* out, size_t ld,
                                                 int r0_block) {  // r0_block: this CTA's first row
    if constexpr (C == 1) {
        __syncthreads();
        constexpr int NP = RB / 2, IT = NK * NP / THREADS;
        static_assert(NK * NP % THREADS == 0 && NP >= 2, "a warp holds at most 16 values");
        const uint32_t on = kept_steps<IT>(keep, [](int i) { return (int)((threadIdx.x & ~31u) + i * THREADS) / NP; });
#pragma unroll
        for (int i = 0; i < IT; ++i) {
            const int e = threadIdx.x + i * THREADS, kk = e / NP, q = e % NP;
            if (!((on >> i) & 1u)) continue;
            const int k = src(kk);
            const float2 a = smem[(2 * q) * SR + pidx(k)], b = smem[(2 * q + 1) * SR + pidx(k)];
            *reinterpret_cast<float4*>(&out[(size_t)dst(kk) * ld + r0_block + 2 * q]) = make_float4(a.x, a.y, b.x, b.y);
        }
        __syncthreads();
    } else {
        constexpr int NP = C * RB / 2, KPC = NK / C, STEP = THREADS / NP, IT = KPC / STEP;
        static_assert(THREADS % NP == 0 && STEP % 16 == 0 && KPC % STEP == 0, "a thread keeps one row pair");
        const int rank = (int)(blockIdx.x % C);
        const int rbase = r0_block - rank * RB;  // first row of the cluster
        const int q = threadIdx.x % NP;                   // rows 2q, 2q + 1 of the cluster
        // src and dst are shifts within a rank's range, so a thread's values are STEP apart
        const int kk0 = rank * KPC + threadIdx.x / NP;
        static_assert(NP >= 2, "a warp holds at most 16 values");
        uint32_t on = 0;
        if constexpr (C == 2) {
            on = kept_steps<IT>(keep, [&](int i) { return rank * KPC + (int)(threadIdx.x & ~31u) / NP + i * STEP; });
        } else {  // (at 2N = 8192 with the ballot: 5.16 instead of 5.10 ms of forward rows)
#pragma unroll
            for (int it = 0; it < IT; ++it) on |= (keep(kk0 + it * STEP) ? 1u : 0u) << it;
        }
        const uint32_t off = (uint32_t)pidx(src(kk0)) * 8u;
        const uint32_t b0 = dsmem_map(smem + ((2 * q) % RB) * SR, (2 * q) / RB) + off;
        const uint32_t b1 = dsmem_map(smem + ((2 * q + 1) % RB) * SR, (2 * q + 1) / RB) + off;
        float2* o = out + (size_t)dst(kk0) * ld + rbase + 2 * q;
        cluster_sync_all();
#pragma unroll
        for (int it = 0; it < IT; ++it) {
            if ((on >> it) & 1u) {
                const float2 a = dsmem_ld2(b0 + padded16(it * STEP) * 8), b = dsmem_ld2(b1 + padded16(it * STEP) * 8);
                *reinterpret_cast<float4*>(o + (size_t)(it * STEP) * ld) = make_float4(a.x, a.y, b.x, b.y);
            }
        }
        cluster_sync_relaxed();  // partners are done reading before the block may exit
    }
}

// ----------------------------------------------------------------------------- row selection
// The column passes transform only the grid rows u of uv-tile rows holding a needed tile
// (tiles no footprint of the bin reaches are neither stored nor read): block b takes rows
// [row[b / bpt] * RG bpt + (b % bpt) RG, + RG), bpt = TS / RG blocks per tile row.  A
// cluster's blocks stay within one tile row (bpt is a multiple of C).  With on = 0 block b
// takes rows [b RG, + RG).  `bits` marks the selected tile rows for the last pass.
struct RowSel {
    int on, bpt, shift;
    uint32_t bits[8];
    uint16_t row[256];
};

__device__ __forceinline__ int sel_row0(const RowSel& sel, int b, int rows_per_blk) {
    return sel.on ? ((int)sel.row[b / sel.bpt] * sel.bpt + b % sel.bpt) * rows_per_blk : b * rows_per_blk;
}

// ----------------------------------------------------------------------------- jobs
// A pass over one (plan, w-bin) is a job.  A launch covers one job (the applies of a plan,
// bin after bin: the job's arguments by value) or a table of jobs of the same transform
// shape (a wideband batch, every channel's every bin in one launch per pass): job j owns
// the launch's blocks [first[j], first[j + 1]), and a block finds its job (job_of) and
// then runs as in a one-job launch, with its block index within the job.
// The image pointer of a rows job counts from the launch's `img` bytes: 0 with the image's
// address in the job, or the image's address with null jobs (a plan's tables, whose images
// come with the call).
struct RowsJob {          // a rows pass: image rows -> transposed half transforms, or back
    const float2* in;
    float2* out;
    ZArgs z;
    RowSel sel;
};
struct ColsJob {          // a cols pass over the selected grid rows
    const float2* in;
    float2* out;
    const uint8_t* need;  // [tu * ntv + tv] of the job's bin: the tile is read or stored
    RowSel sel;
};
template <class J>
struct JobTable {
    const J* jobs;
    const int* first;     // njobs + 1 block offsets (multiples of the cluster size)
    int njobs;
};

// A table's image pointer counts from img (see RowsJob).
template <bool TABLE, class T>
__device__ __forceinline__ T* at_image(T* p, int64_t img) {
    if constexpr (TABLE) return reinterpret_cast<T*>(reinterpret_cast<uintptr_t>(p) + (uintptr_t)img);
    else return p;
}

// This block's job and its block index b within the job.
template <bool TABLE, class J>
__device__ __forceinline__ const J& block_job(const J& one, const JobTable<J>& tab, int& b) {
    b = (int)blockIdx.x;
    if constexpr (TABLE) {
        const int j = job_of(tab.first, tab.njobs, b);
        b -= __ldg(tab.first + j);
        return tab.jobs[j];
    } else {
        (void)tab;
        return one;
    }
}

// Which of a warp's values lie in needed tiles, as one bit per value m < n: the warp's 32
// consecutive cells at pos(m) share a tile (sides 32 and 64), so lane m reads that tile's flag
// and a ballot hands all of them to every lane.  With the flags staged in shared memory behind a
// barrier and a load per value, 4096^2/24M took 3.20 instead of 2.91 ms of forward cols and 5.46
// instead of 5.26 of inverse cols + fold, 2048^2/10M 0.668 for 0.606 and 1.33 for 1.25.
template <class Pos>
__device__ __forceinline__ uint32_t needed(const uint8_t* __restrict__ need_row, int shift, int n, Pos pos) {
    const int lane = threadIdx.x & 31;
    return __ballot_sync(0xffffffffu, lane < n && __ldg(need_row + (pos(lane) >> shift)) != 0);
}

// Likewise which of a warp's values lie in selected tile rows (the bits of a job table are loads
// from memory: one per lane instead of one per value and thread; iteration at 256^2, 4 bins, inverse
// rows 15.4 -> 10.2 us; 2048^2/10M 0.563 -> 0.543 ms, 4096^2/24M 4.05 -> 3.98).
template <class Pos>
__device__ __forceinline__ uint32_t selected(const RowSel& sel, int n, Pos pos) {
    if (!sel.on) return 0xffffffffu;
    const int lane = threadIdx.x & 31, tr = pos(lane) >> sel.shift;
    return __ballot_sync(0xffffffffu, lane < n && ((sel.bits[tr >> 5] >> (tr & 31)) & 1u));
}

// ----------------------------------------------------------------------------- forward rows
// grid: ny / RB blocks of RB * N/8 threads per job; block b transforms image rows
// [b RB, b RB + RB): Z_p times the row, zero-padded to 2N, DFT along l; row i of the result
// is column i of At (At[k][i], k < 2N).
template <int N, int RB, int C, bool TABLE>
__global__ void __launch_bounds__(RB * N / 8, (1024 / (RB * N / 8)) > 0 ? (1024 / (RB * N / 8)) : 1)
    fwd_rows_kernel(const __grid_constant__ RowsJob one, const JobTable<RowsJob> tab, int64_t img, int ny,
                    const float2* __restrict__ tws) {
    constexpr int L = 2 * N, T = L / 16, SR = L + L / 16;
    extern __shared__ float2 smem[];
    int bk;
    const RowsJob& J = block_job<TABLE>(one, tab, bk);
    const float2* __restrict__ x = at_image<TABLE>(J.in, img);
    const ZArgs z = J.z;
    const RowSel& sel = J.sel;
    const int g = threadIdx.x / T, t = threadIdx.x % T;
    float2* sm = smem + g * SR;
    const int i = bk * RB + g;
    const int ic = i - ny / 2;
    const float2* xr = x + (size_t)i * N;
    float2 v[16];
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        if (m >= 4 && m < 12) {
            v[m] = make_float2(0.f, 0.f);
        } else {
            const int p = t + T * m;
            const int jc = m < 4 ? p : p - L;
            const int j = jc + N / 2;
            v[m] = cmul(__ldg(&xr[j]), z_factor(z, i, j, ic, jc));
        }
    }
    fft_n<L, false, true>(v, sm, t, tws);
#pragma unroll
    for (int m = 0; m < 16; ++m) sm[pidx(t) + padded16(T * m)] = v[out_slot<L>(m)];
    // rows k of At the forward column pass does not transform are not stored
    transposed_store<RB, C, SR, L, RB * N / 8>(
        smem, [](int kk) { return kk; }, [](int kk) { return kk; },
        [&](int kk) { return !sel.on || ((sel.bits[(kk >> sel.shift) >> 5] >> ((kk >> sel.shift) & 31)) & 1u); },
        J.out, (size_t)ny, bk * RB);
}

// ----------------------------------------------------------------------------- forward cols
// grid: the selected grid rows / RG blocks per job; row u of At (N = ny samples) ->
// X[u][0 .. 2N).  Tiles of X that no active patch reads are not stored.
template <int N, int RG, bool TABLE>
__global__ void __launch_bounds__(RG * N / 8, (1024 / (RG * N / 8)) > 0 ? (1024 / (RG * N / 8)) : 1)
    fwd_cols_kernel(const __grid_constant__ ColsJob one, const JobTable<ColsJob> tab, int shift,
                    const float2* __restrict__ tws) {
    constexpr int L = 2 * N, T = L / 16, SR = L + L / 16;
    extern __shared__ float2 smem[];
    int bk;
    const ColsJob& J = block_job<TABLE>(one, tab, bk);
    const uint8_t* __restrict__ need = J.need;
    const int ntv = L >> shift;
    uint8_t* s_need = reinterpret_cast<uint8_t*>(smem + RG * SR);
    const int g = threadIdx.x / T, t = threadIdx.x % T;
    float2* sm = smem + g * SR;
    const int r0 = sel_row0(J.sel, bk, RG);
    const size_t u = (size_t)r0 + g;
    const float2* __restrict__ in = J.in + u * N;
    float2* __restrict__ out = J.out + u * L;
    uint32_t on = 0;
    if constexpr (T >= 32) {
        on = needed(need + (u >> shift) * ntv, shift, 16, [&](int m) { return (t & ~31) + T * m; });
    } else {
        for (int e = threadIdx.x; e < RG * ntv; e += blockDim.x) {
            const size_t uu = (size_t)r0 + e / ntv;
            s_need[e] = need[(uu >> shift) * ntv + e % ntv];
        }
    }
    float2 v[16];
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        if (m >= 4 && m < 12) {
            v[m] = make_float2(0.f, 0.f);
        } else {
            const int p = t + T * m;
            const int jc = m < 4 ? p : p - L;
            v[m] = __ldg(&in[jc + N / 2]);
        }
    }
    if constexpr (T < 32) __syncthreads();
    fft_n<L, false, true>(v, sm, t, tws);
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        const int k = t + T * m;
        if (T >= 32 ? (on >> m) & 1u : s_need[g * ntv + (k >> shift)]) out[k] = v[out_slot<L>(m)];
    }
}

// The same pass for N = 4096 with 256 threads of 32 points per row (one row per block).
template <bool TABLE>
__global__ void __launch_bounds__(256, 2)
    fwd_cols32_kernel(const __grid_constant__ ColsJob one, const JobTable<ColsJob> tab, int shift,
                      const float2* __restrict__ tw) {
    constexpr int N = 4096, L = 8192;
    extern __shared__ float2 smem[];
    int bk;
    const ColsJob& J = block_job<TABLE>(one, tab, bk);
    const uint8_t* __restrict__ need = J.need;
    const int ntv = L >> shift;
    const int t = threadIdx.x;
    const int r0 = sel_row0(J.sel, bk, 1);
    const size_t u = (size_t)r0;
    const float2* __restrict__ in = J.in + u * N;
    float2* __restrict__ out = J.out + u * L;
    const uint32_t on = needed(need + (u >> shift) * ntv, shift, 32, [&](int q) { return out_k32(t & ~31, q); });
    float2 v[32];
#pragma unroll
    for (int m = 0; m < 32; ++m) {
        if (m >= 8 && m < 24) {
            v[m] = make_float2(0.f, 0.f);
        } else {
            const int p = t + 256 * m;
            const int jc = m < 8 ? p : p - L;
            v[m] = __ldg(&in[jc + N / 2]);
        }
    }
    fft8192_32<false, true>(v, smem, t, tw);
#pragma unroll
    for (int q = 0; q < 32; ++q) {
        const int k = out_k32(t, q);
        if ((on >> q) & 1u) out[k] = v[q];
    }
}

// Inverse cols, N = 4096, 256 threads of 32 points per row, 4-CTA clusters for the store.
template <bool TABLE>
__global__ void __launch_bounds__(256, 2)
    inv_cols32_kernel(const __grid_constant__ ColsJob one, const JobTable<ColsJob> tab, int gx, int shift,
                      const float2* __restrict__ tw) {
    constexpr int N = 4096, L = 8192, SR = L + L / 16;
    extern __shared__ float2 smem[];
    int bk;
    const ColsJob& J = block_job<TABLE>(one, tab, bk);
    const uint8_t* __restrict__ need = J.need;
    const int ntv = L >> shift;
    const int t = threadIdx.x;
    const int r0 = sel_row0(J.sel, bk, 1);
    const int u = r0;
    const uint32_t on = needed(need + (size_t)(u >> shift) * ntv, shift, 32, [&](int m) { return (t & ~31) + 256 * m; });
    const float2* __restrict__ in = J.in + (size_t)u * L;
    float2 v[32];
#pragma unroll
    for (int m = 0; m < 32; ++m) {
        const int p = t + 256 * m;
        v[m] = (on >> m) & 1u ? __ldg(&in[p]) : make_float2(0.f, 0.f);
    }
    fft8192_32<true, false>(v, smem, t, tw);
#pragma unroll
    for (int q = 0; q < 32; ++q)  // outputs k < N / 2 and k >= 3 N / 2: q mod 16 < 4 and >= 12
        if ((q & 15) < 4 || (q & 15) >= 12) smem[pidx(t) + padded16(out_k32(0, q))] = v[q];
    transposed_store<1, 4, SR, N, 256>(
        smem, [](int kk) { return kk < N / 2 ? kk : kk + N; },
        [](int kk) { return kk < N / 2 ? kk + N / 2 : kk - N / 2; }, KeepAll{}, J.out, (size_t)gx, r0);
}

// ----------------------------------------------------------------------------- patch fold
// The gridded grid Xh of one bin is the sum of the accumulator patches of its active
// uv-tiles: a cell gets its own tile's patch and the halos of the tiles before it along u
// and v.  One block folds one needed tile (TS x TS cells) and writes it to Xh; tiles no
// patch reaches are never written and read as zero by the inverse transform.
struct FoldArgs {
    const float2* patch;   // [slot][PW * PW]
    const FoldRec* recs;   // needed tiles of this bin
    float2* Xh;            // [gx][gy]
    int PW, gy;
};

// TS: the tile side (32 or 64) as a compile-time constant, so the cell indexing is shifts.
// A thread folds pairs of cells of one pair of columns (16-byte loads and stores): the grid step
// writes its boxes widened to whole pairs of columns (the added cells hold zeros), so a pair is
// in a box or not as a whole.  The sources' places and ranges come from the tile's record: with
// slots and boxes looked up and clipped here, one cell per load and 64-bit offsets per cell the
// kernel was bound by its index arithmetic.  Measured, one cell per load / pairs / pairs and
// records: four bins of 1024^2/2M 98 / 67 / 55 us (4.9 TB/s of boxes and tiles).
template <bool TABLE, int TS>
__global__ void __launch_bounds__(256) fold_kernel(const __grid_constant__ FoldArgs one, const JobTable<FoldArgs> tab) {
    int bk;
    const FoldArgs& F = block_job<TABLE>(one, tab, bk);
    constexpr int ROW = TS / 2, STEP = 256 / ROW;  // pairs per row, rows per pass of the block
    const int4 off = __ldg(reinterpret_cast<const int4*>(F.recs + bk));
    const uint4 rng = __ldg(reinterpret_cast<const uint4*>(F.recs + bk) + 1);
    const int a = threadIdx.x / ROW, b = 2 * (threadIdx.x % ROW), PW = F.PW;
    // a source's first row and rows in this pair of columns, and the address of its row 0 there
    struct Src {
        const float2* p;
        int a0, na;
    };
    auto src = [&](int o, uint32_t x) {
        const int a0 = (int)(x & 127u), a1 = (int)((x >> 7) & 127u), b0 = (int)((x >> 14) & 127u);
        const int b1 = (int)((x >> 21) & 127u);
        return Src{F.patch + 2 * (int64_t)o + b, a0, b >= b0 && b < b1 ? a1 - a0 : 0};
    };
    const Src s00 = src(off.x, rng.x), s10 = src(off.y, rng.y), s01 = src(off.z, rng.z), s11 = src(off.w, rng.w);
    const int tu = (int)(rng.x >> 28 | (rng.y >> 28) << 4), tv = (int)(rng.z >> 28 | (rng.w >> 28) << 4);
    float2* __restrict__ Xh = F.Xh + (size_t)(tu * TS + a) * F.gy + tv * TS + b;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
    for (int r = 0; r < TS; r += STEP) {
        // the sources' pairs, then their sum in a fixed order
        bool k00 = (unsigned)(a + r - s00.a0) < (unsigned)s00.na, k10 = (unsigned)(a + r - s10.a0) < (unsigned)s10.na;
        bool k01 = (unsigned)(a + r - s01.a0) < (unsigned)s01.na, k11 = (unsigned)(a + r - s11.a0) < (unsigned)s11.na;
        const int o = (a + r) * PW;
        float4 v = k00 ? __ldg(reinterpret_cast<const float4*>(s00.p + o)) : zero;
        const float4 x10 = k10 ? __ldg(reinterpret_cast<const float4*>(s10.p + o)) : zero;
        const float4 x01 = k01 ? __ldg(reinterpret_cast<const float4*>(s01.p + o)) : zero;
        const float4 x11 = k11 ? __ldg(reinterpret_cast<const float4*>(s11.p + o)) : zero;
        auto add = [&](bool k, const float4& x) {
            if (k) v = make_float4(v.x + x.x, v.y + x.y, v.z + x.z, v.w + x.w);
        };
        add(k10, x10);
        add(k01, x01);
        add(k11, x11);
        *reinterpret_cast<float4*>(Xh + (size_t)r * F.gy) = v;
    }
}

// ----------------------------------------------------------------------------- inverse cols
// grid: the selected grid rows / RB blocks per job; rows u of Xh (2N cells along v; cells
// of tiles without a mark in need[] are zero and not read) -> B[i][u] for the N image rows i.
template <int N, int RB, int C, bool TABLE>
__global__ void __launch_bounds__(RB * N / 8, (1024 / (RB * N / 8)) > 0 ? (1024 / (RB * N / 8)) : 1)
    inv_cols_kernel(const __grid_constant__ ColsJob one, const JobTable<ColsJob> tab, int gx, int shift,
                    const float2* __restrict__ tws) {
    constexpr int L = 2 * N, T = L / 16, SR = L + L / 16;
    extern __shared__ float2 smem[];
    int bk;
    const ColsJob& J = block_job<TABLE>(one, tab, bk);
    const uint8_t* __restrict__ need = J.need;
    const int ntv = L >> shift;
    uint8_t* s_need = reinterpret_cast<uint8_t*>(smem + RB * SR);
    const int g = threadIdx.x / T, t = threadIdx.x % T;
    float2* sm = smem + g * SR;
    const int r0 = sel_row0(J.sel, bk, RB);
    const int u = r0 + g;
    uint32_t on = 0;
    if constexpr (T >= 32) {
        on = needed(need + (size_t)(u >> shift) * ntv, shift, 16, [&](int m) { return (t & ~31) + T * m; });
    } else {
        for (int e = threadIdx.x; e < RB * ntv; e += blockDim.x) {
            const int uu = r0 + e / ntv;
            s_need[e] = need[(size_t)(uu >> shift) * ntv + e % ntv];
        }
        __syncthreads();
    }
    const float2* __restrict__ in = J.in + (size_t)u * L;
    float2 v[16];
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        const int p = t + T * m;
        v[m] = (T >= 32 ? (on >> m) & 1u : s_need[g * ntv + (p >> shift)]) ? __ldg(&in[p]) : make_float2(0.f, 0.f);
    }
    fft_n<L, true>(v, sm, t, tws);
#pragma unroll
    for (int q = 0; q < 8; ++q)
        sm[pidx(t) + padded16(T * kept_slot(q))] = v[out_slot<L>(kept_slot(q))];
    // kept output kk < N: k = kk (kk < N/2) or kk + N; image row i = (k < N/2 ? k : k - L) + N/2
    transposed_store<RB, C, SR, N, RB * N / 8>(
        smem, [](int kk) { return kk < N / 2 ? kk : kk + N; },
        [](int kk) { return kk < N / 2 ? kk + N / 2 : kk - N / 2; }, KeepAll{}, J.out, (size_t)gx,
        r0);
}

// ----------------------------------------------------------------------------- inverse rows
// grid: ny / RG blocks; row i of B (2N cells along u) -> out[i][0 .. N) * conj(Z_p).
// With a table the grid is groups x ny / RG blocks: group c (the w-bins of one channel of a
// batch, jobs [group[c], group[c + 1])) has its bins summed into its image by the same
// block, one bin after the other (Sigma_p of Eq. 7 without a race or a second pass).
template <int N, int RG, bool TABLE>
__global__ void __launch_bounds__(RG * N / 8, (1024 / (RG * N / 8)) > 0 ? (1024 / (RG * N / 8)) : 1)
    inv_rows_kernel(const __grid_constant__ RowsJob one, const JobTable<RowsJob> tab, const int* __restrict__ group,
                    int64_t img, int ny, int accumulate, int real_only, const float2* __restrict__ tws) {
    constexpr int L = 2 * N, T = L / 16, SR = L + L / 16;
    extern __shared__ float2 smem[];
    const int g = threadIdx.x / T, t = threadIdx.x % T;
    float2* sm = smem + g * SR;
    int bk = (int)blockIdx.x, j0 = 0, j1 = 1;
    if constexpr (TABLE) {
        const int per = ny / RG, c = bk / per;
        bk -= c * per;
        j0 = __ldg(group + c);
        j1 = __ldg(group + c + 1);
    }
    const int i = bk * RG + g;
    const int ic = i - ny / 2;
    for (int jj = j0; jj < j1; ++jj) {
        const RowsJob& J = TABLE ? tab.jobs[jj] : one;
        const RowSel& sel = J.sel;
        const ZArgs z = J.z;
        const float2* __restrict__ in = J.in + (size_t)i * L;
        float2* __restrict__ orow = at_image<TABLE>(J.out, img) + (size_t)i * N;
        const int acc = accumulate || jj > j0;
        float2 v[16];
        // columns u of tile rows the inverse column pass skipped are zero (not stored)
        uint32_t keep = 0xffffu;
        if constexpr (T >= 32) {
            keep = selected(sel, 16, [&](int m) { return (t & ~31) + T * m; });
        } else if (sel.on) {
            keep = 0;
#pragma unroll
            for (int m = 0; m < 16; ++m) {
                const int tr = (t + T * m) >> sel.shift;
                keep |= ((sel.bits[tr >> 5] >> (tr & 31)) & 1u) << m;
            }
        }
#pragma unroll
        for (int m = 0; m < 16; ++m) v[m] = (keep >> m) & 1u ? __ldg(&in[t + T * m]) : make_float2(0.f, 0.f);
        fft_n<L, true>(v, sm, t, tws);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int m = kept_slot(q), jc = t + T * m - (m < 4 ? 0 : L);
            const int j = jc + N / 2;
            float2 val = cmulc(v[out_slot<L>(m)], z_factor(z, i, j, ic, jc));
            if (acc) val = cadd<false>(val, orow[j]);
            if (real_only) val.y = 0.f;
            orow[j] = val;
        }
        // the next bin's first stage rewrites the exchange buffer this one's last stage read
        if (jj + 1 < j1) __syncthreads();
    }
}

// The same pass with the bins of a group side by side: a block of 4096 / N slots takes
// 4096 / N / BP image rows, BP bins of each at a time (BP = 1 << lb slots), whose products meet in
// shared memory and are summed there in the order of the bins, so the sums are those of
// inv_rows_kernel bit for bit.  For launches whose blocks, each with its bins one after the
// other, would not fill the GPU (N <= 512; four bins of 256^2 22.6 -> 15.0 us, of 512^2 24.8 ->
// 15.8 us; at 1024^2, with four rows per block, it was slower: 0.164 -> 0.172 ms per apply).
template <int N, int RG>
__global__ void __launch_bounds__(RG * N / 8, 2)
    inv_rows_bins_kernel(const JobTable<RowsJob> tab, const int* __restrict__ group, int64_t img, int ny,
                         int accumulate, int real_only, int lb, const float2* __restrict__ tws) {
    constexpr int L = 2 * N, T = L / 16, SR = L + L / 16, THREADS = RG * N / 8;
    extern __shared__ float2 smem[];
    const int g = threadIdx.x / T, t = threadIdx.x % T;
    float2* sm = smem + g * SR;
    const int BP = 1 << lb, rows = RG >> lb, per = ny / rows;
    const int c = (int)blockIdx.x / per, row0 = ((int)blockIdx.x - c * per) * rows;
    const int j0 = __ldg(group + c), j1 = __ldg(group + c + 1);
    const int i = row0 + (g >> lb), ic = i - ny / 2;
    float2* __restrict__ out = at_image<true>(tab.jobs[j0].out, img) + (size_t)row0 * N;
    for (int jc = j0; jc < j1; jc += BP) {
        const int nb = min(BP, j1 - jc);
        const bool on = (g & (BP - 1)) < nb;
        const RowsJob& J = tab.jobs[on ? jc + (g & (BP - 1)) : j0];
        const RowSel& sel = J.sel;
        const float2* __restrict__ in = J.in + (size_t)i * L;
        // (a warp's threads share a slot when a row has 32 threads or more)
        uint32_t sels = 0;
        if constexpr (T >= 32) sels = on ? selected(sel, 16, [&](int m) { return (t & ~31) + T * m; }) : 0u;
        float2 v[16];
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const int tr = (t + T * m) >> sel.shift;
            const bool keep = T >= 32 ? (sels >> m) & 1u : on && (!sel.on || ((sel.bits[tr >> 5] >> (tr & 31)) & 1u));
            v[m] = keep ? __ldg(&in[t + T * m]) : make_float2(0.f, 0.f);
        }
        fft_n<L, true, false, false>(v, sm, t, tws);
        const ZArgs z = J.z;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int m = kept_slot(q), jc2 = t + T * m - (m < 4 ? 0 : L);
            sm[jc2 + N / 2] = cmulc(v[out_slot<L>(m)], z_factor(z, i, jc2 + N / 2, ic, jc2));
        }
        __syncthreads();
        for (int e = threadIdx.x; e < rows * N; e += THREADS) {
            const float2* p = smem + (size_t)((e / N) << lb) * SR + e % N;
            float2 val = p[0];
            if (accumulate || jc > j0) val = cadd<false>(val, out[e]);
            for (int s = 1; s < nb; ++s) val = cadd<false>(p[s * SR], val);
            if (real_only) val.y = 0.f;
            out[e] = val;
        }
        __syncthreads();  // the next bins' first stage rewrites the slots
    }
}

// ----------------------------------------------------------------------------- Z_p
// Z_p(i, j) of every pixel, as the row passes apply it (for checking the w-phase).
__global__ void __launch_bounds__(256) zlayer_kernel(ZArgs z, int nx, int ny, float2* __restrict__ out) {
    const int64_t n = (int64_t)nx * ny;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(e / nx), j = (int)(e - (int64_t)i * nx);
        out[e] = z_factor(z, i, j, i - ny / 2, j - nx / 2);
    }
}

// ----------------------------------------------------------------------------- launchers
static ZArgs zargs(const rimo_plan* p, int bin) {
    ZArgs z;
    z.zq = p->tab.zq;
    z.zq_ld = p->nx / 2 + 1;
    z.w_hi = p->bins[bin].w_hi;
    z.w_lo = p->bins[bin].w_lo;
    return z;
}

void launch_zlayer(const rimo_plan* p, int bin, float2* out, cudaStream_t s) {
    const int64_t n = (int64_t)p->nx * p->ny;
    const int blocks = (int)std::min<int64_t>((n + 255) / 256, 8 * (int64_t)p->n_sm);
    zlayer_kernel<<<blocks, 256, 0, s>>>(zargs(p, bin), p->nx, p->ny, out);
}

void launch_image_bound(const rimo_plan* p, const float2* x, cudaStream_t s) {
    const int64_t n = (int64_t)p->nx * p->ny;
    const int blocks = (int)std::min<int64_t>((n + 255) / 256, std::min<int64_t>(FX_NPART, 4 * (int64_t)p->n_sm));
    image_bound_kernel<<<blocks, 256, 0, s>>>(x, p->nx, p->ny, zargs(p, 0), p->d_fx, p->d_status);
}

// rows per block of the 2N-point passes: 512 threads (N / 8 per row), ~70 KB of shared memory
template <int N>
static constexpr int rows_per_block() { return 4096 / N; }
// CTAs per cluster of the transposed-store passes: 4 rows per cluster, so that every write
// is one whole 32-byte sector (measured at 2N = 8192, forward-rows plus inverse-cols time
// per 32-bin apply: 13.1 ms with 4-row clusters, 14.4 ms with 8-row clusters and 64-byte
// writes, about 14.2 ms with 2-row clusters and 16-byte writes)
template <int RB>
static constexpr int cluster_of() { return RB >= 4 ? 1 : 4 / RB; }

template <class... KArgs, class... Args>
static void launch_clustered(void (*kernel)(KArgs...), int grid, int block, size_t smem, int C, cudaStream_t s,
                             Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    // clusters placed where the SMs are least loaded: forward rows 5.19 -> 5.10 ms and inverse cols +
    // fold 5.54 -> 5.46 per 4096^2/24M apply (equal at 2048^2; spread over the SMs: as the default)
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    at[1].id = cudaLaunchAttributeClusterSchedulingPolicyPreference;
    at[1].val.clusterSchedulingPolicyPreference = cudaClusterSchedulingPolicyLoadBalancing;
    cfg.numAttrs = 2;
    RIMO_CUDA(cudaLaunchKernelEx(&cfg, kernel, args...));
}

#define RIMO_DISPATCH_N(N_, CALL)                                                      \
    switch (N_) {                                                                      \
        case 64: { constexpr int NN = 64; CALL; } break;                               \
        case 128: { constexpr int NN = 128; CALL; } break;                             \
        case 256: { constexpr int NN = 256; CALL; } break;                             \
        case 512: { constexpr int NN = 512; CALL; } break;                             \
        case 1024: { constexpr int NN = 1024; CALL; } break;                           \
        case 2048: { constexpr int NN = 2048; CALL; } break;                           \
        case 4096: { constexpr int NN = 4096; CALL; } break;                           \
        default: fail(RIMO_ERR_INVALID_ARG, "unsupported transform length");           \
    }

// Row selection of `bin` for blocks of rpb rows (off when a block would span tile rows)
static RowSel row_sel(const rimo_plan* p, int bin, int rpb) {
    RowSel r;
    std::memset(&r, 0, sizeof(r));
    const auto& tr = p->trows[bin];
    const int ntu = p->gx / p->TS;
    if (rpb > p->TS || ntu > 256) return r;
    r.on = 1;
    r.bpt = p->TS / rpb;
    r.shift = p->TS == 64 ? 6 : 5;
    for (size_t i = 0; i < tr.size(); ++i) {
        r.row[i] = tr[i];
        r.bits[tr[i] >> 5] |= 1u << (tr[i] & 31);
    }
    return r;
}
static int sel_blocks(const rimo_plan* p, int bin, const RowSel& r, int rpb) {
    return r.on ? (int)p->trows[bin].size() * r.bpt : p->gx / rpb;
}
// the forward column pass's selection (blocks of 4096 / ny rows), shared with the forward
// row pass that writes its input
static RowSel fwd_sel(const rimo_plan* p, int bin) { return row_sel(p, bin, 4096 / p->ny); }
// the inverse column pass's selection (blocks of RB rows, clusters of C blocks; transform
// length 2 ny), shared with the inverse row pass that reads its output
static RowSel inv_sel(const rimo_plan* p, int bin) {
    const int RB = 4096 / p->ny, C = RB >= 4 ? 1 : 4 / RB;
    return row_sel(p, bin, C * RB <= p->TS ? RB : p->TS + 1);
}

static RowsJob rows_job(const rimo_plan* p, int bin, const float2* in, float2* out, const RowSel& sel) {
    RowsJob J;
    std::memset(&J, 0, sizeof(J));
    J.in = in;
    J.out = out;
    J.z = zargs(p, bin);
    J.sel = sel;
    return J;
}
static ColsJob cols_job(const rimo_plan* p, int bin, const float2* in, float2* out, const RowSel& sel) {
    ColsJob J;
    std::memset(&J, 0, sizeof(J));
    J.in = in;
    J.out = out;
    J.need = p->d_need + (size_t)bin * (size_t)(p->gx / p->TS) * (p->gy / p->TS);
    J.sel = sel;
    return J;
}
// the grid step's patches (one per active tile, merged, over their boxes) or, with `holo`, the
// holographic apply's (one per needed tile, whole): both cover [tile origin, + PW) on each axis
static FoldArgs fold_args(const rimo_plan* p, int bin, const float2* patch, bool holo, float2* Xh) {
    FoldArgs F;
    F.patch = patch;
    F.recs = (holo ? p->d_hfold : p->d_fold) + p->bins[bin].n0;
    F.Xh = Xh;
    F.PW = p->PW;
    F.gy = p->gy;
    return F;
}
static int tile_shift(int TS) { return TS == 64 ? 6 : 5; }

// One launch of each pass, for one job (TABLE = false: `one`) or a job table.
template <int N, bool TABLE>
static void run_fwd_rows(const RowsJob& one, const JobTable<RowsJob>& tab, int64_t img, int grid, int ny,
                         const float2* tws, cudaStream_t s) {
    constexpr int RB = rows_per_block<N>();
    constexpr int C = cluster_of<RB>();
    const size_t sm = (size_t)RB * (2 * N + N / 8) * sizeof(float2);
    if (grid == 0) return;
    if constexpr (C > 1) {
        if (grid % C != 0) fail(RIMO_ERR_UNSUPPORTED, "image rows do not fill the transposed-store clusters");
        set_smem(fwd_rows_kernel<N, RB, C, TABLE>, sm);
        launch_clustered(fwd_rows_kernel<N, RB, C, TABLE>, grid, RB * N / 8, sm, C, s, one, tab, img, ny, tws);
    } else {
        set_smem(fwd_rows_kernel<N, RB, 1, TABLE>, sm);
        fwd_rows_kernel<N, RB, 1, TABLE><<<grid, RB * N / 8, sm, s>>>(one, tab, img, ny, tws);
    }
}

// The column passes at 2N = 8192 use the 32-points-per-thread transform (tw32: the plan's
// tws32), the others the 16-point one.
template <int N, bool TABLE>
static void run_fwd_cols(const ColsJob& one, const JobTable<ColsJob>& tab, int grid, int TS, const float2* tws,
                         cudaStream_t s, const float2* tw32) {
    if constexpr (N == 4096) {
        if (!tw32) fail(RIMO_ERR_STATE, "8192-point column transforms without their twiddle table");
        const size_t sm = (size_t)(8192 + 8192 / 32) * sizeof(float2);
        if (grid == 0) return;
        set_smem(fwd_cols32_kernel<TABLE>, sm);
        fwd_cols32_kernel<TABLE><<<grid, 256, sm, s>>>(one, tab, tile_shift(TS), tw32);
    } else {
        constexpr int RG = rows_per_block<N>();
        const int ntv = (2 * N) / TS;
        const size_t sm = (size_t)RG * (2 * N + N / 8) * sizeof(float2) + (N < 256 ? (size_t)RG * ntv : 0);  // N < 256: flags
        if (grid == 0) return;
        set_smem(fwd_cols_kernel<N, RG, TABLE>, sm);
        fwd_cols_kernel<N, RG, TABLE><<<grid, RG * N / 8, sm, s>>>(one, tab, tile_shift(TS), tws);
    }
}

template <bool TABLE>
static void run_fold(const FoldArgs& one, const JobTable<FoldArgs>& tab, int grid, int TS, cudaStream_t s) {
    if (grid == 0) return;
    if (TS == 32) fold_kernel<TABLE, 32><<<grid, 256, 0, s>>>(one, tab);
    else fold_kernel<TABLE, 64><<<grid, 256, 0, s>>>(one, tab);  // plans hold TS = 32 or 64
}

template <int N, bool TABLE>
static void run_inv_cols(const ColsJob& one, const JobTable<ColsJob>& tab, int grid, int gx, int TS,
                         const float2* tws, cudaStream_t s, const float2* tw32) {
    if constexpr (N == 4096) {
        if (!tw32) fail(RIMO_ERR_STATE, "8192-point column transforms without their twiddle table");
        const size_t sm = (size_t)(8192 + 8192 / 16) * sizeof(float2);
        if (grid == 0) return;
        if (grid % 4 != 0) fail(RIMO_ERR_UNSUPPORTED, "grid rows do not fill the transposed-store clusters");
        set_smem(inv_cols32_kernel<TABLE>, sm);
        launch_clustered(inv_cols32_kernel<TABLE>, grid, 256, sm, 4, s, one, tab, gx, tile_shift(TS), tw32);
    } else {
        constexpr int RB = rows_per_block<N>();
        constexpr int C = cluster_of<RB>();
        const int ntv = (2 * N) / TS;
        const size_t sm = (size_t)RB * (2 * N + N / 8) * sizeof(float2) + (N < 256 ? (size_t)RB * ntv : 0);  // N < 256: flags
        if (grid == 0) return;
        // C consecutive blocks of a cluster stay in one tile row: TS / RB is a multiple of C
        if constexpr (C > 1) {
            if (grid % C != 0) fail(RIMO_ERR_UNSUPPORTED, "grid rows do not fill the transposed-store clusters");
            set_smem(inv_cols_kernel<N, RB, C, TABLE>, sm);
            launch_clustered(inv_cols_kernel<N, RB, C, TABLE>, grid, RB * N / 8, sm, C, s, one, tab, gx,
                             tile_shift(TS), tws);
        } else {
            set_smem(inv_cols_kernel<N, RB, 1, TABLE>, sm);
            inv_cols_kernel<N, RB, 1, TABLE><<<grid, RB * N / 8, sm, s>>>(one, tab, gx, tile_shift(TS), tws);
        }
    }
}

template <int N, bool TABLE>
static void run_inv_rows(const RowsJob& one, const JobTable<RowsJob>& tab, const int* group, int64_t img, int grid,
                         int ny, int acc, int re, const float2* tws, cudaStream_t s) {
    constexpr int RG = rows_per_block<N>();
    const size_t sm = (size_t)RG * (2 * N + N / 8) * sizeof(float2);
    if (grid == 0) return;
    set_smem(inv_rows_kernel<N, RG, TABLE>, sm);
    inv_rows_kernel<N, RG, TABLE><<<grid, RG * N / 8, sm, s>>>(one, tab, group, img, ny, acc, re, tws);
}

template <class J>
static JobTable<J> no_table() {
    JobTable<J> t;
    t.jobs = nullptr;
    t.first = nullptr;
    t.njobs = 0;
    return t;
}

template <int N>
static void fwd_rows(const rimo_plan* p, int bin, const float2* x, float2* At, cudaStream_t s) {
    run_fwd_rows<N, false>(rows_job(p, bin, x, At, fwd_sel(p, bin)), no_table<RowsJob>(), 0,
                           p->ny / rows_per_block<N>(), p->ny, p->tab.tws_x, s);
}

template <int N>
static void fwd_cols(const rimo_plan* p, int bin, const float2* At, float2* X, cudaStream_t s) {
    const RowSel sel = fwd_sel(p, bin);
    run_fwd_cols<N, false>(cols_job(p, bin, At, X, sel), no_table<ColsJob>(),
                           sel_blocks(p, bin, sel, rows_per_block<N>()), p->TS, p->tab.tws_y, s, p->tab.tws32);
}

template <int N>
static void inv_cols(const rimo_plan* p, int bin, bool holo, float2* B, cudaStream_t s) {
    const auto& br = p->bins[bin];
    run_fold<false>(fold_args(p, bin, holo ? p->d_hpatch : p->d_patch, holo, p->d_X),
                    no_table<FoldArgs>(), br.n1 - br.n0, p->TS, s);
    const RowSel sel = inv_sel(p, bin);
    run_inv_cols<N, false>(cols_job(p, bin, p->d_X, B, sel), no_table<ColsJob>(),
                           sel_blocks(p, bin, sel, rows_per_block<N>()), p->gx, p->TS, p->tab.tws_y, s, p->tab.tws32);
}

template <int N>
static void inv_rows(const rimo_plan* p, int bin, const float2* B, float2* out, int acc, int re,
                     cudaStream_t s) {
    run_inv_rows<N, false>(rows_job(p, bin, B, out, inv_sel(p, bin)), no_table<RowsJob>(), nullptr, 0,
                           p->ny / rows_per_block<N>(), p->ny, acc, re, p->tab.tws_x, s);
}

// ----------------------------------------------------------------------------- job tables
// The transform passes of a stage-batched apply: one launch per pass over every job.
struct WideFft {
    int nx = 0, ny = 0, gx = 0, TS = 0, ngroups = 0;
    int group_max = 0;     // jobs of the largest group
    const float2* tws_x = nullptr;
    const float2* tws_y = nullptr;
    const float2* tws32 = nullptr;
    struct Pass {
        void* jobs = nullptr;
        int* first = nullptr;
        int njobs = 0, blocks = 0;
    };
    Pass rows_fwd, cols_fwd, fold, cols_inv, rows_inv;
    int* group = nullptr;  // rows_inv: jobs of channel c are [group[c], group[c + 1])
    char* tables = nullptr;  // every table, one allocation
    ~WideFft() { cudaFree(tables); }
};

// Appends an array to the host image of the tables (256-byte aligned); its offset.
template <class T>
static size_t append(std::vector<char>& blob, const std::vector<T>& v) {
    const size_t at = (blob.size() + 255) & ~(size_t)255;
    blob.resize(at + v.size() * sizeof(T));
    if (!v.empty()) std::memcpy(blob.data() + at, v.data(), v.size() * sizeof(T));
    return at;
}

WideFft* wide_fft_create(const std::vector<WideJob>& jobs, const std::vector<const float2*>& x,
                         const std::vector<float2*>& out, cudaStream_t s, bool holographic) {
    if (jobs.empty()) fail(RIMO_ERR_INVALID_ARG, "no jobs");
    auto* w = new WideFft();
    try {
        const rimo_plan* p0 = jobs[0].p;
        w->nx = p0->nx;
        w->ny = p0->ny;
        w->gx = p0->gx;
        w->TS = p0->TS;
        w->tws_x = p0->tab.tws_x;
        w->tws_y = p0->tab.tws_y;
        w->tws32 = p0->tab.tws32;
        w->ngroups = (int)x.size();
        const int rb = 4096 / p0->nx, cb = 4096 / p0->ny;  // rows per block of the rows and the cols passes
        std::vector<RowsJob> rf, ri;
        std::vector<ColsJob> cf, ci;
        std::vector<FoldArgs> fo;
        std::vector<int> frf{0}, fcf{0}, ffo{0}, fci{0}, grp(w->ngroups + 1, 0);
        for (const WideJob& j : jobs) {
            const rimo_plan* p = j.p;
            const RowSel fs = fwd_sel(p, j.bin), is = inv_sel(p, j.bin);
            rf.push_back(rows_job(p, j.bin, x[j.group], j.AB, fs));
            frf.push_back(frf.back() + p->ny / rb);
            cf.push_back(cols_job(p, j.bin, j.AB, j.X, fs));
            fcf.push_back(fcf.back() + sel_blocks(p, j.bin, fs, cb));
            fo.push_back(fold_args(p, j.bin, j.patch, holographic, j.X));
            ffo.push_back(ffo.back() + (p->bins[j.bin].n1 - p->bins[j.bin].n0));
            ci.push_back(cols_job(p, j.bin, j.X, j.AB, is));
            fci.push_back(fci.back() + sel_blocks(p, j.bin, is, cb));
            ri.push_back(rows_job(p, j.bin, j.AB, out[j.group], is));
            grp[j.group + 1]++;
        }
        for (int c = 0; c < w->ngroups; ++c) w->group_max = std::max(w->group_max, grp[c + 1]);
        for (int c = 0; c < w->ngroups; ++c) grp[c + 1] += grp[c];
        std::vector<char> blob;
        std::vector<std::pair<WideFft::Pass*, std::pair<size_t, size_t>>> at;
        auto pass = [&](WideFft::Pass& ps, const auto& jobs, const std::vector<int>& first) {
            ps.njobs = (int)jobs.size();
            ps.blocks = first.back();
            const size_t a = append(blob, jobs);
            at.push_back({&ps, {a, append(blob, first)}});
        };
        pass(w->rows_fwd, rf, frf);
        pass(w->cols_fwd, cf, fcf);
        pass(w->fold, fo, ffo);
        pass(w->cols_inv, ci, fci);
        pass(w->rows_inv, ri, std::vector<int>{0, w->ngroups * (p0->ny / rb)});
        const size_t gat = append(blob, grp);
        RIMO_CUDA(device_malloc(&w->tables, blob.size()));
        RIMO_CUDA(cudaMemcpyAsync(w->tables, blob.data(), blob.size(), cudaMemcpyHostToDevice, s));
        for (auto& q : at) {
            q.first->jobs = w->tables + q.second.first;
            q.first->first = reinterpret_cast<int*>(w->tables + q.second.second);
        }
        w->group = reinterpret_cast<int*>(w->tables + gat);
        RIMO_CUDA(cudaStreamSynchronize(s));  // the host image goes out of scope
    } catch (...) {
        delete w;
        throw;
    }
    return w;
}

void wide_fft_destroy(WideFft* w) { delete w; }

template <class J>
static JobTable<J> table_of(const WideFft::Pass& ps) {
    JobTable<J> t;
    t.jobs = (const J*)ps.jobs;
    t.first = ps.first;
    t.njobs = ps.njobs;
    return t;
}

template <class J>
static J no_job() {
    J j;
    std::memset(&j, 0, sizeof(j));
    return j;
}

template <int N>
static void wide_rows_fwd(const WideFft* w, int64_t img, cudaStream_t s) {
    run_fwd_rows<N, true>(no_job<RowsJob>(), table_of<RowsJob>(w->rows_fwd), img, w->rows_fwd.blocks, w->ny, w->tws_x, s);
}
template <int N>
static void wide_cols_fwd(const WideFft* w, cudaStream_t s) {
    run_fwd_cols<N, true>(no_job<ColsJob>(), table_of<ColsJob>(w->cols_fwd), w->cols_fwd.blocks, w->TS, w->tws_y, s,
                          w->tws32);
}
template <int N>
static void wide_cols_inv(const WideFft* w, cudaStream_t s) {
    run_inv_cols<N, true>(no_job<ColsJob>(), table_of<ColsJob>(w->cols_inv), w->cols_inv.blocks, w->gx, w->TS, w->tws_y,
                          s, w->tws32);
}
template <int N>
static void wide_rows_inv(const WideFft* w, int64_t img, int acc, int real_only, cudaStream_t s) {
    // under two waves of 304 blocks, several bins side by side (more, smaller blocks' worth of rows)
    if constexpr (N <= 512) {
        constexpr int RG = rows_per_block<N>();
        int lb = 0;
        while ((RG >> (lb + 1)) >= 1 && (1 << lb) < w->group_max && (w->rows_inv.blocks << lb) < 608) ++lb;
        if (lb > 0) {
            const size_t sm = (size_t)RG * (2 * N + N / 8) * sizeof(float2);
            set_smem(inv_rows_bins_kernel<N, RG>, sm);
            inv_rows_bins_kernel<N, RG><<<w->rows_inv.blocks << lb, RG * N / 8, sm, s>>>(
                table_of<RowsJob>(w->rows_inv), w->group, img, w->ny, acc, real_only, lb, w->tws_x);
            return;
        }
    }
    run_inv_rows<N, true>(no_job<RowsJob>(), table_of<RowsJob>(w->rows_inv), w->group, img, w->rows_inv.blocks, w->ny,
                          acc, real_only, w->tws_x, s);
}

void wide_fwd_rows(const WideFft* w, const float2* x, cudaStream_t s) {
    RIMO_DISPATCH_N(w->nx, wide_rows_fwd<NN>(w, (int64_t)(uintptr_t)x, s));
}
void wide_fwd_cols(const WideFft* w, cudaStream_t s) { RIMO_DISPATCH_N(w->ny, wide_cols_fwd<NN>(w, s)); }
void wide_inv_cols(const WideFft* w, cudaStream_t s) {
    run_fold<true>(no_job<FoldArgs>(), table_of<FoldArgs>(w->fold), w->fold.blocks, w->TS, s);
    RIMO_DISPATCH_N(w->ny, wide_cols_inv<NN>(w, s));
}
void wide_inv_rows(const WideFft* w, float2* out, int acc, int real_only, cudaStream_t s) {
    RIMO_DISPATCH_N(w->nx, wide_rows_inv<NN>(w, (int64_t)(uintptr_t)out, acc, real_only, s));
}

void launch_fwd_rows(const rimo_plan* p, int bin, const float2* x, float2* At, cudaStream_t s) {
    RIMO_DISPATCH_N(p->nx, fwd_rows<NN>(p, bin, x, At, s));
}
void launch_fwd_cols(const rimo_plan* p, int bin, const float2* At, float2* X, cudaStream_t s) {
    RIMO_DISPATCH_N(p->ny, fwd_cols<NN>(p, bin, At, X, s));
}
void launch_inv_cols(const rimo_plan* p, int bin, float2* B, cudaStream_t s) {
    RIMO_DISPATCH_N(p->ny, inv_cols<NN>(p, bin, false, B, s));
}
void launch_inv_cols_from(const rimo_plan* p, int bin, bool holographic, float2* B, cudaStream_t s) {
    RIMO_DISPATCH_N(p->ny, inv_cols<NN>(p, bin, holographic, B, s));
}
void launch_inv_rows(const rimo_plan* p, int bin, const float2* B, float2* out, int accumulate,
                     int real_only, cudaStream_t s) {
    RIMO_DISPATCH_N(p->nx, inv_rows<NN>(p, bin, B, out, accumulate, real_only, s));
}

}  // namespace rimo
