// Kernel-surrogate MLP: (phi_u, phi_v, w_r) -> 128 -> GELU -> 128 -> GELU -> 450 reals
// (the 15 x 15 complex de-gridding tile of a visibility), trained on tiles of the exact
// method.  bf16 weights and activations feed tcgen05 tensor-core GEMMs with FP32
// accumulation in tensor memory; the elementwise steps (bias, GELU, loss, derivatives)
// run on the CUDA cores in FP32; Adam keeps FP32 master weights.
//
// Training step on a batch of B samples (B a multiple of 128):
//   Z1 = X W1^T + b1, H1 = bf16(gelu(Z1))              (CUDA cores, K = 3)
//   Z2 = H1 W2^T + b2, H2 = bf16(gelu(Z2))              (tcgen05)
//   Y  = H2 W3^T + b3, dY = 2 (Y - T) / (450 B)          (tcgen05, loss on CUDA cores)
//   dW3 = bf16(dY)^T H2, dH2 = bf16(dY) W3               (tcgen05, split-K over the batch)
//   dZ2 = dH2 gelu'(Z2); dW2 = bf16(dZ2)^T H1, dH1 = bf16(dZ2) W2
//   dZ1 = dH1 gelu'(Z1); dW1 = dZ1^T X                   (CUDA cores)
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <random>

#include "internal.h"
#include "mlp.h"
#include "tc.cuh"

namespace rimo {

typedef __nv_bfloat16 bf16;

// erf by the rational approximation of Abramowitz & Stegun (1964), eq. 7.1.26:
// erf(x) = 1 - t (a1 + t (a2 + t (a3 + t (a4 + t a5)))) e^{-x^2}, t = 1 / (1 + p x), x >= 0,
// |error| <= 1.5e-7 (odd extension to x < 0); one reciprocal and one exponential.
__device__ __forceinline__ float erf_as(float x) {
    const float ax = fabsf(x);
    const float t = __fdividef(1.f, fmaf(0.3275911f, ax, 1.f));
    const float poly =
        t * fmaf(t, fmaf(t, fmaf(t, fmaf(t, 1.061405429f, -1.453152027f), 1.421413741f), -0.284496736f), 0.254829592f);
    return copysignf(fmaf(-poly, __expf(-ax * ax), 1.f), x);
}
// GELU(z) = z Phi(z) = z (1 + erf(z / sqrt 2)) / 2 (the network's activation everywhere it
// runs forward: training, batched forward, tile generation)
__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.f + erf_as(z * 0.70710678118654752f)); }
// derivative of that same function (training follows the gradient of the GELU the network
// evaluates): with x = z / sqrt 2, E = erf_as and t, poly as in erf_as,
// dE/dx = e^{-x^2} (2 |x| poly(t) + p t^2 poly'(t)) (even in x), so
// GELU'(z) = (1 + E(x)) / 2 + z dE/dx / (2 sqrt 2).
__device__ __forceinline__ float gelu_grad_f(float z) {
    const float x = z * 0.70710678118654752f;
    const float ax = fabsf(x);
    const float t = __fdividef(1.f, fmaf(0.3275911f, ax, 1.f));
    const float poly =
        t * fmaf(t, fmaf(t, fmaf(t, fmaf(t, 1.061405429f, -1.453152027f), 1.421413741f), -0.284496736f), 0.254829592f);
    // d poly / dt = a1 + 2 a2 t + 3 a3 t^2 + 4 a4 t^3 + 5 a5 t^4
    const float dpoly =
        fmaf(t, fmaf(t, fmaf(t, fmaf(t, 5.f * 1.061405429f, 4.f * -1.453152027f), 3.f * 1.421413741f),
                     2.f * -0.284496736f),
             0.254829592f);
    const float e = __expf(-ax * ax);
    const float E = copysignf(fmaf(-poly, e, 1.f), x);
    const float dE = e * fmaf(2.f * ax, poly, 0.3275911f * t * t * dpoly);
    return fmaf(0.5f, 1.f + E, z * dE * 0.35355339059327376f);
}

__device__ __forceinline__ void mbar_init_(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tc::smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(tc::smem_addr(bar)), "r"(parity), "r"(100000u)
        : "memory");
    return ok != 0;
}
// bounded: at most 2^15 polls of <= 100 us each
__device__ __forceinline__ bool mbar_wait_(uint64_t* bar, uint32_t parity) {
    for (uint32_t it = 0; it < (1u << 15); ++it)
        if (mbar_try_wait_(bar, parity)) return true;
    return false;
}

// --------------------------------------------------------------------------------------
// C[m][n] (+)= sum_k A[m][k] B[n][k]: A (M x K) and B (N x K) bf16 row-major with K
// contiguous, C fp32.  Block: 128 threads, tile 128 (m) x nt (n), K staged in chunks of 64
// into shared memory in the canonical K-major layout by 16-byte asynchronous copies, two
// chunks deep; one thread issues the tcgen05.mma (K = 16 each), the accumulator lives in
// tensor memory.  These products are a few hundred MFLOP: they are bound by the latency of a
// block's chunks (loads, barrier, MMA, wait), so the copies of a chunk are all in flight at
// once and the tiles are small enough for 64 blocks or more (B = 4096, serialised: dY W3 67 -> 13 us,
// dY^T H2 91 -> 10 us, dZ2^T H1 93 -> 7 us, H1 W2^T 22 -> 7 us; loss and gradients with their copy to
// the host 460 -> 155 us).
constexpr int GEMM_KC = 64;
constexpr int GEMM_MAX_NT = 128;

struct GemmArgs {
    const bf16* A;
    const bf16* B;
    float* C;
    int lda, ldb, ldc;
    int M, N, K;
    int nt;      // columns of a tile: 64 or 128 (tensor-memory columns)
    int m_store; // rows of C stored
    int kspan;   // K range of one split (grid.z)
    int atomic;  // add into C (split-K) instead of storing
    int* status;
};

__device__ __forceinline__ void cp_async16_(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

__global__ void __launch_bounds__(128) gemm_tc_kernel(GemmArgs g) {
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ uint32_t tslot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n0 = blockIdx.x * g.nt, m0 = blockIdx.y * 128;
    const int nt = min(g.nt, g.N - n0);
    const int k_begin = blockIdx.z * g.kspan, k_end = min(g.K, k_begin + g.kspan);
    const uint32_t sA = tc::smem_addr(sm), stage = 128 * GEMM_KC * 2 + g.nt * GEMM_KC * 2;
    if (warp == 0) tc::tmem_alloc(&tslot, g.nt);
    if (tid == 0) {
        mbar_init_(&bar[0], 1);
        mbar_init_(&bar[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const int nch = (k_end - k_begin + GEMM_KC - 1) / GEMM_KC;
    // starts the copies of chunk c into its stage (c & 1): 128 rows of A, nt rows of B
    auto load = [&](int c) {
        const int k0 = k_begin + c * GEMM_KC, nv = min(GEMM_KC, k_end - k0) / 8;  // 16-byte vectors per row
        const uint32_t a = sA + (c & 1) * stage, b = a + 128 * GEMM_KC * 2;
        const int r0 = tid >> 3, v = tid & 7;
        if (v < nv) {
#pragma unroll
            for (int r = r0; r < 128; r += 16)
                cp_async16_(a + tc::kmajor_offset(r, v * 8, 128), g.A + (size_t)(m0 + r) * g.lda + k0 + v * 8);
            for (int r = r0; r < nt; r += 16)
                cp_async16_(b + tc::kmajor_offset(r, v * 8, nt), g.B + (size_t)(n0 + r) * g.ldb + k0 + v * 8);
        }
    };
    auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
    if (nch > 0) load(0);
    commit();
    if (nch > 1) load(1);
    commit();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tslot;
    const uint32_t idesc = tc::idesc_bf16_f32(128, nt);
    bool ok = true;
    for (int c = 0; c < nch; ++c) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");  // chunk c (the later group may be under way)
        tc::fence_proxy_async();
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
        if (tid == 0) {
            const uint32_t a = sA + (c & 1) * stage, b = a + 128 * GEMM_KC * 2;
            const int ns = min(GEMM_KC, k_end - k_begin - c * GEMM_KC) / 16;
            for (int s = 0; s < ns; ++s)
                tc::mma_bf16(tmem, tc::smem_desc(a + s * 128 * 32, 128, 256), tc::smem_desc(b + s * nt * 32, 128, 256),
                             idesc, (c > 0 || s > 0) ? 1u : 0u);
            tc::mma_commit(&bar[c & 1]);
        }
        if (c + 2 < nch || c + 1 == nch) {  // the stage is read: refill it, or the product is complete
            ok = mbar_wait_(&bar[c & 1], (c >> 1) & 1);
            if (__syncthreads_or(!ok)) {
                ok = false;
                break;
            }
            if (c + 2 < nch) load(c + 2);
        }
        commit();
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (!ok) {
        if (tid == 0) atomicExch(g.status, 2);
    } else if (nch > 0) {
        tc::fence_after_sync();
        const int row = m0 + 32 * warp + lane;
        for (int c = 0; c < nt; c += 16) {
            float v[16];
            tc::tmem_ld16(tmem + ((uint32_t)(32 * warp) << 16) + c, v);
            // (the warp that holds row m_store is whole again before its next, warp-collective load)
            if (row < g.m_store) {
                float4* dst = reinterpret_cast<float4*>(g.C + (size_t)row * g.ldc + n0 + c);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 x = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                    if (g.atomic) atomicAdd(dst + i, x);
                    else dst[i] = x;
                }
            }
            __syncwarp();
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) {
        tc::tmem_dealloc(tmem, g.nt);
        tc::tmem_relinquish();
    }
}

// nt: columns of a tile (64 or 128); splits: of K, added into C
static void gemm(const bf16* A, int lda, const bf16* B, int ldb, float* C, int ldc, int M, int N, int K, int nt,
                 int splits, bool atomic, int* status, cudaStream_t s, int m_store = 1 << 30) {
    constexpr int most = 2 * (128 + GEMM_MAX_NT) * GEMM_KC * 2;
    set_smem(gemm_tc_kernel, most);
    GemmArgs g;
    g.A = A;
    g.B = B;
    g.C = C;
    g.lda = lda;
    g.ldb = ldb;
    g.ldc = ldc;
    g.M = M;
    g.N = N;
    g.K = K;
    g.nt = nt;
    g.m_store = m_store;
    g.kspan = ((K / splits + 15) / 16) * 16;
    g.atomic = atomic ? 1 : 0;
    g.status = status;
    dim3 grid((N + nt - 1) / nt, M / 128, (K + g.kspan - 1) / g.kspan);
    gemm_tc_kernel<<<grid, 128, (size_t)2 * (128 + nt) * GEMM_KC * 2, s>>>(g);
}

// --------------------------------------------------------------------------------------
// elementwise steps
// Each takes EL_ROWS samples per block (256 threads: two samples at a time, one hidden unit per
// thread), reads and writes whole rows, and also writes the bf16 result transposed (through
// shared memory), the operand of the weight-gradient products.
constexpr int EL_ROWS = 16;

// block-wide transposed store of a [EL_ROWS][ncol <= 128] tile: dst[col0 + c][b0 + r]
__device__ __forceinline__ void store_transposed(const bf16 (*t)[MLP_H + 2], bf16* __restrict__ dst, size_t ld, int col0,
                                                 int ncol, int b0) {
    // a thread writes two samples (4 bytes) of a column: 8 threads per 32-byte column segment
    for (int e = threadIdx.x; e < ncol * (EL_ROWS / 2); e += 256) {
        const int c = e / (EL_ROWS / 2), r = 2 * (e % (EL_ROWS / 2));
        __nv_bfloat162 h;
        h.x = t[r][c];
        h.y = t[r + 1][c];
        *reinterpret_cast<__nv_bfloat162*>(dst + (size_t)(col0 + c) * ld + b0 + r) = h;
    }
}

__global__ void __launch_bounds__(256) l1_fwd_kernel(const float* __restrict__ X, const float* __restrict__ W1,
                                                     const float* __restrict__ b1, float* __restrict__ Z1,
                                                     bf16* __restrict__ H1, bf16* __restrict__ H1T, int B) {
    __shared__ bf16 t[EL_ROWS][MLP_H + 2];
    const int j = threadIdx.x % MLP_H, b0 = blockIdx.x * EL_ROWS;
    const float w0 = __bfloat162float(__float2bfloat16(W1[j * 3 + 0]));
    const float w1 = __bfloat162float(__float2bfloat16(W1[j * 3 + 1]));
    const float w2 = __bfloat162float(__float2bfloat16(W1[j * 3 + 2]));
    const float bias = b1[j];
#pragma unroll
    for (int r = threadIdx.x / MLP_H; r < EL_ROWS; r += 2) {
        const int b = b0 + r;
        const float z = fmaf(X[b * 3 + 0], w0, fmaf(X[b * 3 + 1], w1, fmaf(X[b * 3 + 2], w2, bias)));
        const bf16 h = __float2bfloat16(gelu_f(z));
        Z1[(size_t)b * MLP_H + j] = z;
        H1[(size_t)b * MLP_H + j] = h;
        t[r][j] = h;
    }
    if (!H1T) return;
    __syncthreads();
    store_transposed(t, H1T, B, 0, MLP_H, b0);
}

// Z (in place) += bias; H = bf16(gelu(Z)), and transposed when HT is given
__global__ void __launch_bounds__(256) act_fwd_kernel(float* __restrict__ Z, const float* __restrict__ bias,
                                                      bf16* __restrict__ H, bf16* __restrict__ HT, int B) {
    __shared__ bf16 t[EL_ROWS][MLP_H + 2];
    const int j = threadIdx.x % MLP_H, b0 = blockIdx.x * EL_ROWS;
    const float bj = bias[j];
#pragma unroll
    for (int r = threadIdx.x / MLP_H; r < EL_ROWS; r += 2) {
        const size_t e = (size_t)(b0 + r) * MLP_H + j;
        const float z = Z[e] + bj;
        const bf16 h = __float2bfloat16(gelu_f(z));
        Z[e] = z;
        H[e] = h;
        t[r][j] = h;
    }
    if (!HT) return;
    __syncthreads();
    store_transposed(t, HT, B, 0, MLP_H, b0);
}

// r = Y + b3 - T; loss += r^2; dY = 2 r / (450 B) as bf16 (columns 450 .. 463 zero) and its
// transpose; db3 += dY.  (One block per output column before: strided reads of every row,
// 72 us at B = 4096; now 9 us.)
__global__ void __launch_bounds__(256) loss_bwd_kernel(const float* __restrict__ Y, int ldy, const float* __restrict__ b3,
                                                       const float* __restrict__ T, bf16* __restrict__ dY, int ld_dy,
                                                       bf16* __restrict__ dYT, float* __restrict__ db3,
                                                       float* __restrict__ loss, int B) {
    __shared__ bf16 t[EL_ROWS][MLP_H + 2];
    __shared__ float part[256];
    const int jj = threadIdx.x % MLP_H, half = threadIdx.x / MLP_H, b0 = blockIdx.x * EL_ROWS;
    const float scale = 2.f / ((float)MLP_OUT * (float)B);
    float sq = 0.f;
    const int c0 = blockIdx.y * MLP_H, ncol = min(MLP_H, MLP_OUT_PAD - c0), j = c0 + jj;
    float db = 0.f;
    if (jj < ncol) {
        const bool real = j < MLP_OUT;
        const float bj = real ? b3[j] : 0.f;
#pragma unroll
        for (int r = half; r < EL_ROWS; r += 2) {
            const size_t b = (size_t)(b0 + r);
            const float res = real ? Y[b * ldy + j] + bj - T[b * MLP_OUT + j] : 0.f;
            const float d = scale * res;
            sq = fmaf(res, res, sq);
            db += d;
            const bf16 h = __float2bfloat16(d);
            dY[b * ld_dy + j] = h;
            t[r][jj] = h;
        }
    }
    part[threadIdx.x] = db;
    __syncthreads();
    if (half == 0 && j < MLP_OUT) atomicAdd(&db3[j], part[jj] + part[jj + MLP_H]);
    store_transposed(t, dYT, B, c0, ncol, b0);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = sq;
    __syncthreads();
    if (threadIdx.x == 0) {
        float v = 0.f;
        for (int w = 0; w < 8; ++w) v += part[w];
        atomicAdd(loss, v);
    }
}

// dZ = dH * gelu'(Z) -> bf16, and transposed; db += dZ (fp32)
__global__ void __launch_bounds__(256) act_bwd_kernel(const float* __restrict__ dH, const float* __restrict__ Z,
                                                      bf16* __restrict__ dZ, bf16* __restrict__ dZT,
                                                      float* __restrict__ db, int B) {
    __shared__ bf16 t[EL_ROWS][MLP_H + 2];
    __shared__ float part[256];
    const int j = threadIdx.x % MLP_H, half = threadIdx.x / MLP_H, b0 = blockIdx.x * EL_ROWS;
    float acc = 0.f;
#pragma unroll
    for (int r = half; r < EL_ROWS; r += 2) {
        const size_t e = (size_t)(b0 + r) * MLP_H + j;
        const float d = dH[e] * gelu_grad_f(Z[e]);
        const bf16 h = __float2bfloat16(d);
        dZ[e] = h;
        t[r][j] = h;
        acc += d;
    }
    part[threadIdx.x] = acc;
    __syncthreads();
    if (half == 0) atomicAdd(&db[j], part[j] + part[j + MLP_H]);
    store_transposed(t, dZT, B, 0, MLP_H, b0);
}

// dZ1 = dH1 * gelu'(Z1); dW1[j][i] += dZ1[b][j] X[b][i]; db1[j] += dZ1[b][j]
__global__ void __launch_bounds__(256) l1_bwd_kernel(const float* __restrict__ dH1, const float* __restrict__ Z1,
                                                     const float* __restrict__ X, float* __restrict__ dW1,
                                                     float* __restrict__ db1) {
    __shared__ float4 part[256];
    const int j = threadIdx.x % MLP_H, half = threadIdx.x / MLP_H, b0 = blockIdx.x * EL_ROWS;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int r = half; r < EL_ROWS; r += 2) {
        const int b = b0 + r;
        const size_t e = (size_t)b * MLP_H + j;
        const float d = dH1[e] * gelu_grad_f(Z1[e]);
        a.x = fmaf(d, X[b * 3 + 0], a.x);
        a.y = fmaf(d, X[b * 3 + 1], a.y);
        a.z = fmaf(d, X[b * 3 + 2], a.z);
        a.w += d;
    }
    part[threadIdx.x] = a;
    __syncthreads();
    if (half == 0) {
        const float4 q = part[j + MLP_H];
        atomicAdd(&dW1[j * 3 + 0], a.x + q.x);
        atomicAdd(&dW1[j * 3 + 1], a.y + q.y);
        atomicAdd(&dW1[j * 3 + 2], a.z + q.z);
        atomicAdd(&db1[j], a.w + q.w);
    }
}

// Adam on the FP32 masters, then the bf16 operand copies: W2 [128][128], W2^T, W3 [464][128]
// (rows >= 450 zero) and W3^T [128][512] (columns >= 450 zero).
__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, int n, float lr, float b1, float b2, float eps, float c1,
                            float c2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

__global__ void pack_weights_kernel(const float* __restrict__ P, bf16* __restrict__ W2b, bf16* __restrict__ W2Tb,
                                    bf16* __restrict__ W3b, bf16* __restrict__ W3Tb) {
    const float* W2 = P + MLP_OFF_W2;
    const float* W3 = P + MLP_OFF_W3;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < MLP_H * MLP_H) {
        const int r = i / MLP_H, c = i % MLP_H;
        const bf16 w = __float2bfloat16(W2[i]);
        W2b[i] = w;
        W2Tb[c * MLP_H + r] = w;
    }
    if (i < MLP_OUT_PAD * MLP_H) {
        const int r = i / MLP_H, c = i % MLP_H;
        const bf16 w = __float2bfloat16(r < MLP_OUT ? W3[r * MLP_H + c] : 0.f);
        W3b[i] = w;
        W3Tb[c * MLP_K3 + r] = w;
    }
    if (i < MLP_H * (MLP_K3 - MLP_OUT_PAD)) {
        const int c = i / (MLP_K3 - MLP_OUT_PAD), r = MLP_OUT_PAD + i % (MLP_K3 - MLP_OUT_PAD);
        W3Tb[c * MLP_K3 + r] = __float2bfloat16(0.f);
    }
}

// --------------------------------------------------------------------------------------
Mlp::~Mlp() {
    for (void* p : owned) cudaFree(p);
    cudaFree(acts);
    if (host) cudaFreeHost(host);
}

void* Mlp::alloc(size_t bytes) {
    void* p = nullptr;
    if (device_malloc(&p, bytes) != cudaSuccess) {
        cudaGetLastError();
        fail(RIMO_ERR_OOM, "cudaMalloc of " + std::to_string(bytes) + " bytes for the surrogate failed");
    }
    owned.push_back(p);
    return p;
}

void Mlp::init(uint64_t seed) {
    P = (float*)alloc(MLP_NPARAM * sizeof(float));
    // gradients, the batch loss and the status word: one buffer, one copy to the host
    G = (float*)alloc((MLP_NPARAM + 2) * sizeof(float));
    loss = G + MLP_NPARAM;
    status = reinterpret_cast<int*>(G + MLP_NPARAM + 1);
    if (cudaMallocHost(&host, (MLP_NPARAM + 2) * sizeof(float)) != cudaSuccess) {
        cudaGetLastError();
        fail(RIMO_ERR_OOM, "host buffer of the surrogate's gradients");
    }
    Mom = (float*)alloc(MLP_NPARAM * sizeof(float));
    Vel = (float*)alloc(MLP_NPARAM * sizeof(float));
    W2b = (bf16*)alloc(MLP_H * MLP_H * sizeof(bf16));
    W2Tb = (bf16*)alloc(MLP_H * MLP_H * sizeof(bf16));
    W3b = (bf16*)alloc(MLP_OUT_PAD * MLP_H * sizeof(bf16));
    W3Tb = (bf16*)alloc(MLP_H * MLP_K3 * sizeof(bf16));
    RIMO_CUDA(cudaMemset(status, 0, sizeof(int)));
    // uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) from a seeded host generator
    std::vector<float> h(MLP_NPARAM);
    std::mt19937_64 rng(seed);
    std::uniform_real_distribution<double> U(-1.0, 1.0);
    auto fill = [&](int off, int n, int fan_in) {
        const double a = 1.0 / std::sqrt((double)fan_in);
        for (int i = 0; i < n; ++i) h[off + i] = (float)(a * U(rng));
    };
    fill(MLP_OFF_W1, MLP_H * MLP_IN, MLP_IN);
    fill(MLP_OFF_B1, MLP_H, MLP_IN);
    fill(MLP_OFF_W2, MLP_H * MLP_H, MLP_H);
    fill(MLP_OFF_B2, MLP_H, MLP_H);
    fill(MLP_OFF_W3, MLP_OUT * MLP_H, MLP_H);
    fill(MLP_OFF_B3, MLP_OUT, MLP_H);
    set_params(h.data(), 0);
}

void Mlp::set_params(const float* host, cudaStream_t s) {
    RIMO_CUDA(cudaMemcpyAsync(P, host, MLP_NPARAM * sizeof(float), cudaMemcpyHostToDevice, s));
    RIMO_CUDA(cudaMemsetAsync(Mom, 0, MLP_NPARAM * sizeof(float), s));
    RIMO_CUDA(cudaMemsetAsync(Vel, 0, MLP_NPARAM * sizeof(float), s));
    t = 0;
    pack(s);
}

void Mlp::pack(cudaStream_t s) {
    const int n = MLP_OUT_PAD * MLP_H;
    pack_weights_kernel<<<(n + 255) / 256, 256, 0, s>>>(P, W2b, W2Tb, W3b, W3Tb);
}

// The activations of a batch of B: one allocation, which takes the place of the previous, smaller
// one only when it is there, so that after a failure the buffers and cap still match.
void Mlp::reserve(int B, cudaStream_t s) {
    if (B <= cap) return;
    size_t total = 0;
    auto place = [&](size_t bytes) {  // 256-byte aligned parts
        const size_t at = total;
        total += (bytes + 255) & ~(size_t)255;
        return at;
    };
    const size_t f = (size_t)B * MLP_H * sizeof(float), h = (size_t)B * MLP_H * sizeof(bf16);
    const size_t y = (size_t)B * MLP_OUT_PAD * sizeof(float), d = (size_t)B * MLP_K3 * sizeof(bf16);
    const size_t z1 = place(f), z2 = place(f), oy = place(y), dh = place(f), h1 = place(h), h1t = place(h), h2 = place(h),
                 h2t = place(h), ody = place(d), dyt = place(d), dz = place(h), dzt = place(h);
    char* q = nullptr;
    if (device_malloc(&q, total) != cudaSuccess) {
        cudaGetLastError();
        fail(RIMO_ERR_OOM, "activations of " + std::to_string(B) + " samples: " + std::to_string(total) + " bytes");
    }
    // rows past the padded outputs only fill the last 128-row tile of dW3
    const cudaError_t e = cudaMemsetAsync(q + dyt, 0, d, s);
    if (e != cudaSuccess) cudaFree(q);
    RIMO_CUDA(e);
    cudaFree(acts);  // (waits for the kernels that use it)
    acts = q;
    Z1 = (float*)(q + z1);
    Z2 = (float*)(q + z2);
    Y = (float*)(q + oy);
    dH = (float*)(q + dh);
    H1 = (bf16*)(q + h1);
    H1T = (bf16*)(q + h1t);
    H2 = (bf16*)(q + h2);
    H2T = (bf16*)(q + h2t);
    dY = (bf16*)(q + ody);
    dYT = (bf16*)(q + dyt);
    dZ = (bf16*)(q + dz);
    dZT = (bf16*)(q + dzt);
    cap = B;
}

void Mlp::forward(const float* X, int B, cudaStream_t s, bool train) {
    reserve(B, s);
    const int blocks = B / EL_ROWS;
    l1_fwd_kernel<<<blocks, 256, 0, s>>>(X, P + MLP_OFF_W1, P + MLP_OFF_B1, Z1, H1, train ? H1T : nullptr, B);
    gemm(H1, MLP_H, W2b, MLP_H, Z2, MLP_H, B, MLP_H, MLP_H, 64, 1, false, status, s);
    act_fwd_kernel<<<blocks, 256, 0, s>>>(Z2, P + MLP_OFF_B2, H2, train ? H2T : nullptr, B);
    gemm(H2, MLP_H, W3b, MLP_H, Y, MLP_OUT_PAD, B, MLP_OUT_PAD, MLP_H, 128, 1, false, status, s);
}

void Mlp::grads(const float* X, const float* T, int B, cudaStream_t s) {
    forward(X, B, s, true);
    RIMO_CUDA(cudaMemsetAsync(G, 0, (MLP_NPARAM + 1) * sizeof(float), s));  // and the loss
    const int blocks = B / EL_ROWS;
    loss_bwd_kernel<<<dim3(blocks, (MLP_OUT_PAD + MLP_H - 1) / MLP_H), 256, 0, s>>>(
        Y, MLP_OUT_PAD, P + MLP_OFF_B3, T, dY, MLP_K3, dYT, G + MLP_OFF_B3, loss, B);
    const int splits = std::max(1, B / 128);
    // dH2 = dY W3 (K = 464 padded output dimension)
    gemm(dY, MLP_K3, W3Tb, MLP_K3, dH, MLP_H, B, MLP_H, MLP_OUT_PAD, 64, 1, false, status, s);
    // dW3 = dY^T H2 (M = 512: the rows past the outputs are not stored)
    gemm(dYT, B, H2T, B, G + MLP_OFF_W3, MLP_H, 512, MLP_H, B, 128, splits, true, status, s, MLP_OUT);
    act_bwd_kernel<<<blocks, 256, 0, s>>>(dH, Z2, dZ, dZT, G + MLP_OFF_B2, B);
    gemm(dZT, B, H1T, B, G + MLP_OFF_W2, MLP_H, MLP_H, MLP_H, B, 64, splits, true, status, s);
    gemm(dZ, MLP_H, W2Tb, MLP_H, dH, MLP_H, B, MLP_H, MLP_H, 64, 1, false, status, s);
    l1_bwd_kernel<<<blocks, 256, 0, s>>>(dH, Z1, X, G + MLP_OFF_W1, G + MLP_OFF_B1);
}

void Mlp::step(const float* X, const float* T, int B, float lr, cudaStream_t s) {
    grads(X, T, B, s);
    ++t;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - std::pow(b1, (float)t), c2 = 1.f - std::pow(b2, (float)t);
    adam_kernel<<<(MLP_NPARAM + 255) / 256, 256, 0, s>>>(P, G, Mom, Vel, MLP_NPARAM, lr, b1, b2, 1e-8f, c1, c2);
    pack(s);
}

}  // namespace rimo

// --------------------------------------------------------------------------------------
// C ABI
struct rimo_surrogate {
    rimo::Mlp mlp;
    float w_scale = 0.f;          // input normalisation of w_r (set by rimo_surrogate_fit)
    __nv_bfloat16* W3g = nullptr;  // layer 3 for the tile generator: [480][128], see sur_gen_kernel
};

namespace rimo {

__global__ void add_bias_out_kernel(const float* __restrict__ Y, const float* __restrict__ b3, float* __restrict__ out,
                                    int B) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)B * MLP_OUT) return;
    const int b = (int)(e / MLP_OUT), j = (int)(e % MLP_OUT);
    out[e] = Y[(size_t)b * MLP_OUT_PAD + j] + b3[j];
}

static void check_batch(int64_t B) {
    if (B <= 0 || B % 128 != 0 || B > (1 << 24)) fail(RIMO_ERR_INVALID_ARG, "batch must be a positive multiple of 128");
}

static void check_status(Mlp& m, cudaStream_t s) {
    int st = 0;
    RIMO_CUDA(cudaMemcpyAsync(&st, m.status, sizeof(int), cudaMemcpyDeviceToHost, s));
    RIMO_CUDA(cudaStreamSynchronize(s));
    if (st) {
        RIMO_CUDA(cudaMemsetAsync(m.status, 0, sizeof(int), s));
        fail(RIMO_ERR_TIMEOUT, "a bounded tensor-core wait ran out");
    }
}

}  // namespace rimo

using namespace rimo;

#define SUR_BEGIN try {
#define SUR_END                       \
    return RIMO_OK;                   \
    }                                 \
    catch (const Error& e) {          \
        set_last_error(e.msg);        \
        return e.status;              \
    }                                 \
    catch (const std::exception& e) { \
        set_last_error(e.what());     \
        return RIMO_ERR_OOM;          \
    }

namespace rimo {

constexpr int SUR_S = 15;         // tile side the network outputs
constexpr int SUR_TAPS = SUR_S * SUR_S;

// SplitMix64 (Steele, Lea, Flood 2014): counter-based draws for the training samples.
__host__ __device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
    uint64_t z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// ---- tile generator: the whole network per 128 visibilities in one persistent CTA per SM
// Layer 1 (3 -> 128) on CUDA cores into shared memory (bf16, canonical K-major); layer 2 as
// 8 MMAs (M 128, N 128, K 16) into TMEM columns [0, 128); GELU read-out back into the same
// shared buffer; layer 3 as 2 x 8 MMAs (N 256 + 224) into TMEM columns [0, 480); the read-out
// adds b3 and writes each visibility's 15 x 15 complex tile (plus its even-count pad) to
// the tap scratch at the visibility's offset.  W2 and W3 stay in shared memory (bf16).
// Layer 3's rows are packed so that real and imaginary outputs start at 16-aligned TMEM
// columns: rows [0, 225) the real parts, [240, 465) the imaginary parts, the rest zero.
// One CTA per SM holds 222 KB; the GELU read-outs, the tile stores and the next rows' features
// overlap only across its own warps: 8 warps 0.806 ms, 16 warps 0.787 ms per 10^6 tiles
// (4.6 TB/s of tiles written).
constexpr int GEN_THREADS = 512;
constexpr int GEN_WG = GEN_THREADS / 128;  // warp groups: each covers the 128 TMEM lanes once
constexpr int GEN_HW = MLP_H / GEN_WG;      // hidden units (columns) per warp group
constexpr int GEN_N3 = 480, GEN_IM = 240;
constexpr size_t GEN_SW2 = (size_t)MLP_H * MLP_H * 2, GEN_SW3 = (size_t)GEN_N3 * MLP_H * 2, GEN_SA = 128 * MLP_H * 2;
constexpr size_t GEN_STAGE = (size_t)(GEN_THREADS / 32) * 4096;  // read-out staging, over the A operand
constexpr size_t GEN_SMEM = GEN_SW2 + GEN_SW3 + (GEN_SA > GEN_STAGE ? GEN_SA : GEN_STAGE) + (384 + 128 + 128 + GEN_N3 + 384) * 4 + 128 * 8;

__global__ void pack_w3g_kernel(const float* __restrict__ P, bf16* __restrict__ W3g) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= GEN_N3 * MLP_H) return;
    const int r = i / MLP_H, c = i % MLP_H;
    int src = -1;
    if (r < SUR_TAPS) src = r;
    else if (r >= GEN_IM && r < GEN_IM + SUR_TAPS) src = SUR_TAPS + (r - GEN_IM);
    W3g[i] = __float2bfloat16(src >= 0 ? P[MLP_OFF_W3 + src * MLP_H + c] : 0.f);
}

struct GenArgs {
    const VisMeta* meta;
    float2* const* gblk;
    const float* phiu;
    const float* phiv;
    const float* wr;
    int64_t v0;
    int n;
    float inv_w;
    const float* P;    // FP32 parameters (W1, b1, b2, b3)
    const bf16* W2b;   // [128][128]
    const bf16* W3g;   // [480][128]
    uint32_t* fx;
    int* status;
    const float* wt;   // data weights (sorted order) multiplying the tiles, or null
};

__device__ __forceinline__ uint32_t pack_bf2(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}

__global__ void __launch_bounds__(GEN_THREADS, 1) sur_gen_kernel(GenArgs A) {
    extern __shared__ __align__(1024) unsigned char sm[];
    unsigned char* sW2 = sm;
    unsigned char* sW3 = sm + GEN_SW2;
    unsigned char* sA = sW3 + GEN_SW3;
    float* sW1 = reinterpret_cast<float*>(sA + (GEN_SA > GEN_STAGE ? GEN_SA : GEN_STAGE));
    float* sb1 = sW1 + 384;
    float* sb2 = sb1 + 128;
    float* sb3 = sb2 + 128;
    float* sx = sb3 + GEN_N3;
    float2** sdst = reinterpret_cast<float2**>(sx + 384);  // each row's tile
    __shared__ float swt[128];  // data weight of each row
    __shared__ float s_tsum[GEN_WG][128];  // per warp group: partial tap sums of each row
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tslot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int e = tid; e < MLP_H * 16; e += GEN_THREADS) {
        const int r = e >> 4, v = e & 15;
        *reinterpret_cast<uint4*>(sW2 + tc::kmajor_offset(r, v * 8, MLP_H)) =
            *reinterpret_cast<const uint4*>(A.W2b + (size_t)r * MLP_H + v * 8);
    }
    for (int e = tid; e < GEN_N3 * 16; e += GEN_THREADS) {
        const int r = e >> 4, v = e & 15;
        *reinterpret_cast<uint4*>(sW3 + tc::kmajor_offset(r, v * 8, GEN_N3)) =
            *reinterpret_cast<const uint4*>(A.W3g + (size_t)r * MLP_H + v * 8);
    }
    for (int e = tid; e < 384; e += GEN_THREADS) sW1[e] = __bfloat162float(__float2bfloat16(A.P[MLP_OFF_W1 + e]));
    for (int e = tid; e < 128; e += GEN_THREADS) {
        sb1[e] = A.P[MLP_OFF_B1 + e];
        sb2[e] = A.P[MLP_OFF_B2 + e];
    }
    for (int e = tid; e < GEN_N3; e += GEN_THREADS) {
        int src = -1;
        if (e < SUR_TAPS) src = e;
        else if (e >= GEN_IM && e < GEN_IM + SUR_TAPS) src = SUR_TAPS + (e - GEN_IM);
        sb3[e] = src >= 0 ? A.P[MLP_OFF_B3 + src] : 0.f;
    }
    if (warp == 0) tc::tmem_alloc(&tslot, 512);
    if (tid == 0) {
        mbar_init_(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tslot;
    const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;  // this warp's TMEM lanes
    uint32_t phase = 0;
    bool ok = true;
    float run_tmax = 0.f, run_t1 = 0.f;  // running bounds over this thread's tiles
    const int ntile = (A.n + 127) / 128;
    // the next tile's inputs are loaded (raw) while this tile computes
    float in_u = 0.f, in_v = 0.f, in_w = 0.f, in_wt = 1.f;
    float2* in_dst = nullptr;
    auto load_inputs = [&](int t) {
        if (tid < 128 && t < ntile) {
            const int j = t * 128 + tid < A.n ? t * 128 + tid : A.n - 1;
            const int64_t k = A.v0 + j;
            in_u = __ldg(A.phiu + k);
            in_v = __ldg(A.phiv + k);
            in_w = __ldg(A.wr + k);
            const VisMeta mt = A.meta[k];
            in_dst = A.gblk[mt.pos >> 24] + mt.off;
            in_wt = A.wt ? __ldg(A.wt + k) : 1.f;
        }
    };
    load_inputs(blockIdx.x);
    for (int tile = blockIdx.x; tile < ntile && ok; tile += gridDim.x) {
        const int base = tile * 128;
        if (tid < 128) {
            sx[3 * tid + 0] = 2.f * in_u - 1.f;
            sx[3 * tid + 1] = 2.f * in_v - 1.f;
            sx[3 * tid + 2] = in_w * A.inv_w;
            sdst[tid] = in_dst;
            swt[tid] = in_wt;
        }
        load_inputs(tile + gridDim.x);
        __syncthreads();
        {   // layer 1: row r, hidden units [GEN_HW h, GEN_HW (h + 1))
            const int r = tid & 127, h = tid >> 7;
            const float x0 = sx[3 * r], x1 = sx[3 * r + 1], x2 = sx[3 * r + 2];
#pragma unroll 1
            for (int g = 0; g < GEN_HW / 8; ++g) {
                uint32_t w[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float z[2];
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const int j = GEN_HW * h + 8 * g + 2 * q + u;
                        z[u] = gelu_f(fmaf(x0, sW1[3 * j], fmaf(x1, sW1[3 * j + 1], fmaf(x2, sW1[3 * j + 2], sb1[j]))));
                    }
                    w[q] = pack_bf2(z[0], z[1]);
                }
                *reinterpret_cast<uint4*>(sA + tc::kmajor_offset(r, GEN_HW * h + 8 * g, 128)) =
                    make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
        tc::fence_proxy_async();
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
        if (tid == 0) {  // layer 2
            for (int s = 0; s < MLP_H / 16; ++s)
                tc::mma_bf16(tmem, tc::smem_desc(tc::smem_addr(sA) + s * 128 * 32, 128, 256),
                             tc::smem_desc(tc::smem_addr(sW2) + s * MLP_H * 32, 128, 256), tc::idesc_bf16_f32(128, 128),
                             s > 0 ? 1u : 0u);
            tc::mma_commit(&bar);
        }
        ok = mbar_wait_(&bar, phase);
        phase ^= 1;
        if (__syncthreads_or(!ok)) break;
        tc::fence_after_sync();
        {   // layer-2 read-out: row 32 (warp % 4) + lane, columns [GEN_HW (warp / 4), + GEN_HW)
            const int r = 32 * (warp & 3) + lane;
#pragma unroll 1
            for (int c0 = 0; c0 < GEN_HW; c0 += 32) {  // two 16-column loads in flight per wait
                const int col = GEN_HW * (warp >> 2) + c0;
                uint32_t va[16], vb[16];
                tc::tmem_ld16_async(tmem + lane_base + (uint32_t)col, va);
                tc::tmem_ld16_async(tmem + lane_base + (uint32_t)(col + 16), vb);
                tc::tmem_wait_ld_tied(va);
                tc::reg_tie(vb);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t* v = h ? vb : va;
                    const int cc = col + 16 * h;
                    uint32_t w[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        w[i] = pack_bf2(gelu_f(__uint_as_float(v[2 * i]) + sb2[cc + 2 * i]),
                                        gelu_f(__uint_as_float(v[2 * i + 1]) + sb2[cc + 2 * i + 1]));
                    *reinterpret_cast<uint4*>(sA + tc::kmajor_offset(r, cc, 128)) = make_uint4(w[0], w[1], w[2], w[3]);
                    *reinterpret_cast<uint4*>(sA + tc::kmajor_offset(r, cc + 8, 128)) = make_uint4(w[4], w[5], w[6], w[7]);
                }
            }
        }
        tc::fence_proxy_async();
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
        if (tid == 0) {  // layer 3: rows [0, 256) and [256, 480) of W3g
            for (int s = 0; s < MLP_H / 16; ++s) {
                const uint64_t ad = tc::smem_desc(tc::smem_addr(sA) + s * 128 * 32, 128, 256);
                const uint32_t b0 = tc::smem_addr(sW3) + s * GEN_N3 * 32;
                tc::mma_bf16(tmem, ad, tc::smem_desc(b0, 128, 256), tc::idesc_bf16_f32(128, 256), s > 0 ? 1u : 0u);
                tc::mma_bf16(tmem + 256, ad, tc::smem_desc(b0 + (256 / 8) * 256, 128, 256),
                             tc::idesc_bf16_f32(128, GEN_N3 - 256), s > 0 ? 1u : 0u);
            }
            tc::mma_commit(&bar);
        }
        ok = mbar_wait_(&bar, phase);
        phase ^= 1;
        if (__syncthreads_or(!ok)) break;
        tc::fence_after_sync();
        {   // layer-3 read-out: chunks of 16 taps (warp groups take every GEN_WG-th chunk).  The
            // chunk's 32 rows pass through a warp-private 4 KB laid over the A buffer (free once the
            // layer-3 MMAs completed) so that the warp writes 128-byte row segments, not
            // scattered 16-byte pieces; pieces are XOR-swizzled by row against bank conflicts.
            const int r = 32 * (warp & 3) + lane;
            const bool valid = base + r < A.n;
            const float wk = swt[r];
            float4* stage = reinterpret_cast<float4*>(sA) + warp * 256;  // [32 rows][8 pieces]
            float tmax = 0.f, tsum = 0.f;
#pragma unroll 1
            for (int c = warp >> 2; c < (SUR_TAPS + 15) / 16; c += GEN_WG) {
                const int q0 = 16 * c;
                uint32_t rr[16], ri[16];
                tc::tmem_ld16_async(tmem + lane_base + (uint32_t)q0, rr);
                tc::tmem_ld16_async(tmem + lane_base + (uint32_t)(GEN_IM + q0), ri);
                tc::tmem_wait_ld_tied(rr);
                tc::reg_tie(ri);
#pragma unroll
                for (int j = 0; j < 8; ++j) {  // piece j: taps q0 + 2j, q0 + 2j + 1 (zero past the tile)
                    const int q = q0 + 2 * j;
                    const float2 t0 = q < SUR_TAPS ? make_float2(wk * (__uint_as_float(rr[2 * j]) + sb3[q]),
                                                                 wk * (__uint_as_float(ri[2 * j]) + sb3[GEN_IM + q]))
                                                   : make_float2(0.f, 0.f);
                    const float2 t1 = q + 1 < SUR_TAPS
                                          ? make_float2(wk * (__uint_as_float(rr[2 * j + 1]) + sb3[q + 1]),
                                                        wk * (__uint_as_float(ri[2 * j + 1]) + sb3[GEN_IM + q + 1]))
                                          : make_float2(0.f, 0.f);
                    const float m0 = fabsf(t0.x) + fabsf(t0.y), m1 = fabsf(t1.x) + fabsf(t1.y);
                    tmax = fmaxf(tmax, fmaxf(m0, m1));
                    tsum += m0 + m1;
                    stage[lane * 8 + (j ^ (lane & 7))] = make_float4(t0.x, t0.y, t1.x, t1.y);
                }
                __syncwarp();
                // a tile holds 226 taps (225 and the pad): the last chunk has one piece
                const int npc = q0 + 16 <= SUR_TAPS + 1 ? 8 : (SUR_TAPS + 1 - q0) / 2;
#pragma unroll
                for (int it = 0; it < 8; ++it) {
                    const int row = 4 * it + (lane >> 3), pc = lane & 7;
                    const int rg = 32 * (warp & 3) + row;
                    if (pc < npc && base + rg < A.n)
                        *reinterpret_cast<float4*>(sdst[rg] + q0 + 2 * pc) = stage[row * 8 + (pc ^ (row & 7))];
                }
                __syncwarp();
            }
            if (valid) run_tmax = fmaxf(run_tmax, tmax);
            s_tsum[warp >> 2][r] = valid ? tsum : 0.f;  // each warp group holds a share of the row
        }
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
        if (tid < 128 && base + tid < A.n) {
            float t = 0.f;
#pragma unroll
            for (int q = 0; q < GEN_WG; ++q) t += s_tsum[q][tid];
            run_t1 = fmaxf(run_t1, t);
        }
    }
    // the bounds: one atomic per warp for the whole launch (not one per visibility)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        run_tmax = fmaxf(run_tmax, __shfl_xor_sync(0xffffffffu, run_tmax, o));
        run_t1 = fmaxf(run_t1, __shfl_xor_sync(0xffffffffu, run_t1, o));
    }
    if (lane == 0) {
        atomicMax(A.fx + FX_TMAX, __float_as_uint(run_tmax));
        atomicMax(A.fx + FX_T1, __float_as_uint(run_t1));
    }
    if (!ok && tid == 0) atomicExch(A.status, 2);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) {
        tc::tmem_dealloc(tmem, 512);
        tc::tmem_relinquish();
    }
}

void reset_surrogate_bounds(rimo_plan* p, cudaStream_t s) {
    RIMO_CUDA(cudaMemsetAsync(p->d_fx + FX_TMAX, 0, 2 * sizeof(uint32_t), s));  // FX_TMAX, FX_T1
    if (p->mode == RIMO_MODE_SURROGATE)  // this apply's network (it may have trained since)
        pack_w3g_kernel<<<(GEN_N3 * MLP_H + 255) / 256, 256, 0, s>>>(p->sur->mlp.P, p->sur->W3g);
}

int surrogate_generate(rimo_plan* p, int64_t v0, int64_t n, cudaStream_t s) {
    rimo_surrogate* sur = p->sur;
    const float ws = sur->w_scale > 0.f ? sur->w_scale : (p->info.wr_max > 0 ? (float)p->info.wr_max : 1.f);
    if (n <= 0) return 0;
    GenArgs A;
    A.meta = p->d_meta;
    A.gblk = p->d_gblock_ptrs;
    A.phiu = p->d_phiu;
    A.phiv = p->d_phiv;
    A.wr = p->d_wr;
    A.v0 = v0;
    A.n = (int)n;
    A.inv_w = 1.f / ws;
    A.P = sur->mlp.P;
    A.W2b = sur->mlp.W2b;
    A.W3g = sur->W3g;
    A.fx = p->d_fx;
    A.status = p->d_status;
    A.wt = p->d_wt;
    set_smem(sur_gen_kernel, GEN_SMEM);
    const int64_t ntile = (n + 127) / 128;
    const int grid = (int)std::min<int64_t>(ntile, (int64_t)p->n_sm);
    sur_gen_kernel<<<grid, GEN_THREADS, GEN_SMEM, s>>>(A);
    return 1;
}

// training sample i: a visibility k drawn uniformly, its inputs, and its exact tile embedded
// at the centre of 15 x 15 (a smaller support S sits at offset (15 - S) / 2)
__global__ void sur_dataset_kernel(const VisMeta* __restrict__ meta, float2* const* __restrict__ gblk,
                                   const float* __restrict__ phiu, const float* __restrict__ phiv,
                                   const float* __restrict__ wr, int64_t M, uint64_t seed, int64_t n, float inv_w,
                                   float* X, float* T) {
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (i >= n) return;
    const int64_t k = (int64_t)(splitmix64(seed + (uint64_t)i) % (uint64_t)M);
    const VisMeta mt = meta[k];
    const int S = (mt.pos >> 16) & 255, off = (SUR_S - S) / 2;
    const float2* G = gblk[mt.pos >> 24] + mt.off;
    if (lane == 0) {
        X[3 * i + 0] = 2.f * phiu[k] - 1.f;
        X[3 * i + 1] = 2.f * phiv[k] - 1.f;
        X[3 * i + 2] = wr[k] * inv_w;
    }
    float* t = T + (size_t)i * MLP_OUT;
    for (int q = lane; q < SUR_TAPS; q += 32) {
        const int a = q / SUR_S - off, b = q % SUR_S - off;
        const float2 v = (a >= 0 && a < S && b >= 0 && b < S) ? G[a * S + b] : make_float2(0.f, 0.f);
        t[q] = v.x;
        t[SUR_TAPS + q] = v.y;
    }
}

__global__ void sur_batch_kernel(const float* __restrict__ X, const float* __restrict__ T, int64_t n, uint64_t seed,
                                 int B, float* Xb, float* Tb) {
    const int j = blockIdx.x;
    const int64_t i = (int64_t)(splitmix64(seed + (uint64_t)j) % (uint64_t)n);
    for (int e = threadIdx.x; e < MLP_OUT; e += blockDim.x) Tb[(size_t)j * MLP_OUT + e] = T[(size_t)i * MLP_OUT + e];
    if (threadIdx.x < 3) Xb[3 * j + threadIdx.x] = X[3 * i + threadIdx.x];
}

struct DevScratch {
    std::vector<void*> v;
    void* get(size_t bytes) {
        void* ptr = nullptr;
        if (device_malloc(&ptr, bytes) != cudaSuccess) {
            cudaGetLastError();
            fail(RIMO_ERR_OOM, "cudaMalloc of " + std::to_string(bytes) + " bytes for the training set failed");
        }
        v.push_back(ptr);
        return ptr;
    }
    ~DevScratch() {
        for (void* ptr : v) cudaFree(ptr);
    }
};

}  // namespace rimo

extern "C" {

rimo_status rimo_surrogate_create(uint64_t seed, rimo_surrogate_t* out) {
    if (out) *out = nullptr;
    rimo_surrogate* s = nullptr;
    try {
        if (!out) fail(RIMO_ERR_INVALID_ARG, "null output");
        s = new rimo_surrogate();
        s->mlp.init(seed);
        RIMO_CUDA(cudaDeviceSynchronize());
        *out = s;
        return RIMO_OK;
    } catch (const Error& e) {
        set_last_error(e.msg);
        delete s;
        return e.status;
    }
}

rimo_status rimo_surrogate_destroy(rimo_surrogate_t s) {
    delete s;
    return RIMO_OK;
}

rimo_status rimo_surrogate_get_params(rimo_surrogate_t s, float* params) {
    SUR_BEGIN
    if (!s || !params) fail(RIMO_ERR_INVALID_ARG, "null argument");
    RIMO_CUDA(cudaMemcpy(params, s->mlp.P, MLP_NPARAM * sizeof(float), cudaMemcpyDeviceToHost));
    SUR_END
}

rimo_status rimo_surrogate_set_params(rimo_surrogate_t s, const float* params) {
    SUR_BEGIN
    if (!s || !params) fail(RIMO_ERR_INVALID_ARG, "null argument");
    s->mlp.set_params(params, 0);
    RIMO_CUDA(cudaDeviceSynchronize());
    SUR_END
}

rimo_status rimo_surrogate_forward(rimo_surrogate_t s, const float* x, int64_t B, float* y, void* stream) {
    SUR_BEGIN
    if (!s || !x || !y) fail(RIMO_ERR_INVALID_ARG, "null argument");
    check_batch(B);
    cudaStream_t st = (cudaStream_t)stream;
    s->mlp.forward(x, (int)B, st);
    const int64_t n = B * MLP_OUT;
    add_bias_out_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(s->mlp.Y, s->mlp.P + MLP_OFF_B3, y, (int)B);
    RIMO_CUDA(cudaGetLastError());
    SUR_END
}

rimo_status rimo_surrogate_gradients(rimo_surrogate_t s, const float* x, const float* t, int64_t B, float* grads,
                                     float* loss, void* stream) {
    SUR_BEGIN
    if (!s || !x || !t) fail(RIMO_ERR_INVALID_ARG, "null argument");
    check_batch(B);
    cudaStream_t st = (cudaStream_t)stream;
    Mlp& m = s->mlp;
    m.grads(x, t, (int)B, st);
    RIMO_CUDA(cudaGetLastError());
    RIMO_CUDA(cudaMemcpyAsync(m.host, m.G, (MLP_NPARAM + 2) * sizeof(float), cudaMemcpyDeviceToHost, st));
    RIMO_CUDA(cudaStreamSynchronize(st));
    int failed = 0;
    std::memcpy(&failed, m.host + MLP_NPARAM + 1, sizeof(int));
    if (failed) check_status(m, st);  // clears it and reports
    if (grads) std::memcpy(grads, m.host, MLP_NPARAM * sizeof(float));
    if (loss) *loss = m.host[MLP_NPARAM] / ((float)B * MLP_OUT);
    SUR_END
}

rimo_status rimo_surrogate_train_step(rimo_surrogate_t s, const float* x, const float* t, int64_t B, float lr,
                                      float* loss, void* stream) {
    SUR_BEGIN
    if (!s || !x || !t) fail(RIMO_ERR_INVALID_ARG, "null argument");
    check_batch(B);
    cudaStream_t st = (cudaStream_t)stream;
    s->mlp.step(x, t, (int)B, lr, st);
    RIMO_CUDA(cudaGetLastError());
    if (loss) {
        float l = 0.f;
        RIMO_CUDA(cudaMemcpyAsync(&l, s->mlp.loss, sizeof(float), cudaMemcpyDeviceToHost, st));
        RIMO_CUDA(cudaStreamSynchronize(st));
        *loss = l / ((float)B * MLP_OUT);
    }
    SUR_END
}


rimo_status rimo_plan_set_surrogate(rimo_plan_t p, rimo_surrogate_t s) {
    SUR_BEGIN
    if (!p || !s) fail(RIMO_ERR_INVALID_ARG, "null argument");
    if (p->mode != RIMO_MODE_SURROGATE) fail(RIMO_ERR_INVALID_ARG, "the plan was not created in surrogate mode");
    int dev = 0;
    RIMO_CUDA(cudaGetDevice(&dev));
    if (dev != p->device) fail(RIMO_ERR_INVALID_ARG, "plan and surrogate on different devices");
    // everything the generation needs is allocated here, not during an apply
    if (!s->W3g) s->W3g = (bf16*)s->mlp.alloc((size_t)GEN_N3 * MLP_H * sizeof(bf16));
    p->sur = s;
    SUR_END
}

rimo_status rimo_surrogate_fit(rimo_surrogate_t s, rimo_plan_t exact, int64_t n_samples, int32_t steps,
                               int32_t batch, float lr, uint64_t seed, float* losses, void* stream) {
    SUR_BEGIN
    if (!s || !exact) fail(RIMO_ERR_INVALID_ARG, "null argument");
    if (exact->mode == RIMO_MODE_SURROGATE || exact->d_gblocks.empty())
        fail(RIMO_ERR_INVALID_ARG, "training needs a plan with stored exact tiles");
    if (exact->d_wt) fail(RIMO_ERR_STATE, "training needs unweighted tiles (remove the plan's weighting first)");
    if (exact->J + exact->prm.max_wsupport - 1 != SUR_S)
        fail(RIMO_ERR_INVALID_ARG, "training tiles must be 15 x 15 (kb_support + max_wsupport - 1 = 15)");
    if (n_samples <= 0 || steps <= 0 || !(lr > 0.f)) fail(RIMO_ERR_INVALID_ARG, "n_samples, steps, lr must be > 0");
    check_batch(batch);
    cudaStream_t st = (cudaStream_t)stream;
    const float ws = exact->info.wr_max > 0 ? (float)exact->info.wr_max : 1.f;
    DevScratch tmp;
    float* X = (float*)tmp.get((size_t)n_samples * 3 * sizeof(float));
    float* T = (float*)tmp.get((size_t)n_samples * MLP_OUT * sizeof(float));
    float* Xb = (float*)tmp.get((size_t)batch * 3 * sizeof(float));
    float* Tb = (float*)tmp.get((size_t)batch * MLP_OUT * sizeof(float));
    float* L = (float*)tmp.get((size_t)steps * sizeof(float));
    const uint64_t sample_seed = splitmix64(seed ^ 0x5EEDull);
    sur_dataset_kernel<<<(unsigned)((n_samples * 32 + 255) / 256), 256, 0, st>>>(
        exact->d_meta, exact->d_gblock_ptrs, exact->d_phiu, exact->d_phiv, exact->d_wr, exact->M, sample_seed,
        n_samples, 1.f / ws, X, T);
    RIMO_CUDA(cudaGetLastError());
    s->mlp.reserve(batch, st);
    for (int k = 0; k < steps; ++k) {
        // cosine decay from lr to lr / 100
        const float lr_k = lr * (0.01f + 0.99f * 0.5f * (1.f + std::cos(3.14159265358979f * (float)k / (float)steps)));
        sur_batch_kernel<<<batch, 128, 0, st>>>(X, T, n_samples, splitmix64(seed + 0x9E37ull * (uint64_t)(k + 1)),
                                                 batch, Xb, Tb);
        s->mlp.step(Xb, Tb, batch, lr_k, st);
        RIMO_CUDA(cudaMemcpyAsync(L + k, s->mlp.loss, sizeof(float), cudaMemcpyDeviceToDevice, st));
    }
    RIMO_CUDA(cudaGetLastError());
    check_status(s->mlp, st);
    if (losses) {
        RIMO_CUDA(cudaMemcpyAsync(losses, L, (size_t)steps * sizeof(float), cudaMemcpyDeviceToHost, st));
        RIMO_CUDA(cudaStreamSynchronize(st));
        for (int k = 0; k < steps; ++k) losses[k] /= (float)batch * MLP_OUT;
    }
    RIMO_CUDA(cudaStreamSynchronize(st));
    s->w_scale = ws;
    SUR_END
}

rimo_status rimo_surrogate_get_w_scale(rimo_surrogate_t s, float* w_scale) {
    SUR_BEGIN
    if (!s || !w_scale) fail(RIMO_ERR_INVALID_ARG, "null argument");
    *w_scale = s->w_scale;
    SUR_END
}

rimo_status rimo_surrogate_set_w_scale(rimo_surrogate_t s, float w_scale) {
    SUR_BEGIN
    if (!s || !(w_scale > 0.f)) fail(RIMO_ERR_INVALID_ARG, "null surrogate or w_scale <= 0");
    s->w_scale = w_scale;
    SUR_END
}

}  // extern "C"
