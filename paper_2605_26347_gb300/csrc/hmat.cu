// Holographic matrices H_p = G_p^dagger G_p (Section 3.3): device build and apply.
//
// H_p[c1][c2] = sum_k conj(G_p[k][c1]) G_p[k][c2] couples two grid cells when some
// visibility's S x S footprint covers both, so |c2 - c1| <= D = S_max - 1 per axis.  H_p is
// Hermitian; each unordered pair is stored once, at its owner: the top-left corner of the
// pair's bounding box.  Owner o stores
//   type A: (a, b) in [0, D]^2                 H[o][o + (a, b)]
//   type B: a in [1, D], b in [1, D]           H[o + (0, b)][o + (a, 0)]
// ((D+1)^2 + D^2 entries; pairs with du = 0 > dv are type A of the swapped pair).  Every
// cell an owner's entries touch lies in o + [0, D]^2, so the apply writes the same patch
// geometry as the gridding step ([tile origin, + TS + D) per axis), and the same fold
// sums the patches into the grid.
//
// Only owners that some footprint covers get a row: a coverage pass marks the covered
// cells of each needed tile (bitmap), the host turns the counts into row offsets, and the
// build pass writes the rows.  Where cells see one or a few visibilities most pairs are
// never covered together, so a bin's rows keep only their non-zero entries (value and entry
// number, rows found by offsets) when that is smaller than the dense rows: the build writes
// the bin's rows densely to a temporary, a count pass decides, and a compaction pass keeps
// each row's non-zero values; a bin of dense coverage keeps the dense rows as they are.  Build: one CTA per 4 x 4 block of owners, one warp per
// owner keeping its entries in shared memory (no atomics); the candidate visibilities
// (anchor within D before the block) come from an anchor index sorted by (g0, h0) that the
// host prepares.  Apply: one CTA per needed tile, one warp per owner; the gathered sum
// of the type-A row, its scattered conjugate terms and the type-B block's row and column sums
// are accumulated in the two-word fixed-point patch of the gridding step.
#include <algorithm>
#include <cstring>
#include <numeric>
#include <vector>

#include "fixed.cuh"
#include "internal.h"
#include "planner.h"

using namespace rimo;

namespace rimo {

namespace {

constexpr int HB_OWN = 4;                 // owner block edge of the build
constexpr int HB_WARPS = HB_OWN * HB_OWN;  // one warp per owner
constexpr int HB_CHUNK = 16;              // candidate visibilities staged at a time
constexpr int HA_WARPS = 8;               // apply: warps per CTA, two CTAs per SM

// entry e of an owner row -> (type, a, b), packed type << 16 | a << 8 | b
std::vector<int32_t> entry_table(int D) {
    std::vector<int32_t> t;
    for (int a = 0; a <= D; ++a)
        for (int b = 0; b <= D; ++b) t.push_back((0 << 16) | (a << 8) | b);
    for (int a = 1; a <= D; ++a)
        for (int b = 1; b <= D; ++b) t.push_back((1 << 16) | (a << 8) | b);
    return t;
}

struct AnchorIndex {
    int32_t* pos = nullptr;      // sorted position of each visibility, ordered by (g0, h0) per bin
    uint16_t* h0 = nullptr;      // its anchor column (grid cells < 65536)
    int64_t* row = nullptr;      // [bin][g0 + 1]: first index of anchor row g0 (bin ranges [vb, ve))
    ~AnchorIndex() {
        cudaFree(pos);
        cudaFree(h0);
        cudaFree(row);
    }
};

__device__ __forceinline__ int wrap(int x, int n) { return x < 0 ? x + n : (x >= n ? x - n : x); }

// candidate ranges: anchors in rows [r0, r0 + nr) and columns [c0, c0 + nc) (mod grid); a
// column window that wraps splits in two.  Writes up to 2 nr ranges [lo, hi) into rng.
__device__ int candidate_ranges(const int64_t* __restrict__ row, const uint16_t* __restrict__ h0, int gx, int gy,
                                int r0, int nr, int c0, int nc, int64_t* rng_lo, int64_t* rng_hi, int* rng_row,
                                int tid, int nthreads) {
    // windows along v: [c0, c0 + nc) possibly wrapping
    int wlo[2], whi[2], nw = 0;
    const int cs = wrap(c0, gy);
    if (cs + nc <= gy) {
        wlo[0] = cs, whi[0] = cs + nc, nw = 1;
    } else {
        wlo[0] = cs, whi[0] = gy, wlo[1] = 0, whi[1] = cs + nc - gy, nw = 2;
    }
    for (int q = tid; q < nr * nw; q += nthreads) {
        const int r = wrap(r0 + q / nw, gx), w = q % nw;
        int64_t lo = row[r], hi = row[r + 1];
        // first index with h0 >= wlo, first with h0 >= whi (h0 ascending within a row)
        int64_t a = lo, b = hi;
        while (a < b) {
            const int64_t m = (a + b) >> 1;
            if ((int)h0[m] < wlo[w]) a = m + 1;
            else b = m;
        }
        const int64_t first = a;
        b = hi;
        while (a < b) {
            const int64_t m = (a + b) >> 1;
            if ((int)h0[m] < whi[w]) a = m + 1;
            else b = m;
        }
        rng_lo[q] = first;
        rng_hi[q] = a;
        rng_row[q] = r;
    }
    return nr * nw;
}

struct HArgs {
    const VisMeta* meta;
    float2* const* gblk;
    const int32_t* apos;     // anchor index (this bin's slice starts at 0 of row[])
    const uint16_t* ah0;
    const int64_t* arow;     // [gx + 1]
    const int32_t* need;     // needed tiles of the bin
    uint32_t* bits;          // [needed tile][TS*TS/32]
    int64_t* count;          // [needed tile] covered cells (coverage pass)
    const int64_t* hoff;     // [needed tile + 1]
    float2* rows;            // [owner][ne]
    uint32_t* tmax;          // [needed tile] max |h.x| + |h.y| over the tile's rows (float bits)
    const int32_t* ent;      // entry table
    uint32_t* fx;
    int gx, gy, ntv, TS, D, ne;
};

// Coverage pass: one CTA per needed tile marks the cells that some footprint covers.
__global__ void __launch_bounds__(256) hcover_kernel(HArgs A) {
    extern __shared__ __align__(16) unsigned char csm[];
    const int words = A.TS * A.TS / 32;
    const int nrmax = 2 * (A.TS + A.D);
    int64_t* rlo = reinterpret_cast<int64_t*>(csm);
    int64_t* rhi = rlo + nrmax;
    int* rrow = reinterpret_cast<int*>(rhi + nrmax);
    uint32_t* bm = reinterpret_cast<uint32_t*>(rrow + nrmax);
    const int tile = A.need[blockIdx.x];
    const int tu = tile / A.ntv, tv = tile - tu * A.ntv;
    const int u0 = tu * A.TS, v0 = tv * A.TS;
    for (int e = threadIdx.x; e < words; e += blockDim.x) bm[e] = 0u;
    // anchors whose footprint (at most D + 1 cells from the anchor) can reach the tile
    const int nrng = candidate_ranges(A.arow, A.ah0, A.gx, A.gy, u0 - A.D, A.TS + A.D, v0 - A.D, A.TS + A.D, rlo,
                                      rhi, rrow, threadIdx.x, blockDim.x);
    __syncthreads();
    for (int q = 0; q < nrng; ++q) {
        const int g0 = rrow[q];
        for (int64_t j = rlo[q] + threadIdx.x; j < rhi[q]; j += blockDim.x) {
            const VisMeta mt = A.meta[A.apos[j]];
            const int S = (mt.pos >> 16) & 255;
            const int h0 = A.ah0[j];
            for (int a = 0; a < S; ++a) {
                const int rr = wrap(g0 + a - u0, A.gx);  // row of the footprint relative to the tile
                if (rr >= A.TS) continue;
                for (int b = 0; b < S; ++b) {
                    const int cc = wrap(h0 + b - v0, A.gy);
                    if (cc >= A.TS) continue;
                    const int cell = rr * A.TS + cc;
                    atomicOr(&bm[cell >> 5], 1u << (cell & 31));
                }
            }
        }
    }
    __syncthreads();
    int cnt = 0;
    for (int e = threadIdx.x; e < words; e += blockDim.x) {
        A.bits[(size_t)blockIdx.x * words + e] = bm[e];
        cnt += __popc(bm[e]);
    }
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    __shared__ int wsum[8];
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += wsum[w];
        A.count[blockIdx.x] = t;
    }
}

// Rank of cell `cell` among the covered cells of a tile (row-major) from its bitmap.
__device__ __forceinline__ int64_t owner_rank(const uint32_t* bm, int cell) {
    int r = 0;
    for (int w = 0; w < (cell >> 5); ++w) r += __popc(bm[w]);
    return r + __popc(bm[cell >> 5] & ((1u << (cell & 31)) - 1u));
}

// Build pass: one CTA per HB_OWN x HB_OWN owners of a needed tile.
__global__ void __launch_bounds__(HB_WARPS * 32, 1) hbuild_kernel(HArgs A, int S_max) {
    extern __shared__ __align__(16) unsigned char hsm[];
    const int ne = A.ne;
    float2* acc = reinterpret_cast<float2*>(hsm);                       // [HB_WARPS][ne]
    float2* taps = acc + (size_t)HB_WARPS * ne;                          // [HB_CHUNK][S_max^2]
    int4* cmeta = reinterpret_cast<int4*>(taps + (size_t)HB_CHUNK * S_max * S_max);  // g0, h0, S, -
    int* sent = reinterpret_cast<int*>(cmeta + HB_CHUNK);               // [ne]
    int64_t* rlo = reinterpret_cast<int64_t*>(sent + ne + (ne & 1));
    const int nrmax = 2 * (HB_OWN + A.D);
    int64_t* rhi = rlo + nrmax;
    int* rrow = reinterpret_cast<int*>(rhi + nrmax);
    __shared__ uint32_t tbits[128];

    const int per_side = A.TS / HB_OWN;
    const int t_idx = blockIdx.x / (per_side * per_side);
    const int sub = blockIdx.x - t_idx * per_side * per_side;
    const int tile = A.need[t_idx];
    const int tu = tile / A.ntv, tv = tile - tu * A.ntv;
    const int su0 = tu * A.TS + (sub / per_side) * HB_OWN, sv0 = tv * A.TS + (sub % per_side) * HB_OWN;
    const int words = A.TS * A.TS / 32;
    for (int e = threadIdx.x; e < words; e += blockDim.x) tbits[e] = A.bits[(size_t)t_idx * words + e];
    for (int e = threadIdx.x; e < ne; e += blockDim.x) sent[e] = A.ent[e];
    for (int e = threadIdx.x; e < HB_WARPS * ne; e += blockDim.x) acc[e] = make_float2(0.f, 0.f);
    const int nrng = candidate_ranges(A.arow, A.ah0, A.gx, A.gy, su0 - A.D, HB_OWN + A.D, sv0 - A.D, HB_OWN + A.D,
                                      rlo, rhi, rrow, threadIdx.x, blockDim.x);
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ou = su0 + warp / HB_OWN, ov = sv0 + warp % HB_OWN;  // this warp's owner (grid cell)
    const int lcell = (ou - tu * A.TS) * A.TS + (ov - tv * A.TS);
    const bool covered = (tbits[lcell >> 5] >> (lcell & 31)) & 1u;
    float2* my = acc + (size_t)warp * ne;

    // walk the candidates in chunks
    int q = 0;
    int64_t j = nrng > 0 ? rlo[0] : 0;
    while (true) {
        // gather the next chunk's indices (same on every thread)
        int64_t idx[HB_CHUNK];
        int irow[HB_CHUNK];
        int nvis = 0;
        while (nvis < HB_CHUNK && q < nrng) {
            if (j >= rhi[q]) {
                ++q;
                if (q < nrng) j = rlo[q];
                continue;
            }
            irow[nvis] = rrow[q];
            idx[nvis++] = j++;
        }
        if (nvis == 0) break;
        __syncthreads();  // previous chunk consumed
        if (threadIdx.x < nvis) {
            int64_t jj = 0;
            int g0 = 0;
#pragma unroll
            for (int t = 0; t < HB_CHUNK; ++t)
                if (t == (int)threadIdx.x) jj = idx[t], g0 = irow[t];
            const VisMeta mt = A.meta[A.apos[jj]];
            cmeta[threadIdx.x] = make_int4(g0, (int)A.ah0[jj], (mt.pos >> 16) & 255, 0);
        }
        __syncthreads();
        for (int v = 0; v < nvis; ++v) {
            const int64_t jj = idx[v];
            const VisMeta mt = A.meta[A.apos[jj]];
            const int S = cmeta[v].z;
            const float2* src = A.gblk[mt.pos >> 24] + mt.off;
            for (int e = threadIdx.x; e < S * S; e += blockDim.x) taps[(size_t)v * S_max * S_max + e] = src[e];
        }
        __syncthreads();
        if (covered) {
            for (int v = 0; v < nvis; ++v) {
                const int4 cm = cmeta[v];
                const int S = cm.z;
                const int pu = wrap(ou - cm.x, A.gx), pv = wrap(ov - cm.y, A.gy);
                if (pu >= S || pv >= S) continue;  // the footprint misses this owner
                const float2* T = taps + (size_t)v * S_max * S_max;
                for (int e = lane; e < ne; e += 32) {
                    const int en = sent[e];
                    const int a = (en >> 8) & 255, b = en & 255;
                    int u1, v1, u2, v2;
                    if ((en >> 16) == 0) {
                        u1 = pu, v1 = pv, u2 = pu + a, v2 = pv + b;
                    } else {
                        u1 = pu, v1 = pv + b, u2 = pu + a, v2 = pv;
                    }
                    if (u2 >= S || v1 >= S || v2 >= S) continue;
                    const float2 t1 = T[u1 * S + v1], t2 = T[u2 * S + v2];
                    // conj(t1) t2; the diagonal (e = 0) is |t1|^2, real by construction
                    my[e].x = fmaf(t1.x, t2.x, fmaf(t1.y, t2.y, my[e].x));
                    if (e != 0) my[e].y = fmaf(t1.x, t2.y, fmaf(-t1.y, t2.x, my[e].y));
                }
            }
        }
    }
    __syncthreads();
    if (!covered) return;
    const int64_t row = A.hoff[t_idx] + owner_rank(tbits, lcell);
    float2* dst = A.rows + (size_t)row * ne;
    float m = 0.f;
    for (int e = lane; e < ne; e += 32) {
        const float2 h = my[e];
        dst[e] = h;
        m = fmaxf(m, fabsf(h.x) + fabsf(h.y));
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) {
        atomicMax(A.fx + FX_HMAX, __float_as_uint(m));
        atomicMax(A.tmax + t_idx, __float_as_uint(m));
    }
}

// ---- apply
struct HApplyArgs {
    const float2* X;          // forward grid [gx][gy] (valid on needed tiles)
    const uint8_t* need_mask; // [tile] of this bin
    const int32_t* need;      // needed tiles of the bin
    const uint32_t* bits;
    const int64_t* hoff;
    const float2* val;        // the owner rows: dense [owner][ne], or their non-zero entries
    const uint16_t* idx;      // compressed: the entry numbers
    const int64_t* roff;      // compressed: [owner + 1] first entry of each owner row (null: dense)
    const uint32_t* tmax;     // [needed tile] max |h|_1 of the tile's rows
    float2* patch;            // [needed tile][PW * PW]
    int gx, gy, ntv, TS, PW, pitch, shift;
};

// sum over the W lanes of a group (W a power of two, lanes of one group consecutive) of W values
// per lane: lane l of the group gets the sum of value l (W - 1 exchanges instead of W log W)
template <int W>
__device__ __forceinline__ float lane_sums(float (&v)[W], int lane) {
#pragma unroll
    for (int w = W / 2; w >= 1; w >>= 1) {
        const bool up = lane & w;
#pragma unroll
        for (int j = 0; j < w; ++j) {
            const float send = up ? v[j] : v[j + w];
            v[j] = (up ? v[j + w] : v[j]) + __shfl_xor_sync(0xffffffffu, send, w);
        }
    }
    return v[0];
}

// One owner's dense row in registers, spread over a warp as in the grid step's vis_tile: CW
// lanes hold the columns of a row, 32 / CW rows per step.
template <int S>
struct HRow {
    static constexpr int CW = S <= 8 ? 8 : (S <= 16 ? 16 : 32), RPI = 32 / CW, D = S - 1;
    static constexpr int NA = (S + RPI - 1) / RPI, NB = (D + RPI - 1) / RPI;
    f32x2 a[NA], b[NB];  // type A: h[a][b], a, b in [0, D]; type B: a, b in [1, D]
    template <class Ld>  // ld(e): entry e
    __device__ __forceinline__ void load(int lane, Ld ld) {
        const int c = lane % CW, ro = lane / CW;
#pragma unroll
        for (int i = 0; i < NA; ++i) a[i] = c < S && i * RPI + ro < S ? ld((i * RPI + ro) * S + c) : 0ull;
#pragma unroll
        for (int i = 0; i < NB; ++i) b[i] = c < D && i * RPI + ro < D ? ld(S * S + (i * RPI + ro) * D + c) : 0ull;
    }
};

// The products of one owner's row (cell (lu, lv) of the patch) with the input patch Z, added to
// the accumulator planes.
//   type A (the owner with the cells c2 below and right of it): the row's sum h z[c2] is the
//     owner's, conj(h) z[owner] goes to each c2;
//   type B (the cells c1 right of the owner with the cells c2 below it): with lanes along b and
//     steps along a the sums over a stay in registers (h z[c2] of c1) and those over b are one
//     exchange tree for all of them (conj(h) z[c1] of c2), so only the (2 D) sums are added to
//     the patch, not every product.
template <int S>
__device__ __forceinline__ void h_owner(const HRow<S>& h, const float2* Z, int* acc, int PW, int pitch, int plane,
                                        int lu, int lv, float s1, int lane) {
    constexpr int CW = HRow<S>::CW, RPI = HRow<S>::RPI, NA = HRow<S>::NA, NB = HRow<S>::NB, D = S - 1;
    const int c = lane % CW, ro = lane / CW;
    const float2 zo = Z[lu * PW + lv];
    {
        const bool row_ok = (NA - 1) * RPI + ro < S;
        const f32x2* Zl = reinterpret_cast<const f32x2*>(Z) + (lu + ro) * PW + lv + c;
        f32x2 p = 0ull;
        float q1 = 0.f, q2 = 0.f;
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            const f32x2 z = (i + 1) * RPI <= S || row_ok ? Zl[i * RPI * PW] : 0ull;
            p = fma2(h.a[i], z, p);
            const float2 hs = upk(h.a[i]), zs = upk(z);
            q1 = fmaf(hs.x, zs.y, q1);
            q2 = fmaf(hs.y, zs.x, q2);
        }
        const float2 ps = upk(p);
        const float re = c < S ? ps.x - ps.y : 0.f, im = c < S ? q1 + q2 : 0.f;
        const bool hi = lane & 16;
        float v = hi ? im : re;
        v += __shfl_xor_sync(0xffffffffu, hi ? re : im, 16);
        v += __shfl_xor_sync(0xffffffffu, v, 8);
        v += __shfl_xor_sync(0xffffffffu, v, 4);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        const float o = __shfl_xor_sync(0xffffffffu, v, 16);  // lane 0: the sum is (v, o)
        const float zr = zo.x * s1, zi = zo.y * s1, nzr = -zr;
        int* al = acc + (lu + ro) * pitch + lv + c;
        if (c < S) {
#pragma unroll
            for (int i = 0; i < NA; ++i) {
                if ((i + 1) * RPI <= S || row_ok) {
                    const float2 hs = upk(h.a[i]);
                    f32x2 d = pk(fmaf(hs.x, zr, hs.y * zi), fmaf(hs.x, zi, hs.y * nzr));
                    if (i == 0 && lane == 0) d = pk(v * s1, o * s1);  // the owner's own cell: the row's sum
                    fx_add2(al + i * RPI * pitch, plane, d);
                }
            }
        }
    }
    {
        const float2 zero = make_float2(0.f, 0.f);
        const float2 z1 = c < D ? Z[lu * PW + lv + c + 1] : zero;  // z[c1]
        float rx = 0.f, ry = 0.f;
        constexpr int NC = (2 * NB + CW - 1) / CW;
        float w[NC][CW];
#pragma unroll
        for (int i = 0; i < NC * CW; ++i) w[i / CW][i % CW] = 0.f;
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int a = i * RPI + ro;
            const float2 z2 = (i + 1) * RPI <= D || a < D ? Z[(lu + a + 1) * PW + lv] : zero;  // z[c2]
            const float2 hs = upk(h.b[i]);
            rx = fmaf(hs.x, z2.x, fmaf(-hs.y, z2.y, rx));
            ry = fmaf(hs.x, z2.y, fmaf(hs.y, z2.x, ry));
            w[2 * i / CW][2 * i % CW] = fmaf(hs.x, z1.x, hs.y * z1.y);
            w[(2 * i + 1) / CW][(2 * i + 1) % CW] = fmaf(hs.x, z1.y, -hs.y * z1.x);
        }
#pragma unroll
        for (int o = CW; o < 32; o <<= 1) {
            rx += __shfl_xor_sync(0xffffffffu, rx, o);
            ry += __shfl_xor_sync(0xffffffffu, ry, o);
        }
        if (ro == 0 && c < D) fx_add2(acc + lu * pitch + lv + c + 1, plane, pk(rx * s1, ry * s1));
#pragma unroll
        for (int q = 0; q < NC; ++q) {
            const float t = lane_sums<CW>(w[q], lane) * s1;
            const int e = q * CW + c, a = (e >> 1) * RPI + ro;
            if (e < 2 * NB && a < D) {
                const float tq = __fadd_rn(t, FX_MAGIC);
                const float rf = __fsub_rn(t, __fsub_rn(tq, FX_MAGIC));
                int* p = acc + (lu + a + 1) * pitch + lv + (e & 1) * plane;
                atomicAdd(p, __float_as_int(tq) - FX_MAGIC_BITS);
                atomicAdd(p + 2 * plane, __float_as_int(__fmaf_rn(rf, 65536.f, FX_MAGIC)) - FX_MAGIC_BITS);
            }
        }
    }
}

// One block per needed tile, one warp per owner (covered cells round robin).  A warp loads the
// row of its next owner (dense rows: into registers, coalesced) while it multiplies the
// current one, which keeps about 54 KB per SM in flight; a compressed row is first spread into
// a dense one in the warp's shared buffer.
// Bound by HBM at best (8 bytes per entry); before, with one entry per lane and every product
// added to the patch (8 shared reductions per type-B entry, no load ahead of the reductions),
// 256^2/1M/4 bins (1M rows, 3.4 GB) took 3.00 ms; now 0.75 ms, 4.7 TB/s, in one launch over the
// bins (the rows' 120-byte segments fetch 1.6 times their bytes from L2).
template <int S>
__global__ void __launch_bounds__(HA_WARPS * 32, 2)
    happly_kernel(const __grid_constant__ HApplyArgs one, const HApplyArgs* __restrict__ jobs,
                  const int* __restrict__ first, int njobs) {
    constexpr int D = S - 1, NE = S * S + D * D;
    extern __shared__ __align__(16) unsigned char hsm[];
    __shared__ uint32_t tbits[128];
    __shared__ int wsum[129];          // covered cells before each bitmap word
    __shared__ uint16_t cells[4096];   // the covered cells in row-major order
    __shared__ uint32_t s_zmax;
    int t_idx = (int)blockIdx.x;
    const HApplyArgs* pa = &one;
    if (jobs) {
        const int j = job_of(first, njobs, t_idx);
        t_idx -= __ldg(first + j);
        pa = jobs + j;
    }
    const HApplyArgs& A = *pa;
    const int PW = A.PW, np = PW * PW, TS = A.TS, pitch = A.pitch, plane = PW * pitch;
    float2* Z = reinterpret_cast<float2*>(hsm);               // input patch
    int* acc = reinterpret_cast<int*>(Z + np);                // planes [hi re, hi im, lo re, lo im]
    f32x2* rows = reinterpret_cast<f32x2*>(acc + 4 * plane);  // compressed rows spread out, one per warp
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tile = A.need[t_idx];
    const int tu = tile / A.ntv, tv = tile - tu * A.ntv;
    const int u0 = tu * TS, v0 = tv * TS;
    const int words = TS * TS / 32;
    for (int e = tid; e < words; e += blockDim.x) tbits[e] = A.bits[(size_t)t_idx * words + e];
    for (int e = tid; e < 4 * plane; e += blockDim.x) acc[e] = 0;
    if (tid == 0) s_zmax = 0u;
    __syncthreads();
    if (warp == 0) {  // running count over the bitmap words
        int base = 0;
        for (int q = 0; q < words; q += 32) {
            int n = __popc(tbits[q + lane]);
            const int own = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int m = __shfl_up_sync(0xffffffffu, n, o);
                if (lane >= o) n += m;
            }
            wsum[q + lane] = base + n - own;
            base += __shfl_sync(0xffffffffu, n, 31);
        }
    }
    float zm = 0.f;
    for (int e = tid; e < np; e += blockDim.x) {
        const int a = e / PW, b = e - a * PW;
        const int gu = wrap(u0 + a, A.gx), gv = wrap(v0 + b, A.gy);
        const int tt = (gu >> A.shift) * A.ntv + (gv >> A.shift);
        const float2 z = A.need_mask[tt] ? A.X[(size_t)gu * A.gy + gv] : make_float2(0.f, 0.f);
        Z[e] = z;
        zm = fmaxf(zm, fabsf(z.x) + fabsf(z.y));
    }
    zm = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(zm)));
    if (lane == 0) atomicMax(&s_zmax, __float_as_uint(zm));
    __syncthreads();
    for (int e = tid; e < TS * TS; e += blockDim.x) {
        const uint32_t w = tbits[e >> 5], m = 1u << (e & 31);
        if (w & m) cells[wsum[e >> 5] + __popc(w & (m - 1u))] = (uint16_t)e;
    }
    __syncthreads();
    // bound on one accumulated term of this tile: the gathered type-A sum, (D+1)^2
    // entries of |h|_1 <= the tile's max times |z|_1 <= the patch's max (margin 2);
    // at most 2 ne terms per cell.  Per-tile bounds keep the fixed-point resolution
    // relative to the tile's own values where H spans orders of magnitude.
    float s1 = 1.f, inv = 1.f;
    const float mt = 2.f * (float)(S * S) * __uint_as_float(__ldg(A.tmax + t_idx)) * __uint_as_float(s_zmax);
    if (mt > 0.f) {
        const float lim = fminf(2097152.f, 1073741824.f / (float)(2 * NE));
        int ex = (int)((__float_as_uint(lim / mt) >> 23) & 255u) - 127;
        ex = ex < -120 ? -120 : (ex > 120 ? 120 : ex);
        s1 = __uint_as_float((uint32_t)(ex + 127) << 23);
        inv = __uint_as_float((uint32_t)(127 - ex) << 23);
    }
    const int64_t base = A.hoff[t_idx];
    const int nown = (int)(A.hoff[t_idx + 1] - base);
    auto multiply = [&](const HRow<S>& h, int k) {
        const int cell = cells[k], lu = cell >> A.shift, lv = cell & (TS - 1);
        h_owner<S>(h, Z, acc, PW, pitch, plane, lu, lv, s1, lane);
    };
    if (A.roff == nullptr) {
        const f32x2* val = reinterpret_cast<const f32x2*>(A.val) + base * NE;
        auto fetch = [&](HRow<S>& h, int k) {
            const f32x2* row = val + (int64_t)k * NE;
            h.load(lane, [&](int e) { return (f32x2)__ldg(row + e); });
        };
        HRow<S> h0, h1;
        int k = warp;
        if (k < nown) fetch(h0, k);
        for (; k < nown; k += 2 * HA_WARPS) {
            if (k + HA_WARPS < nown) fetch(h1, k + HA_WARPS);
            multiply(h0, k);
            if (k + HA_WARPS >= nown) break;
            if (k + 2 * HA_WARPS < nown) fetch(h0, k + 2 * HA_WARPS);
            multiply(h1, k + HA_WARPS);
        }
    } else {
        f32x2* row = rows + warp * NE;
        const f32x2* val = reinterpret_cast<const f32x2*>(A.val);
        for (int k = warp; k < nown; k += HA_WARPS) {
            const int64_t q0 = __ldg(&A.roff[base + k]), q1 = __ldg(&A.roff[base + k + 1]);
            for (int e = lane; e < NE; e += 32) row[e] = 0ull;
            __syncwarp();
            for (int64_t q = q0 + lane; q < q1; q += 32 * 7) {
                f32x2 h[7];
                int e[7];
#pragma unroll
                for (int i = 0; i < 7; ++i) {
                    const bool on = q + 32 * i < q1;
                    h[i] = on ? (f32x2)__ldg(val + q + 32 * i) : 0ull;
                    e[i] = on ? (int)__ldg(A.idx + q + 32 * i) : -1;
                }
#pragma unroll
                for (int i = 0; i < 7; ++i)
                    if (e[i] >= 0) row[e[i]] = h[i];
            }
            __syncwarp();
            HRow<S> h;
            h.load(lane, [&](int e) { return row[e]; });
            multiply(h, k);
            __syncwarp();  // every lane has read the row
        }
    }
    __syncthreads();
    const float inv_lo = inv * (1.f / 65536.f);
    float2* dst = A.patch + (size_t)t_idx * np;
    for (int e = tid; e < np; e += blockDim.x) {
        const int a = e / PW, q = a * pitch + (e - a * PW);
        dst[e] = make_float2(fmaf((float)acc[q + 2 * plane], inv_lo, (float)acc[q] * inv),
                             fmaf((float)acc[q + 3 * plane], inv_lo, (float)acc[q + plane] * inv));
    }
}

static void (*happly_for(int S))(HApplyArgs, const HApplyArgs*, const int*, int) {
    switch (S) {
        case 3: return happly_kernel<3>;
        case 5: return happly_kernel<5>;
        case 7: return happly_kernel<7>;
        case 9: return happly_kernel<9>;
        case 11: return happly_kernel<11>;
        case 13: return happly_kernel<13>;
        case 15: return happly_kernel<15>;
        case 17: return happly_kernel<17>;
        default: return happly_kernel<19>;
    }
}

// (the row buffers only where some bin's rows are compressed)
size_t happly_smem(int PW, int S, bool compressed) {
    const size_t ne = (size_t)S * S + (size_t)(S - 1) * (S - 1);
    return (size_t)PW * PW * sizeof(float2) + (size_t)4 * PW * pitch_of(PW, S) * sizeof(int) +
           (compressed ? HA_WARPS * ne * sizeof(float2) : 0);
}

size_t hbuild_smem(int ne, int S_max, int D) {
    return (size_t)HB_WARPS * ne * sizeof(float2) + (size_t)HB_CHUNK * S_max * S_max * sizeof(float2) +
           HB_CHUNK * sizeof(int4) + (size_t)(ne + 2) * sizeof(int) +
           (size_t)2 * (HB_OWN + D) * (2 * sizeof(int64_t) + sizeof(int)) + 64;
}

struct DevBuf {
    void* p = nullptr;
    ~DevBuf() { cudaFree(p); }
};

// Non-zero entries of each dense owner row (one warp per row); diag[0] += the rows whose
// entry 0 (H[o][o]) is non-zero.
__global__ void __launch_bounds__(256) hrowcount_kernel(const float2* __restrict__ rows, int64_t nown, int ne,
                                                        int32_t* __restrict__ counts, unsigned long long* diag) {
    const int lane = threadIdx.x & 31;
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (r >= nown) return;
    const float2* row = rows + (size_t)r * ne;
    int n = 0;
    for (int e = lane; e < ne; e += 32) {
        const float2 h = row[e];
        n += (h.x != 0.f || h.y != 0.f) ? 1 : 0;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
    if (lane == 0) {
        counts[r] = n;
        const float2 h0 = row[0];
        if (h0.x != 0.f || h0.y != 0.f) atomicAdd(diag, 1ull);
    }
}

// Keeps the non-zero entries of each dense owner row at roff[row] (one warp per row,
// entries in row order).
__global__ void __launch_bounds__(256) hcompact_kernel(const float2* __restrict__ rows, int64_t nown, int ne,
                                                       const int64_t* __restrict__ roff, float2* __restrict__ val,
                                                       uint16_t* __restrict__ idx) {
    const int lane = threadIdx.x & 31;
    const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (r >= nown) return;
    const float2* row = rows + (size_t)r * ne;
    int64_t q = roff[r];
    for (int e0 = 0; e0 < ne; e0 += 32) {
        const int e = e0 + lane;
        const float2 h = e < ne ? row[e] : make_float2(0.f, 0.f);
        const bool on = h.x != 0.f || h.y != 0.f;
        const uint32_t m = __ballot_sync(0xffffffffu, on);
        if (on) {
            const int64_t at = q + __popc(m & ((1u << lane) - 1u));
            val[at] = h;
            idx[at] = (uint16_t)e;
        }
        q += __popc(m);
    }
}

}  // namespace

static HApplyArgs happly_args(const rimo_plan* p, int bin, const float2* X, float2* patch) {
    const auto& br = p->bins[bin];
    const size_t ntile = (size_t)(p->gx / p->TS) * (p->gy / p->TS);
    HApplyArgs A;
    std::memset(&A, 0, sizeof(A));
    A.X = X;
    A.need_mask = p->d_need + (size_t)bin * ntile;
    A.need = p->d_need_list + br.n0;
    A.bits = p->d_hbits[bin];
    A.hoff = p->d_hoff[bin];
    A.val = p->d_hval[bin];
    A.idx = p->h_dense[bin] ? nullptr : p->d_hidx[bin];
    A.roff = p->h_dense[bin] ? nullptr : p->d_hroff[bin];
    A.tmax = p->d_htmax[bin];
    A.patch = patch;
    A.gx = p->gx;
    A.gy = p->gy;
    A.ntv = p->gy / p->TS;
    A.TS = p->TS;
    A.PW = p->PW;
    A.pitch = pitch_of(p->PW, p->max_S);
    A.shift = p->TS == 64 ? 6 : 5;
    return A;
}

static void happly_launch(const rimo_plan* p, const HApplyArgs& one, const HApplyArgs* jobs, const int* first, int njobs,
                          int blocks, bool compressed, cudaStream_t s) {
    if (blocks <= 0) return;
    auto kern = happly_for(p->max_S);
    const size_t sm = happly_smem(p->PW, p->max_S, compressed);
    set_smem(kern, sm);
    kern<<<blocks, HA_WARPS * 32, sm, s>>>(one, jobs, first, njobs);
}

void launch_happly(const rimo_plan* p, int bin, cudaStream_t s) {
    happly_launch(p, happly_args(p, bin, p->d_X, p->d_hpatch), nullptr, nullptr, 0, p->bins[bin].n1 - p->bins[bin].n0,
                  !p->h_dense[bin], s);
}

// The holographic applies of a group of bins as one launch over a table of jobs.
struct WideH {
    const rimo_plan* p = nullptr;
    HApplyArgs* jobs = nullptr;
    int* first = nullptr;
    int njobs = 0, blocks = 0;
    bool compressed = false;
    ~WideH() {
        cudaFree(jobs);
        cudaFree(first);
    }
};

static WideH* wide_h_create(const rimo_plan* p, const std::vector<WideJob>& jobs, cudaStream_t s) {
    auto* w = new WideH();
    try {
        w->p = p;
        std::vector<HApplyArgs> a;
        std::vector<int> f{0};
        for (const WideJob& j : jobs) {
            a.push_back(happly_args(p, j.bin, j.X, j.patch));
            f.push_back(f.back() + (p->bins[j.bin].n1 - p->bins[j.bin].n0));
            w->compressed = w->compressed || !p->h_dense[j.bin];
        }
        w->njobs = (int)a.size();
        w->blocks = f.back();
        RIMO_CUDA(device_malloc(&w->jobs, a.size() * sizeof(HApplyArgs)));
        RIMO_CUDA(device_malloc(&w->first, f.size() * sizeof(int)));
        RIMO_CUDA(cudaMemcpyAsync(w->jobs, a.data(), a.size() * sizeof(HApplyArgs), cudaMemcpyHostToDevice, s));
        RIMO_CUDA(cudaMemcpyAsync(w->first, f.data(), f.size() * sizeof(int), cudaMemcpyHostToDevice, s));
        RIMO_CUDA(cudaStreamSynchronize(s));
    } catch (...) {
        delete w;
        throw;
    }
    return w;
}
void wide_h_destroy(WideH* w) { delete w; }
void wide_happly(const WideH* w, cudaStream_t s) {
    HApplyArgs none;
    std::memset(&none, 0, sizeof(none));
    happly_launch(w->p, none, w->jobs, w->first, w->njobs, w->blocks, w->compressed, s);
}

// Once H is built, the plan's groups of bins apply it too, with patches of their own; where
// those or the tables do not fit, or memory is not plentiful (as in stage_plan), one bin at a time.
static void stage_holographic(rimo_plan* p, int max_need, cudaStream_t s) {
    PlanStage* st = p->stage;
    if (!st) return;
    size_t most = 0;
    for (const auto& g : st->groups) most = std::max(most, g.jobs.size());
    const size_t each = (size_t)max_need * p->PW * p->PW, bytes = most * each * sizeof(float2);
    if (bytes > ((size_t)512 << 20)) return;
    size_t room = 0, total = 0;
    RIMO_CUDA(cudaMemGetInfo(&room, &total));
    if (room < 4 * bytes) return;
    try {
        RIMO_CUDA(device_malloc(&st->hpatch, bytes));
        for (auto& g : st->groups) {
            std::vector<WideJob> jobs = g.jobs;
            for (size_t k = 0; k < jobs.size(); ++k) jobs[k].patch = static_cast<float2*>(st->hpatch) + k * each;
            g.hfft = wide_fft_create(jobs, {nullptr}, {nullptr}, s, true);
            g.h = wide_h_create(p, jobs, s);
        }
    } catch (const Error& e) {
        st->drop_holographic();
        if (e.status == RIMO_ERR_CUDA) throw;
        return;
    }
    p->info.scratch_bytes += (int64_t)bytes;
}

// Builds H for every bin; see the file comment.  Synchronises s.
static void build_holographic(rimo_plan* p, cudaStream_t s) {
    const int P = p->P, TS = p->TS, D = p->H, gx = p->gx, gy = p->gy;
    const int ntu = gx / TS, ntv = gy / TS;
    const size_t ntile = (size_t)ntu * ntv;
    if (gy > 65536) fail(RIMO_ERR_UNSUPPORTED, "holographic build needs grid columns < 65536");
    if (TS * TS / 32 > 128) fail(RIMO_ERR_UNSUPPORTED, "tile too large for the coverage bitmap");
    const int ne = (D + 1) * (D + 1) + D * D;
    const int words = TS * TS / 32;

    // ---- anchor index on the host: per bin, sorted positions ordered by (g0, h0)
    std::vector<VisMeta> meta((size_t)p->M);
    RIMO_CUDA(cudaMemcpyAsync(meta.data(), p->d_meta, meta.size() * sizeof(VisMeta), cudaMemcpyDeviceToHost, s));
    RIMO_CUDA(cudaStreamSynchronize(s));
    std::vector<int32_t> g0((size_t)p->M), h0((size_t)p->M);
    for (const auto& u : p->tiles_host)
        for (int64_t i = u.vb; i < u.ve; ++i) {
            g0[i] = u.tu * TS + (int)(meta[i].pos & 255u);
            h0[i] = u.tv * TS + (int)((meta[i].pos >> 8) & 255u);
        }
    std::vector<int32_t> apos((size_t)p->M);
    std::vector<uint16_t> ah0((size_t)p->M);
    std::vector<int64_t> arow((size_t)P * (gx + 1), 0);
    planner::parallel_for(P, [&](int64_t b0, int64_t b1) {
        std::vector<int64_t> ccount;
        for (int64_t b = b0; b < b1; ++b) {
            const int64_t vb = p->bins[b].vb, ve = p->bins[b].ve;
            const int64_t n = ve - vb;
            if (n == 0) continue;
            // stable counting sort by h0, then by g0
            std::vector<int32_t> t1((size_t)n), t2((size_t)n);
            ccount.assign((size_t)gy + 1, 0);
            for (int64_t i = vb; i < ve; ++i) ccount[h0[i] + 1]++;
            for (int c = 0; c < gy; ++c) ccount[c + 1] += ccount[c];
            for (int64_t i = vb; i < ve; ++i) t1[ccount[h0[i]]++] = (int32_t)i;
            int64_t* row = &arow[(size_t)b * (gx + 1)];
            std::vector<int64_t> rc((size_t)gx + 1, 0);
            for (int64_t k = 0; k < n; ++k) rc[g0[t1[k]] + 1]++;
            for (int g = 0; g < gx; ++g) rc[g + 1] += rc[g];
            for (int g = 0; g <= gx; ++g) row[g] = vb + rc[g];  // absolute indices into pos / h0
            for (int64_t k = 0; k < n; ++k) t2[rc[g0[t1[k]]]++] = t1[k];
            for (int64_t k = 0; k < n; ++k) {
                apos[vb + k] = t2[k];
                ah0[vb + k] = (uint16_t)h0[t2[k]];
            }
        }
    }, 1);
    AnchorIndex ai;
    RIMO_CUDA(device_malloc(&ai.pos, apos.size() * sizeof(int32_t)));
    RIMO_CUDA(device_malloc(&ai.h0, ah0.size() * sizeof(uint16_t)));
    RIMO_CUDA(device_malloc(&ai.row, arow.size() * sizeof(int64_t)));
    RIMO_CUDA(cudaMemcpyAsync(ai.pos, apos.data(), apos.size() * sizeof(int32_t), cudaMemcpyHostToDevice, s));
    RIMO_CUDA(cudaMemcpyAsync(ai.h0, ah0.data(), ah0.size() * sizeof(uint16_t), cudaMemcpyHostToDevice, s));
    RIMO_CUDA(cudaMemcpyAsync(ai.row, arow.data(), arow.size() * sizeof(int64_t), cudaMemcpyHostToDevice, s));

    // ---- entry table, slots, coverage
    p->d_hent = upload_vec(p, entry_table(D), s);
    std::vector<int32_t> hslot((size_t)P * ntile, -1);
    for (int b = 0; b < P; ++b)
        for (int k = p->bins[b].n0; k < p->bins[b].n1; ++k) hslot[(size_t)b * ntile + p->need_host[k]] = k - p->bins[b].n0;
    p->d_hfold = upload_vec(p, fold_records(p, hslot, true), s);
    p->d_hbits.assign(P, nullptr);
    p->d_hoff.assign(P, nullptr);
    p->d_hval.assign(P, nullptr);
    p->d_hidx.assign(P, nullptr);
    p->d_hroff.assign(P, nullptr);
    p->h_dense.assign(P, 0);
    p->d_htmax.assign(P, nullptr);
    p->hoff_host.assign(P, {});
    int max_need = 1;
    for (int b = 0; b < P; ++b) max_need = std::max(max_need, p->bins[b].n1 - p->bins[b].n0);
    DevBuf counts;
    RIMO_CUDA(device_malloc(&counts.p, (size_t)max_need * sizeof(int64_t)));
    HArgs A;
    std::memset(&A, 0, sizeof(A));
    A.meta = p->d_meta;
    A.gblk = p->d_gblock_ptrs;
    A.apos = ai.pos;
    A.ah0 = ai.h0;
    A.ent = p->d_hent;
    A.fx = p->d_fx;
    A.gx = gx;
    A.gy = gy;
    A.ntv = ntv;
    A.TS = TS;
    A.D = D;
    A.ne = ne;
    int64_t total = 0;
    const size_t cover_sm = (size_t)2 * (TS + D) * (2 * sizeof(int64_t) + sizeof(int)) + (size_t)words * sizeof(uint32_t) + 64;
    for (int b = 0; b < P; ++b) {
        const int nneed = p->bins[b].n1 - p->bins[b].n0;
        p->d_hbits[b] = (uint32_t*)dev_alloc(p, (size_t)std::max(1, nneed) * words * sizeof(uint32_t));
        p->hoff_host[b].assign((size_t)nneed + 1, 0);
        if (nneed == 0) {
            p->d_hoff[b] = upload_vec(p, p->hoff_host[b], s);
            continue;
        }
        A.arow = ai.row + (size_t)b * (gx + 1);
        A.need = p->d_need_list + p->bins[b].n0;
        A.bits = p->d_hbits[b];
        A.count = (int64_t*)counts.p;
        hcover_kernel<<<nneed, 256, cover_sm, s>>>(A);
        RIMO_CUDA(cudaGetLastError());
        std::vector<int64_t> c((size_t)nneed);
        RIMO_CUDA(cudaMemcpyAsync(c.data(), counts.p, c.size() * sizeof(int64_t), cudaMemcpyDeviceToHost, s));
        RIMO_CUDA(cudaStreamSynchronize(s));
        for (int k = 0; k < nneed; ++k) p->hoff_host[b][k + 1] = p->hoff_host[b][k] + c[k];
        total += p->hoff_host[b][nneed];
        p->d_hoff[b] = upload_vec(p, p->hoff_host[b], s);
    }
    const size_t patch_bytes = (size_t)max_need * p->PW * p->PW * sizeof(float2);
    p->d_hpatch = (float2*)dev_alloc(p, patch_bytes);
    const size_t sm = hbuild_smem(ne, p->max_S, D);
    if (sm > 227 * 1024) fail(RIMO_ERR_UNSUPPORTED, "holographic build: owner rows exceed shared memory");
    set_smem(hbuild_kernel, sm);
    const int per_tile = (TS / HB_OWN) * (TS / HB_OWN);
    // bin by bin: dense rows into a temporary, then only their non-zero entries kept
    std::vector<void*> made;  // the compressed arrays, released again if the budget refuses
    auto keep = [&](size_t bytes) {
        void* q = dev_alloc(p, std::max<size_t>(bytes, 16));
        made.push_back(q);
        return q;
    };
    auto release_made = [&]() {
        for (void* q : made) {
            if (!q) continue;
            auto it = std::find(p->owned.begin(), p->owned.end(), q);
            if (it != p->owned.end()) p->owned.erase(it);
            cudaFree(q);
        }
        made.clear();
    };
    int64_t nnz = 0, h_bytes = 0;
    unsigned long long diag = 0;
    DevBuf dcount, ddiag;
    RIMO_CUDA(device_malloc(&ddiag.p, sizeof(unsigned long long)));
    RIMO_CUDA(cudaMemsetAsync(ddiag.p, 0, sizeof(unsigned long long), s));
    try {
        for (int b = 0; b < P; ++b) {
            const int nneed = p->bins[b].n1 - p->bins[b].n0;
            const int64_t nown = p->hoff_host[b][(size_t)nneed];
            p->d_htmax[b] = (uint32_t*)keep((size_t)std::max(1, nneed) * sizeof(uint32_t));
            RIMO_CUDA(cudaMemsetAsync(p->d_htmax[b], 0, (size_t)std::max(1, nneed) * sizeof(uint32_t), s));
            std::vector<int64_t> roff((size_t)nown + 1, 0);
            if (nown > 0) {
                DevBuf dense;
                if (device_malloc(&dense.p, (size_t)nown * ne * sizeof(float2)) != cudaSuccess) {
                    cudaGetLastError();
                    fail(RIMO_ERR_OOM, "holographic build: dense rows of one bin");
                }
                made.push_back(nullptr);  // placeholder: the dense rows may be kept
                A.arow = ai.row + (size_t)b * (gx + 1);
                A.need = p->d_need_list + p->bins[b].n0;
                A.bits = p->d_hbits[b];
                A.hoff = p->d_hoff[b];
                A.rows = (float2*)dense.p;
                A.tmax = p->d_htmax[b];
                // without stored G, the bin's exact tiles are generated into the tap scratch first
                if (p->mode != RIMO_MODE_STORED_G)
                    launch_gbuild_range(p, p->bins[b].vb, p->bins[b].ve - p->bins[b].vb, s);
                hbuild_kernel<<<nneed * per_tile, HB_WARPS * 32, sm, s>>>(A, p->max_S);
                RIMO_CUDA(cudaGetLastError());
                cudaFree(dcount.p);
                dcount.p = nullptr;
                RIMO_CUDA(device_malloc(&dcount.p, (size_t)nown * sizeof(int32_t)));
                const int64_t blocks = (nown * 32 + 255) / 256;
                hrowcount_kernel<<<(unsigned)blocks, 256, 0, s>>>((const float2*)dense.p, nown, ne, (int32_t*)dcount.p,
                                                                  (unsigned long long*)ddiag.p);
                RIMO_CUDA(cudaGetLastError());
                std::vector<int32_t> c((size_t)nown);
                RIMO_CUDA(cudaMemcpyAsync(c.data(), dcount.p, c.size() * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
                RIMO_CUDA(cudaStreamSynchronize(s));
                for (int64_t k = 0; k < nown; ++k) roff[(size_t)k + 1] = roff[(size_t)k] + c[(size_t)k];
                const int64_t nb = roff[(size_t)nown];
                const int64_t dense_bytes = nown * ne * (int64_t)sizeof(float2);
                const int64_t packed_bytes =
                    nb * (int64_t)(sizeof(float2) + sizeof(uint16_t)) + (nown + 1) * (int64_t)sizeof(int64_t);
                const bool keep_dense = dense_bytes <= packed_bytes;
                h_bytes += keep_dense ? dense_bytes : packed_bytes;
                nnz += nb;
                if (p->prm.mem_budget_bytes > 0 && p->info.g_bytes + h_bytes > p->prm.mem_budget_bytes)
                    fail(RIMO_ERR_BUDGET, "holographic matrices need more than the " +
                                              std::to_string(p->prm.mem_budget_bytes - p->info.g_bytes) +
                                              " bytes the budget leaves beyond G");
                if (keep_dense) {
                    // the bin's coverage is dense: the temporary becomes the stored rows
                    p->owned.push_back(dense.p);
                    made.back() = dense.p;
                    p->d_hval[b] = (float2*)dense.p;
                    dense.p = nullptr;
                    p->h_dense[b] = 1;
                    continue;
                }
                made.pop_back();
                p->d_hroff[b] = (int64_t*)keep(roff.size() * sizeof(int64_t));
                RIMO_CUDA(cudaMemcpyAsync(p->d_hroff[b], roff.data(), roff.size() * sizeof(int64_t),
                                          cudaMemcpyHostToDevice, s));
                p->d_hval[b] = (float2*)keep((size_t)nb * sizeof(float2));
                p->d_hidx[b] = (uint16_t*)keep((size_t)nb * sizeof(uint16_t));
                hcompact_kernel<<<(unsigned)blocks, 256, 0, s>>>((const float2*)dense.p, nown, ne, p->d_hroff[b],
                                                                 p->d_hval[b], p->d_hidx[b]);
                RIMO_CUDA(cudaGetLastError());
                RIMO_CUDA(cudaStreamSynchronize(s));  // the dense rows are freed next
            } else {
                p->d_hroff[b] = (int64_t*)keep(roff.size() * sizeof(int64_t));
                RIMO_CUDA(cudaMemcpyAsync(p->d_hroff[b], roff.data(), roff.size() * sizeof(int64_t),
                                          cudaMemcpyHostToDevice, s));
                p->d_hval[b] = (float2*)keep(16);
                p->d_hidx[b] = (uint16_t*)keep(16);
            }
        }
        RIMO_CUDA(cudaMemcpyAsync(&diag, ddiag.p, sizeof(diag), cudaMemcpyDeviceToHost, s));
        RIMO_CUDA(cudaStreamSynchronize(s));
    } catch (...) {
        cudaStreamSynchronize(s);
        release_made();
        throw;
    }
    p->info.h_entries = total * ne;              // a dense stencil per covered cell
    p->info.h_nonzero = nnz;                      // what the rows keep
    p->info.h_nnz = 2 * (nnz - (int64_t)diag) + (int64_t)diag;
    p->h_ne = ne;
    p->info.h_bytes = h_bytes + (int64_t)patch_bytes;
    p->h_built = true;
    stage_holographic(p, max_need, s);
}

}  // namespace rimo

extern "C" {

rimo_status rimo_build_holographic(rimo_plan_t p, void* stream) {
    RIMO_API_BEGIN
    if (!p) fail(RIMO_ERR_INVALID_ARG, "null plan");
    if (p->mode == RIMO_MODE_SURROGATE) fail(RIMO_ERR_UNSUPPORTED, "H is built from exact tiles");
    if (p->prm.shard_count >= 2)
        fail(RIMO_ERR_UNSUPPORTED, "H of a shard plan: not provided (shard plans apply G^dagger G)");
    if (!p->h_built) build_holographic(p, (cudaStream_t)stream);
    RIMO_API_END
}

rimo_status rimo_plan_get_holographic(rimo_plan_t p, int32_t bin, const int32_t* pairs, int64_t n,
                                      rimo_cfloat* out, void* stream) {
    RIMO_API_BEGIN
    if (!p || !pairs || !out || n < 0) fail(RIMO_ERR_INVALID_ARG, "null argument");
    if (!p->h_built) fail(RIMO_ERR_STATE, "rimo_build_holographic has not run");
    if (bin < 0 || bin >= p->P) fail(RIMO_ERR_INVALID_ARG, "bin out of range");
    cudaStream_t s = (cudaStream_t)stream;
    const int TS = p->TS, D = p->H, gx = p->gx, gy = p->gy, ntv = gy / TS;
    const int words = TS * TS / 32;
    auto wrapd = [](int d, int n) {  // signed offset of the shorter way round
        d %= n;
        if (d < 0) d += n;
        return d > n / 2 ? d - n : d;
    };
    for (int64_t q = 0; q < n; ++q) {
        int u1 = pairs[4 * q], v1 = pairs[4 * q + 1], u2 = pairs[4 * q + 2], v2 = pairs[4 * q + 3];
        int du = wrapd(u2 - u1, gx), dv = wrapd(v2 - v1, gy);
        bool conj = false;
        if (du < 0 || (du == 0 && dv < 0)) {  // H[c2][c1] = conj(H[c1][c2])
            std::swap(u1, u2);
            std::swap(v1, v2);
            du = -du;
            dv = -dv;
            conj = true;
        }
        out[q] = rimo_cfloat{0.f, 0.f};
        if (du > D || dv > D || dv < -D) continue;
        int ou, ov, e;
        if (dv >= 0) {
            ou = u1, ov = v1, e = du * (D + 1) + dv;
        } else {
            ou = u1, ov = (v2 % gy + gy) % gy, e = (D + 1) * (D + 1) + (du - 1) * D + (-dv - 1);
        }
        ou = (ou % gx + gx) % gx;
        ov = (ov % gy + gy) % gy;
        const int tile = (ou / TS) * ntv + ov / TS;
        int k = -1;
        for (int i = p->bins[bin].n0; i < p->bins[bin].n1; ++i)
            if (p->need_host[i] == tile) k = i - p->bins[bin].n0;
        if (k < 0) continue;
        std::vector<uint32_t> bm((size_t)words);
        RIMO_CUDA(cudaMemcpyAsync(bm.data(), p->d_hbits[bin] + (size_t)k * words, words * sizeof(uint32_t),
                                  cudaMemcpyDeviceToHost, s));
        RIMO_CUDA(cudaStreamSynchronize(s));
        const int cell = (ou % TS) * TS + ov % TS;
        if (!((bm[cell >> 5] >> (cell & 31)) & 1u)) continue;
        int64_t rank = 0;
        for (int w = 0; w < (cell >> 5); ++w) rank += __builtin_popcount(bm[w]);
        rank += __builtin_popcount(bm[cell >> 5] & ((1u << (cell & 31)) - 1u));
        const int64_t row = p->hoff_host[bin][(size_t)k] + rank;
        if (p->h_dense[bin]) {
            float2 h;
            RIMO_CUDA(cudaMemcpyAsync(&h, p->d_hval[bin] + (size_t)row * p->h_ne + e, sizeof(h),
                                      cudaMemcpyDeviceToHost, s));
            RIMO_CUDA(cudaStreamSynchronize(s));
            out[q] = rimo_cfloat{h.x, conj ? -h.y : h.y};
            continue;
        }
        // the row keeps its non-zero entries, in entry order: find entry e among them
        int64_t span[2];
        RIMO_CUDA(cudaMemcpyAsync(span, p->d_hroff[bin] + row, sizeof(span), cudaMemcpyDeviceToHost, s));
        RIMO_CUDA(cudaStreamSynchronize(s));
        std::vector<uint16_t> ids((size_t)(span[1] - span[0]));
        if (!ids.empty()) {
            RIMO_CUDA(cudaMemcpyAsync(ids.data(), p->d_hidx[bin] + span[0], ids.size() * sizeof(uint16_t),
                                      cudaMemcpyDeviceToHost, s));
            RIMO_CUDA(cudaStreamSynchronize(s));
        }
        const auto it = std::lower_bound(ids.begin(), ids.end(), (uint16_t)e);
        if (it == ids.end() || *it != (uint16_t)e) continue;  // a zero entry
        float2 h;
        RIMO_CUDA(cudaMemcpyAsync(&h, p->d_hval[bin] + span[0] + (it - ids.begin()), sizeof(h), cudaMemcpyDeviceToHost, s));
        RIMO_CUDA(cudaStreamSynchronize(s));
        out[q] = rimo_cfloat{h.x, conj ? -h.y : h.y};
    }
    RIMO_API_END
}

}  // extern "C"
