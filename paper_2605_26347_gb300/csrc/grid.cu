// The sparse de-gridding matrix G_p (Section 3.2, Eq. 6): de-grid (G_p), grid
// (G_p^dagger, Eq. 8) and the fused G_p^dagger G_p of Phi^dagger Phi (the build of G's
// tiles is in gbuild.cu).
//
// Layout.  Visibilities of a w-bin are sorted by the uv-tile (TS x TS grid cells)
// holding their first grid cell, and their taps are stored tile after tile, so the
// taps of consecutive visibilities of a tile are one contiguous byte range.
//
// Kernel.  Persistent thread blocks take work units (a uv-tile, or a slice of a heavy one)
// from a heaviest-first list through an atomic counter.  For a unit, the block stages the
// box of grid cells its visibilities' footprints reach (within the (TS + H)^2 patch, H =
// largest tile side - 1) in shared memory, and its warps take the unit's visibilities round
// robin, each from a ring of its own:
//   de-grid : the warp reads the visibility's S x S taps from its ring slot (half a warp per
//             tile row), gathers the patch and reduces y_k with warp shuffles;
//   grid    : it adds conj(taps) y_k into the block's shared accumulator patch (shared-memory
//             integer reductions: visibilities of different warps may overlap);
//   refill  : it starts the bulk copy (cp.async.bulk, completion on an mbarrier of the slot)
//             of the visibility after the next one, across the unit's end if need be.
// Blocks only synchronise at unit boundaries, and two or three blocks per SM hide each other's.
// What bounds it: with full units (512^2 / 2M visibilities / 4 bins, 488 per unit) the
// shared-memory pipe (86 wavefronts per visibility, 79 % busy; 328 instructions, 73 % of the
// issue slots, 5 TB/s of taps); with small units (1024^2 / 2M / 16 bins, 38 per unit) their
// boundaries and the bookkeeping per visibility (gridding: half the issue slots and half the
// pipe).  Against one block of 20 visibility warps fed by a producer
// warp through a common ring of 20-visibility chunks (386 instructions and 90 wavefronts per
// visibility, a unit's descriptors and the rows of its X box fetched one after the other):
// 512^2 case 1.06 -> 0.74 ms, 1024^2 de-grid 2.46 -> 0.70 ms and grid 1.86 -> 0.98 ms,
// 4096^2 / 24M / 32 bins 15.4 -> 9.8 ms per apply.
// The finished accumulator box is written once to the unit's slot of the patch buffer
// (slices of a split tile are then added into its first slot); the fold of the inverse
// transform sums the overlapping halos of neighbouring patches tile by tile, so the gridded
// grid is never cleared or written with global atomics.
#include <algorithm>
#include <cstring>

#include "fixed.cuh"
#include "internal.h"

namespace rimo {

__device__ __forceinline__ uint32_t smem_u32(const void* ptr) {
    return (uint32_t)__cvta_generic_to_shared(ptr);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

// try_wait suspends the thread until the phase completes or about `hint_ns` elapse.
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(100000u)
        : "memory");
    return ok != 0;
}

// Bounded wait: at most `polls` suspended polls of <= 100 us (2^15: about 3 s); never spins
// forever.
constexpr uint32_t WAIT_POLLS = 1u << 15;
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, uint32_t polls = WAIT_POLLS) {
    for (uint32_t it = 0; it < polls; ++it)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}
// Bulk asynchronous copy global -> shared (16-byte aligned, size a multiple of 16).
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// The lane with p starts a slot's copy: expected bytes and copy, predicated (with a branch around
// them the grid step of 4096^2/24M took 9.83 instead of 9.78 ms).
__device__ __forceinline__ void bulk_fill(bool p, void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %4, 0;\n\t"
        "@p mbarrier.arrive.expect_tx.shared::cta.b64 _, [%3], %2;\n\t"
        "@p cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n\t}" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar)), "r"((uint32_t)p)
        : "memory");
}

// Asynchronous 16-byte copy global -> shared of this thread (cp.async group).
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

constexpr int GTG_MAX_WARPS = 24;  // warps per block (all of them take visibilities)
constexpr int GTG_SLOTS = 2;       // tap-ring slots of a warp
constexpr int GTG_RECS = 4;        // ring of unit records
constexpr int GTG_HDR = GTG_MAX_WARPS * GTG_SLOTS * 8 + GTG_RECS * 64;  // mbarriers, unit records
constexpr int GTG_TAIL = 256;      // the last slot's tile may be read past its end (lanes beyond its columns)

struct GtgArgs {
    const UnitRec* recs;    // the launch's units, heaviest first
    int nunits;
    int* counter;           // units taken beyond the blocks' first GTG_AHEAD (zero at launch)
    const float2* X;        // forward grid [gx][gy] and patches of a one-bin launch (null when
    float2* patch;          //   the records hold the addresses of several jobs)
    const float2* y_in;
    float2* y_out;
    int gx, gy, TS, PW, pitch;
    int slot_bytes;         // taps of the largest tile
    int xbufs;              // X patch buffers: 2 (the next unit's is copied during this one) or 1
    // failure-detection test (rimo_plan_set_wait_test): ring slots are filled once and never
    // again, and the waits for taps give up after `polls`
    int stall;
    uint32_t polls;
};
constexpr int GTG_AHEAD = 2;  // units a block takes by its index; the later ones one round ahead

// Scale of one work unit of n visibilities: the largest power of two s with
// s maxterm <= min(2^21, 2^30 / n) (see the fixed-point layout in internal.h).
__device__ __forceinline__ void fx_scale(float maxterm, int n, float& s1, float& inv) {
    s1 = 1.f;
    inv = 1.f;
    if (!(maxterm > 0.f)) return;  // all contributions vanish (or the input was flagged)
    // = 2^30 / N, N = max(n, 512): with maxterm = m 2^e, 1 <= m < 2, the exponent 30 - e - ceil(log2(m N)),
    // for any normal maxterm (an approximate division gives 0 for divisors above 2^126)
    const uint32_t b = __float_as_uint(maxterm);
    const uint32_t q = __float_as_uint(__uint_as_float((b & 0x7fffffu) | 0x3f800000u) * (float)max(n, 512));
    int ex = 30 - ((int)(b >> 23) - 127) - ((int)((q + 0x7fffffu) >> 23) - 127);
    ex = ex < -120 ? -120 : (ex > 120 ? 120 : ex);
    s1 = __uint_as_float((uint32_t)(ex + 127) << 23);
    inv = __uint_as_float((uint32_t)(127 - ex) << 23);
}

// One visibility by one warp, tile side S known at compile time.
// Lane = cell: CW lanes hold the columns of a tile row (half a warp for the common sides 9 to
// 15), so one instruction covers 32 / CW rows.  A tap and a patch cell are one 64-bit shared
// load each (consecutive lanes, consecutive cells), and the four accumulator planes (real and
// imaginary parts of the words hi and lo) have a row pitch that spreads the rows of one
// instruction over all 32 banks, so a reduction of 30 of 32 lanes is one wavefront.
//   de-grid:  y = sum t x : the pair (Re t Re x, Im t Im x) by one packed multiply-add, the
//             imaginary part by two scalar ones;
//   grid:     conj(t) y s1 (s1 the unit's scale), split into the two integer words with packed
//             arithmetic on the pair (real, imaginary).
// Lanes past the last column or row hold no tap: they are cleared from y's sum and do not
// add to the patch.  Taps stay in registers between the two steps.  Against one lane per
// (column, component) with scalar arithmetic: 21 instructions and 8 shared-memory wavefronts
// per two tile rows instead of 30 and 10.
template <int S, int MODE, int PWC>  // PWC: the patch side when known at compile time, else 0
__device__ __forceinline__ void vis_tile(const float2* __restrict__ T, const float2* __restrict__ Xs, int* acc,
                                         float s1, int du, int dv, int PWr, int pitchr, int planer, int lane,
                                         uint32_t orig, float2 y, float2* __restrict__ y_out) {
    // compile-time strides fold into the address offsets
    const int PW = PWC > 0 ? PWC : PWr, pitch = PWC > 0 ? pitch_of(PWC) : pitchr;
    const int plane = PWC > 0 ? PWC * pitch_of(PWC) : planer;
    constexpr bool GATHER = MODE != 1, SCATTER = MODE != 0;
    constexpr int CW = S <= 8 ? 8 : (S <= 16 ? 16 : 32);  // lanes per tile row
    constexpr int RPI = 32 / CW;                          // rows per instruction
    constexpr int NI = (S + RPI - 1) / RPI;               // row steps
    const int c = lane % CW, ro = lane / CW;
    const bool row_ok = (NI - 1) * RPI + ro < S;          // the last step's row exists
    const f32x2* Tl = reinterpret_cast<const f32x2*>(T) + ro * S + c;
    const f32x2* Xl = reinterpret_cast<const f32x2*>(Xs) + (du + ro) * PW + dv + c;
    f32x2 t[NI];
    f32x2 p = 0ull;
    float q1 = 0.f, q2 = 0.f;
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const bool ok = (i + 1) * RPI <= S || row_ok;
        t[i] = ok ? Tl[i * RPI * S] : 0ull;
        if (GATHER) {
            const f32x2 x = ok ? Xl[i * RPI * PW] : 0ull;
            p = fma2(t[i], x, p);
            const float2 ts = upk(t[i]), xs = upk(x);
            q1 = fmaf(ts.x, xs.y, q1);
            q2 = fmaf(ts.y, xs.x, q2);
        }
    }
    if (GATHER) {
        const float2 ps = upk(p);
        const float re = c < S ? ps.x - ps.y : 0.f, im = c < S ? q1 + q2 : 0.f;
        // the low half of the warp reduces the real part, the high half the imaginary one
        const bool hi = lane & 16;
        float v = hi ? im : re;
        v += __shfl_xor_sync(0xffffffffu, hi ? re : im, 16);
        v += __shfl_xor_sync(0xffffffffu, v, 8);
        v += __shfl_xor_sync(0xffffffffu, v, 4);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        const float o = __shfl_xor_sync(0xffffffffu, v, 16);
        y = hi ? make_float2(o, v) : make_float2(v, o);
        if (MODE == 0 && lane == 0) y_out[orig] = y;
    }
    if (SCATTER) {
        const float yr = y.x * s1, yi = y.y * s1, nyr = -yr;
        int* al = acc + (du + ro) * pitch + dv + c;
        if (c < S) {
#pragma unroll
            for (int i = 0; i < NI; ++i) {
                if ((i + 1) * RPI <= S || row_ok) {
                    const float2 ts = upk(t[i]);
                    fx_add2(al + i * RPI * pitch, plane,
                            pk(fmaf(ts.x, yr, ts.y * yi), fmaf(ts.x, yi, ts.y * nyr)));
                }
            }
        }
    }
}

template <int MODE, int PWC>
__device__ __forceinline__ void vis_dispatch(int S, const float2* T, const float2* Xs, int* acc, float s1, int du,
                                             int dv, int PW, int pitch, int plane, int lane, uint32_t orig,
                                             float2 y, float2* y_out) {
    if (S == 15) {  // the largest support of the common plans, and most of their visibilities
        vis_tile<15, MODE, PWC>(T, Xs, acc, s1, du, dv, PW, pitch, plane, lane, orig, y, y_out);
        return;
    }
    switch (S) {
        case 3: vis_tile<3, MODE, PWC>(T, Xs, acc, s1, du, dv, PW, pitch, plane, lane, orig, y, y_out); break;
        case 5: vis_tile<5, MODE, PWC>(T, Xs, acc, s1, du, dv, PW, pitch, plane, lane, orig, y, y_out); break;
        case 7: vis_tile<7, MODE, PWC>(T, Xs, acc, s1, du, dv, PW, pitch, plane, lane, orig, y, y_out); break;
        case 9: vis_tile<9, MODE, PWC>(T, Xs, acc, s1, du, dv, PW, pitch, plane, lane, orig, y, y_out); break;
        case 11: vis_tile<11, MODE, PWC>(T, Xs, acc, s1, du, dv, PW, pitch, plane, lane, orig, y, y_out); break;
        case 13: vis_tile<13, MODE, PWC>(T, Xs, acc, s1, du, dv, PW, pitch, plane, lane, orig, y, y_out); break;
        default:  // larger tiles have larger patches than the compile-time ones
            if constexpr (PWC == 0) {
                if (S == 17) vis_tile<17, MODE, PWC>(T, Xs, acc, s1, du, dv, PW, pitch, plane, lane, orig, y, y_out);
                else vis_tile<19, MODE, PWC>(T, Xs, acc, s1, du, dv, PW, pitch, plane, lane, orig, y, y_out);
            }
    }
}

// The unit's box in pairs of cells (16 bytes): rows [a0, a0 + na), the columns widened to
// whole pairs, w pairs per row (PW, TS, gy are even: a pair stays within one uv-tile).
struct UnitBox {
    int a0, c0, w, n;
    uint32_t mg;  // e / w = e mg >> 20: e < 2^12 pairs, w <= 41
    __device__ __forceinline__ UnitBox(const UnitRec* rec) {
        const uint32_t box = rec->box;
        a0 = (int)(box & 255u);
        c0 = box_c0(box);
        w = box_pairs(box);
        n = ((int)((box >> 8) & 255u) - a0) * w;
        mg = rec->mg;
    }
    // pair e: patch row a, column c
    __device__ __forceinline__ void at(int e, int& a, int& c) const {
        const int r = (int)(((uint32_t)e * mg) >> 20);
        a = a0 + r;
        c = c0 + 2 * (e - r * w);
    }
};

// Starts the copies of a unit's X box into its patch buffer (rows and columns wrap), as thread t
// of nt.
template <int PWC>
__device__ __forceinline__ void stage_x(const GtgArgs& A, const UnitRec* rec, float2* dst, int t, int nt) {
    const uint32_t g = rec->geom;
    const int PW = PWC > 0 ? PWC : (int)(g >> 16);
    const int u0 = (int)(g & 255u) * A.TS, v0 = (int)((g >> 8) & 255u) * A.TS;
    const float2* X = reinterpret_cast<const float2*>(reinterpret_cast<const char*>(A.X) + rec->X);
    const UnitBox B(rec);
    for (int e = t; e < B.n; e += nt) {
        int a, c;
        B.at(e, a, c);
        int gu = u0 + a, gv = v0 + c;
        if (gu >= A.gx) gu -= A.gx;
        if (gv >= A.gy) gv -= A.gy;
        cp_async16(dst + a * PW + c, X + (size_t)gu * A.gy + gv);
    }
}

// The visibilities of one warp in the order it takes them, unit after unit, in batches of up
// to 32 held one per lane, and the metadata of the batch after the current one.
struct VisCursor {
    int round, base, n;    // the unit's round, the batch's first visibility, the warp's share
    int b, nb;             // next of the batch, its size
    const float2* src;     // the lane's visibility: taps, their bytes, VisMeta::pos and orig
    uint32_t bytes, pos, orig;
    bool ready;            // nxt is loaded
    int4 nxt;
};

// visibilities of a warp: ceil((nvis - warp) / nw), mgw = ceil(2^20 / nw) (nvis <= 2^15)
__device__ __forceinline__ int unit_share(int nvis, int warp, int nw, uint32_t mgw) {
    return (int)(((uint64_t)(uint32_t)max(nvis - warp + nw - 1, 0) * mgw) >> 20);
}
__device__ __forceinline__ int4 load_meta(const UnitRec* rec, int k, int warp, int nw) {
    const int i = warp + k * nw;
    return i < rec->nvis ? __ldg(reinterpret_cast<const int4*>(rec->meta + i)) : make_int4(0, 0, 0, 0);
}

// MODE 0: de-grid (y_out), 1: grid (y_in), 2: fused de-grid + grid; PWC: the patch side
// when known at compile time (the common plans), else 0
// The units may be those of many (plan, bin) jobs: a record holds its job's addresses.
//
// Per round (unit) r of a block:
//   open  : the X box copied during round r - 1 has landed; its max |X| sets the scale;
//   barrier A; the copy of round r + 1's X box starts (other buffer);
//   visibilities, each warp on its own;
//   barrier B; close: the accumulator box goes to the unit's patch slot and back to zero.
// Unit numbers are taken from the counter one round ahead (of the next round's prefetches), so
// that no round waits for its descriptors and the last units still spread over the blocks.
template <int MODE, int PWC>
__global__ void __launch_bounds__(GTG_MAX_WARPS * 32, 1) gtg_kernel(const __grid_constant__ GtgArgs A) {
    constexpr bool GATHER = MODE != 1, SCATTER = MODE != 0;
    extern __shared__ __align__(128) unsigned char smraw[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smraw);  // [warp][slot] taps landed
    UnitRec* recs = reinterpret_cast<UnitRec*>(smraw + GTG_MAX_WARPS * GTG_SLOTS * 8);
    // shared memory laid out for the launch's largest patch (the jobs of a table may have
    // different patch sides; every unit uses its own job's)
    const int PWmax = PWC > 0 ? PWC : A.PW, npmax = PWmax * PWmax;
    const int pitch = PWC > 0 ? pitch_of(PWC) : A.pitch, plane = PWmax * pitch;
    const int NX = A.xbufs;
    float2* Xbuf0 = reinterpret_cast<float2*>(smraw + GTG_HDR);
    int* acc = reinterpret_cast<int*>(Xbuf0 + (GATHER ? NX * npmax : 0));  // planes [hi re, hi im, lo re, lo im]
    unsigned char* ring = reinterpret_cast<unsigned char*>(acc + (SCATTER ? 4 * plane : 0));
    __shared__ int s_idx[GTG_RECS];    // unit of round q (q % GTG_RECS)
    __shared__ uint32_t s_xm[2];       // max |X| of the unit's box (float bits), by round parity

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const int G = gridDim.x;
    const uint32_t mgw = ((1u << 20) + nw - 1) / nw;
    uint64_t* const wfull = full + warp * GTG_SLOTS;
    unsigned char* const wring = ring + (size_t)warp * GTG_SLOTS * A.slot_bytes;
    if (lane == 0)
        for (int b = 0; b < GTG_SLOTS; ++b) mbar_init(&wfull[b], 1);
    if (tid < GTG_AHEAD) s_idx[tid] = blockIdx.x + tid * G;
    if (tid < 2) s_xm[tid] = 0u;
    if (tid < 4 * GTG_AHEAD) {  // their records (16 bytes per thread)
        const int q = tid >> 2, idx = blockIdx.x + q * G;
        if (idx < A.nunits)
            reinterpret_cast<int4*>(recs + q)[tid & 3] =
                __ldg(reinterpret_cast<const int4*>(A.recs + idx) + (tid & 3));
    }
    if (SCATTER)
        for (int e = tid; e < 4 * plane; e += blockDim.x) acc[e] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncthreads();

    // the last third of the warps (the smallest shares of a small unit) copies the X boxes and
    // finds their maxima
    const int st0 = (nw - (nw + 2) / 3) * 32, stn = (int)blockDim.x - st0;
    if (GATHER && tid >= st0) stage_x<PWC>(A, recs, Xbuf0, tid - st0, stn);  // round 0 (every block has a first unit)
    cp_async_commit();

    // ---- this warp's visibilities
    VisCursor C;
    auto unpack = [&](const float2* taps, const int4& m) {  // a lane's visibility of the new batch
        const uint32_t S = ((uint32_t)m.w >> 16) & 255u, n = S * S;
        C.src = taps + (int64_t)(((uint64_t)(uint32_t)m.y << 32) | (uint32_t)m.x);
        C.bytes = (n + (n & 1u)) * (uint32_t)sizeof(float2);
        C.pos = (uint32_t)m.w;
        C.orig = (uint32_t)m.z;
    };
    // loads the batch after the current one, if its unit's record is there in round r
    auto look_ahead = [&](int r) {
        if (C.base + 32 < C.n) {
            C.nxt = load_meta(recs + C.round % GTG_RECS, C.base + 32 + lane, warp, nw);
            C.ready = true;
        } else if (C.round <= r && s_idx[(C.round + 1) % GTG_RECS] < A.nunits) {
            const UnitRec* rec = recs + (C.round + 1) % GTG_RECS;
            if (warp < rec->nvis) {
                C.nxt = load_meta(rec, lane, warp, nw);
                C.ready = true;
            }
        }
    };
    // the next batch, of the unit of round r + 1 at most; false: none
    auto advance = [&](int r) {
        if (A.stall) return false;
        if (C.base + 32 < C.n) {
            C.base += 32;
        } else {
            do {
                if (C.round > r || s_idx[(C.round + 1) % GTG_RECS] >= A.nunits) return false;
                ++C.round;
                C.base = C.n = C.b = C.nb = 0;  // (a unit of fewer visibilities has none for this warp)
            } while (warp >= recs[C.round % GTG_RECS].nvis);
            C.n = unit_share(recs[C.round % GTG_RECS].nvis, warp, nw, mgw);
        }
        const UnitRec* rec = recs + C.round % GTG_RECS;
        unpack(rec->taps, C.ready ? C.nxt : load_meta(rec, C.base + lane, warp, nw));
        C.b = 0;
        C.nb = min(32, C.n - C.base);
        C.ready = false;
        look_ahead(r);
        return true;
    };
    C.round = C.base = C.b = 0;
    C.n = unit_share(recs[0].nvis, warp, nw, mgw);
    C.nb = min(32, C.n);
    unpack(recs[0].taps, load_meta(recs, lane, warp, nw));
    C.ready = false;
    look_ahead(0);
    int inflight = 0, islot = 0, tslot = 0;  // copies under way or landed; next slots to fill and to take
    uint32_t tphase = 0;
    uint32_t posA = 0, posB = 0, origA = 0, origB = 0;  // of the visibilities in slots 0 and 1
    float2 yA = make_float2(0.f, 0.f), yB = yA;
    // starts the copy of the next visibility's taps (and the load of its y when gridding)
    auto refill = [&](int r) {
        if (C.b >= C.nb && !advance(r)) return;
        bulk_fill(lane == C.b, wring + islot * A.slot_bytes, C.src, C.bytes, &wfull[islot]);
        const uint32_t pos = __shfl_sync(0xffffffffu, C.pos, C.b);
        const uint32_t orig = MODE != 2 ? __shfl_sync(0xffffffffu, C.orig, C.b) : 0u;
        if (islot) {
            posB = pos;
            origB = orig;
            if (MODE == 1) yB = __ldg(&A.y_in[orig]);
        } else {
            posA = pos;
            origA = orig;
            if (MODE == 1) yA = __ldg(&A.y_in[orig]);
        }
        ++C.b;
        ++inflight;
        islot ^= 1;
    };
    if (A.stall && C.nb > GTG_SLOTS) C.nb = GTG_SLOTS;
    refill(0);
    refill(0);

    const uint32_t* fxp = nullptr;  // the bounds read last (one plan: read once)
    float fx0 = 0.f, fx1 = 0.f;
    bool bad = false;
    for (int r = 0;; ++r) {
        const UnitRec* rec = recs + r % GTG_RECS;
        const bool have = s_idx[r % GTG_RECS] < A.nunits;
        const int PW = PWC > 0 ? PWC : (have ? (int)(rec->geom >> 16) : A.PW);
        float2* Xs = Xbuf0 + (NX == 2 && (r & 1) ? npmax : 0);
        cp_async_wait_all();
        if (MODE == 2 && have && tid >= st0) {
            // max |X| of the pairs this thread copied
            float xm = 0.f;
            const UnitBox B(rec);
            for (int e = tid - st0; e < B.n; e += stn) {
                int a, c;
                B.at(e, a, c);
                const float4 x = *reinterpret_cast<const float4*>(Xs + a * PW + c);
                const float m0 = fabsf(x.x) + fabsf(x.y), m1 = fabsf(x.z) + fabsf(x.w);
                if (m0 <= 3.4028234e38f) xm = fmaxf(xm, m0);  // non-finite input is flagged elsewhere
                if (m1 <= 3.4028234e38f) xm = fmaxf(xm, m1);
            }
            const uint32_t wm = __reduce_max_sync(0xffffffffu, __float_as_uint(xm));
            if (lane == 0) atomicMax(&s_xm[r & 1], wm);
        }
        // barrier A: the box, the cleared accumulators and the unit ring are visible; every
        // warp learns of a failed wait
        if (__syncthreads_or(bad) || !have) break;
        int next_idx = 0;
        if (tid == (nw - 1) * 32) next_idx = atomicAdd(A.counter, 1) + GTG_AHEAD * G;
        const bool more = s_idx[(r + 1) % GTG_RECS] < A.nunits;
        if (GATHER && NX == 2 && more && tid >= st0)
            stage_x<PWC>(A, recs + (r + 1) % GTG_RECS, Xbuf0 + (r & 1 ? 0 : npmax), tid - st0, stn);
        if (!C.ready && more) look_ahead(r);
        if (warp == nw - 1) {  // the unit of round r + 2 and its record (this warp has the smallest share)
            next_idx = __shfl_sync(0xffffffffu, next_idx, 0);
            const int q = (r + 2) % GTG_RECS;
            if (lane == 0) s_idx[q] = next_idx;
            if (lane < 4 && next_idx < A.nunits)
                cp_async16(reinterpret_cast<int4*>(recs + q) + lane,
                           reinterpret_cast<const int4*>(A.recs + next_idx) + lane);
        }
        cp_async_commit();

        const int nvis = rec->nvis;
        float s1 = 1.f, inv_s1 = 1.f;
        if (MODE == 2) {
            // per-unit bound: a de-gridded y of this unit has |y.x| + |y.y| <= 2 T1 max|X|_1
            // over the box, a contribution component at most tmax times that (margin 2)
            const float xmax = __uint_as_float(s_xm[r & 1]);
            if (rec->fx != fxp) {
                fxp = rec->fx;
                fx0 = __uint_as_float(__ldg(fxp + FX_TMAX));
                fx1 = __uint_as_float(__ldg(fxp + FX_T1));
            }
            const float mt = 4.f * fx0 * fx1 * xmax;
            fx_scale(mt, nvis, s1, inv_s1);
            if (tid == 0) s_xm[(r + 1) & 1] = 0u;  // last read in round r - 1, next used in round r + 1
        } else if (SCATTER) {
            // twice tmax max|y|_1 (rounding margin); both words final before this launch
            if (rec->fx != fxp) {
                fxp = rec->fx;
                fx0 = __uint_as_float(__ldg(fxp + FX_TMAX));
                fx1 = __uint_as_float(__ldg(fxp + FX_YB));
            }
            const float mt = 2.f * fx0 * fx1;
            if (!(mt <= 3.4028234e38f)) atomicExch(rec->status, 3);
            fx_scale(mt, nvis, s1, inv_s1);
        }
        // (nothing is in flight after a unit that left this warp no visibility)
        if (inflight == 0) {
            refill(r);
            refill(r);
        }
        const int mine = unit_share(nvis, warp, nw, mgw);
        for (int k = 0; k < mine; ++k) {
            // the taps have mostly landed: one test first (the polling loop alone: 10.08 instead of 9.83
            // ms per 4096^2/24M apply, 512^2/2M 0.765 instead of 0.742)
            if (!__all_sync(0xffffffffu, mbar_try_wait(&wfull[tslot], tphase)) &&
                !__all_sync(0xffffffffu, mbar_wait_bounded(&wfull[tslot], tphase, A.polls))) {
                bad = true;
                if (lane == 0) atomicExch(rec->status, 1);
                break;
            }
            const uint32_t pos = tslot ? posB : posA, orig = tslot ? origB : origA;
            const float2 y = MODE == 1 ? (tslot ? yB : yA) : make_float2(0.f, 0.f);
            const int du = pos & 255, dv = (pos >> 8) & 255, S = (pos >> 16) & 255;
            vis_dispatch<MODE, PWC>(S, reinterpret_cast<const float2*>(wring + tslot * A.slot_bytes), Xs, acc, s1, du,
                                    dv, PW, pitch, plane, lane, orig, y, A.y_out);
            __syncwarp();  // every lane has read the slot
            --inflight;
            tphase ^= (uint32_t)tslot;
            tslot ^= 1;
            refill(r);
        }
        if (SCATTER || NX == 1) __syncthreads();  // barrier B
        if (GATHER && NX == 1 && more && tid >= st0) {
            stage_x<PWC>(A, recs + (r + 1) % GTG_RECS, Xbuf0, tid - st0, stn);
            cp_async_commit();
        }
        if (SCATTER) {
            // the box of the patch (the fold and the merge read no cell outside it)
            float2* dst = reinterpret_cast<float2*>(reinterpret_cast<char*>(A.patch) + rec->patch);
            const float inv_lo = inv_s1 * (1.f / 65536.f);
            const UnitBox B(rec);
            for (int e = tid; e < B.n; e += blockDim.x) {
                int a, c;
                B.at(e, a, c);
                int2* q = reinterpret_cast<int2*>(acc + a * pitch + c);
                const int2 hr = q[0], hi = q[plane / 2], lr = q[plane], li = q[3 * plane / 2];
                q[0] = q[plane / 2] = q[plane] = q[3 * plane / 2] = make_int2(0, 0);
                *reinterpret_cast<float4*>(dst + a * PW + c) =
                    make_float4(fmaf((float)lr.x, inv_lo, (float)hr.x * inv_s1),
                                fmaf((float)li.x, inv_lo, (float)hi.x * inv_s1),
                                fmaf((float)lr.y, inv_lo, (float)hr.y * inv_s1),
                                fmaf((float)li.y, inv_lo, (float)hi.y * inv_s1));
            }
        }
    }
    // copies in flight land before the block may exit
    cp_async_wait_all();
    for (; inflight > 0; --inflight) {
        (void)mbar_wait_bounded(&wfull[tslot], tphase);
        tphase ^= (uint32_t)tslot;
        tslot ^= 1;
    }
}

// Adds the patches of the extra units of each split tile into its first unit's slot.
// TABLE: job j (one (plan, bin) of a batch) owns blocks [first[j], first[j + 1]).
struct MergeJob {
    float2* patch;
    const int2* groups;   // (first slot, units) of the bin's split tiles
    int npatch;           // cells of one patch
};

template <bool TABLE>
__global__ void __launch_bounds__(256) merge_patches_kernel(const __grid_constant__ MergeJob one,
                                                            const MergeJob* __restrict__ jobs,
                                                            const int* __restrict__ first, int njobs) {
    int bk = (int)blockIdx.x;
    const MergeJob* J = &one;
    if constexpr (TABLE) {
        const int j = job_of(first, njobs, bk);
        bk -= __ldg(first + j);
        J = jobs + j;
    }
    const int2 gr = J->groups[bk];
    float2* patch = J->patch;
    const int npatch = J->npatch;
    float2* dst = patch + (size_t)gr.x * npatch;
    for (int e = threadIdx.x; e < npatch; e += blockDim.x) {
        float2 acc = dst[e];
        for (int q = 1; q < gr.y; ++q) {
            const float2 v = patch[(size_t)(gr.x + q) * npatch + e];
            acc.x += v.x;
            acc.y += v.y;
        }
        dst[e] = acc;
    }
}

static size_t gtg_smem(int PW, int pitch, int slot_bytes, int mode, int warps, int xbufs) {
    return GTG_HDR + (mode != 1 ? (size_t)xbufs * PW * PW * sizeof(float2) : 0) +
           (mode != 0 ? (size_t)4 * PW * pitch * sizeof(int) : 0) + (size_t)warps * GTG_SLOTS * slot_bytes + GTG_TAIL;
}

// Launch shape of the grid step for patches of side PW and tiles of side max_S; `mode` as in
// launch_gtg.  24 warps per SM, as three, two or one block, the most blocks that fit: a
// block's unit boundaries then hide behind the other blocks' visibilities (15 x 15 tiles on
// 32-wide uv-tiles: three blocks when only de-gridding or gridding, two when fused).  A
// single block gives up its second X buffer when that leaves fewer than 16 warps a ring.
struct GtgShape {
    int warps, blocks_per_sm;
    size_t smem;
};
static GtgShape gtg_shape(const rimo_plan* p, int PW, int max_S, int mode, GtgArgs& A) {
    const int n = max_S * max_S;
    A.gx = p->gx;
    A.gy = p->gy;
    A.TS = p->TS;
    A.PW = PW;
    A.pitch = pitch_of(PW, max_S);
    A.slot_bytes = (n + (n & 1)) * (int)sizeof(float2);
    A.stall = p->test_stall;
    A.polls = p->test_stall ? p->test_polls : WAIT_POLLS;
    GtgShape g{};
    A.xbufs = 2;
    for (g.blocks_per_sm = 3; g.blocks_per_sm >= 2; --g.blocks_per_sm) {
        g.warps = GTG_MAX_WARPS / g.blocks_per_sm;
        g.smem = gtg_smem(PW, A.pitch, A.slot_bytes, mode, g.warps, 2);
        // 228 KB per SM, 1 KB of each block's share reserved, 512 bytes for static shared memory
        if (g.smem + 1024 + 512 <= (size_t)(228 * 1024) / g.blocks_per_sm) return g;
    }
    for (A.xbufs = 2; A.xbufs >= 1; --A.xbufs)
        for (g.warps = GTG_MAX_WARPS; g.warps >= (A.xbufs == 2 ? 16 : 1); --g.warps) {
            g.smem = gtg_smem(PW, A.pitch, A.slot_bytes, mode, g.warps, A.xbufs);
            if (g.smem <= 226 * 1024) return g;
        }
    fail(RIMO_ERR_UNSUPPORTED, "tile patch and tap ring exceed shared memory");
}

// the kernel instance: patch sides of the uv-tiles 32 and 64 with 15 x 15 tiles are
// compile-time constants
template <int MODE>
static void (*gtg_kernel_for(int PW))(GtgArgs) {
    return PW == 46 ? gtg_kernel<MODE, 46> : PW == 78 ? gtg_kernel<MODE, 78> : gtg_kernel<MODE, 0>;
}

template <int MODE>
static void gtg_run(const rimo_plan* p, int bin, const float2* y_in, float2* y_out, cudaStream_t s) {
    const auto& br = p->bins[bin];
    const int nu = br.t1 - br.t0;
    if (nu <= 0) return;
    GtgArgs A;
    std::memset(&A, 0, sizeof(A));
    A.recs = p->d_recs + br.t0;
    A.nunits = nu;
    A.counter = p->d_counter + bin;  // zeroed at the start of every apply
    A.X = p->d_X;
    A.patch = p->d_patch;
    A.y_in = y_in;
    A.y_out = y_out;
    const GtgShape g = gtg_shape(p, p->PW, p->max_S, MODE, A);
    void (*kern)(GtgArgs) = gtg_kernel_for<MODE>(p->PW);
    set_smem(kern, g.smem);
    kern<<<std::min(nu, p->n_sm * g.blocks_per_sm), g.warps * 32, g.smem, s>>>(A);
    if (MODE != 0 && br.m1 > br.m0) {
        MergeJob mj;
        mj.patch = A.patch;
        mj.groups = p->d_merge + br.m0;
        mj.npatch = p->PW * p->PW;
        merge_patches_kernel<false><<<br.m1 - br.m0, 256, 0, s>>>(mj, nullptr, nullptr, 0);
    }
}

// ---------------------------------------------------------------------------
// The grid step of a stage-batched apply: one persistent launch over the units of every
// (plan, bin) job, taken heaviest first from one list, then one merge launch.
struct WideGtg {
    const rimo_plan* p0 = nullptr;
    int merge_blocks = 0, njobs = 0;
    int PW = 0, max_S = 0;   // the jobs' largest patch and tile sides
    bool one_pw = true;      // one patch side: its compile-time kernel; several: the kernel reading each record's
    UnitRec* recs = nullptr;
    MergeJob* mjobs = nullptr;
    int* mfirst = nullptr;
    int* counter = nullptr;
    int* own_counter = nullptr;
    int64_t units = 0;
    ~WideGtg() {
        cudaFree(recs);  // and mjobs, mfirst
        cudaFree(own_counter);
    }
};

WideGtg* wide_gtg_create(const std::vector<WideJob>& jobs, int* counter, cudaStream_t s) {
    if (jobs.empty()) fail(RIMO_ERR_INVALID_ARG, "no jobs");
    auto* w = new WideGtg();
    try {
        const rimo_plan* p0 = jobs[0].p;
        w->p0 = p0;
        for (const WideJob& j : jobs) {
            w->PW = std::max(w->PW, j.p->PW);
            w->max_S = std::max(w->max_S, j.p->max_S);
            w->one_pw = w->one_pw && j.p->PW == p0->PW;
        }
        std::vector<MergeJob> mj;
        std::vector<int> mf{0};
        // a sort key per unit, heaviest first over all jobs (ties: job, then the bin's order): the
        // jobs' units come heaviest first already, so their runs are merged two by two
        std::vector<uint64_t> key;
        std::vector<std::pair<const UnitRec*, int>> unit;  // the plan's record, the job
        std::vector<size_t> seg{0};
        size_t nrec = 0;
        for (const WideJob& j : jobs) nrec += (size_t)(j.p->bins[j.bin].t1 - j.p->bins[j.bin].t0);
        // (a unit index plus the blocks' look-ahead stays an int)
        if (nrec > (size_t)0x7fffffff - 8 * 4096) fail(RIMO_ERR_UNSUPPORTED, "too many work units for one launch");
        key.reserve(nrec);
        unit.reserve(nrec);
        for (size_t j = 0; j < jobs.size(); ++j) {
            const rimo_plan* p = jobs[j].p;
            if (p->TS != p0->TS || p->gx != p0->gx || p->gy != p0->gy)
                fail(RIMO_ERR_UNSUPPORTED, "jobs of one grid-step launch need one grid and uv-tile size");
            const auto& br = p->bins[jobs[j].bin];
            for (int u = br.t0; u < br.t1; ++u) {
                const UnitRec& q = p->recs_host[(size_t)u];
                key.push_back(((uint64_t)(0xffffffffu - (uint32_t)q.nvis) << 32) | (uint32_t)unit.size());
                unit.push_back({&q, (int)j});
            }
            seg.push_back(key.size());
            MergeJob m;
            m.patch = jobs[j].patch;
            m.groups = p->d_merge + br.m0;
            m.npatch = p->PW * p->PW;
            mj.push_back(m);
            mf.push_back(mf.back() + (br.m1 - br.m0));
        }
        for (; seg.size() > 2;) {
            std::vector<size_t> up{0};
            for (size_t k = 2; k < seg.size(); k += 2) {
                std::inplace_merge(key.begin() + (long)seg[k - 2], key.begin() + (long)seg[k - 1], key.begin() + (long)seg[k]);
                up.push_back(seg[k]);
            }
            if (seg.size() % 2 == 0) up.push_back(seg.back());
            seg.swap(up);
        }
        std::vector<UnitRec> recs;
        recs.reserve(nrec);
        for (const uint64_t k : key) {
            const auto& u = unit[(uint32_t)k];
            recs.push_back(*u.first);
            recs.back().X = (int64_t)(uintptr_t)jobs[(size_t)u.second].X;
            recs.back().patch += (int64_t)(uintptr_t)jobs[(size_t)u.second].patch;
        }
        w->units = (int64_t)recs.size();
        w->njobs = (int)jobs.size();
        w->merge_blocks = mf.back();
        // one allocation: records, merge jobs, their first blocks
        const size_t at_m = recs.size() * sizeof(UnitRec), at_f = at_m + mj.size() * sizeof(MergeJob);
        char* mem = nullptr;
        RIMO_CUDA(device_malloc(&mem, at_f + mf.size() * sizeof(int)));
        w->recs = reinterpret_cast<UnitRec*>(mem);
        w->mjobs = reinterpret_cast<MergeJob*>(mem + at_m);
        w->mfirst = reinterpret_cast<int*>(mem + at_f);
        if (!counter) RIMO_CUDA(device_malloc(&w->own_counter, sizeof(int)));
        w->counter = counter ? counter : w->own_counter;
        if (!recs.empty())
            RIMO_CUDA(cudaMemcpyAsync(w->recs, recs.data(), recs.size() * sizeof(UnitRec), cudaMemcpyHostToDevice, s));
        RIMO_CUDA(cudaMemcpyAsync(w->mjobs, mj.data(), mj.size() * sizeof(MergeJob), cudaMemcpyHostToDevice, s));
        RIMO_CUDA(cudaMemcpyAsync(w->mfirst, mf.data(), mf.size() * sizeof(int), cudaMemcpyHostToDevice, s));
        RIMO_CUDA(cudaStreamSynchronize(s));
    } catch (...) {
        delete w;
        throw;
    }
    return w;
}

void wide_gtg_destroy(WideGtg* w) { delete w; }

int64_t wide_gtg_units(const WideGtg* w) { return w->units; }

int wide_gtg(const WideGtg* w, int mode, const float2* y_in, float2* y_out, cudaStream_t s) {
    if (w->units == 0) return 0;
    GtgArgs A;
    std::memset(&A, 0, sizeof(A));
    const GtgShape g = gtg_shape(w->p0, w->PW, w->max_S, mode, A);
    A.recs = w->recs;
    A.nunits = (int)w->units;
    A.counter = w->counter;
    A.y_in = y_in;
    A.y_out = y_out;
    const int pw = w->one_pw ? w->PW : 0;
    void (*kern)(GtgArgs) = mode == 0 ? gtg_kernel_for<0>(pw) : mode == 1 ? gtg_kernel_for<1>(pw) : gtg_kernel_for<2>(pw);
    set_smem(kern, g.smem);
    if (w->own_counter) RIMO_CUDA(cudaMemsetAsync(w->counter, 0, sizeof(int), s));
    kern<<<(int)std::min<int64_t>(w->units, (int64_t)w->p0->n_sm * g.blocks_per_sm), g.warps * 32, g.smem, s>>>(A);
    if (mode == 0 || w->merge_blocks == 0) return 1;
    MergeJob none;
    none.patch = nullptr;
    none.groups = nullptr;
    none.npatch = 0;
    merge_patches_kernel<true><<<w->merge_blocks, 256, 0, s>>>(none, w->mjobs, w->mfirst, w->njobs);
    return 2;
}

void launch_gtg(const rimo_plan* p, int bin, int mode, const float2* y_in, float2* y_out,
                cudaStream_t s) {
    if (mode == 0) gtg_run<0>(p, bin, y_in, y_out, s);
    else if (mode == 1) gtg_run<1>(p, bin, y_in, y_out, s);
    else gtg_run<2>(p, bin, y_in, y_out, s);
}

// ---------------------------------------------------------------------------
// Bound on the y of Phi^dagger y: max_k(|y_k.x| + |y_k.y|) goes to d_fx[FX_YB] (a grid-step
// contribution component is at most that times max_taps(|t.x| + |t.y|)).  Non-finite y
// sets status 3.  The last block to finish (counter in d_fx[FX_COUNT]) writes the bound and
// resets the running words.
__global__ void __launch_bounds__(256) y_bound_kernel(const float2* __restrict__ y, int64_t M, uint32_t* fx,
                                                      int* status) {
    float mx = 0.f;
    bool bad = false;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < M; k += (int64_t)gridDim.x * blockDim.x) {
        const float2 v = y[k];
        const float m = fabsf(v.x) + fabsf(v.y);
        bad |= !(m <= 3.4028234e38f);
        mx = fmaxf(mx, m);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) atomicMax(fx + FX_YMAX, __float_as_uint(mx));
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicExch(status, 3);
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(fx + FX_COUNT, 1u) == gridDim.x - 1;
    __syncthreads();
    if (last && threadIdx.x == 0) {
        __threadfence();
        // the gridding step combines it with the tap bound current when it runs (tiles
        // generated per bin at apply time raise the tap bound bin by bin)
        fx[FX_YB] = atomicExch(fx + FX_YMAX, 0u);
        fx[FX_COUNT] = 0u;
    }
}

void launch_y_bound(const rimo_plan* p, const float2* y, cudaStream_t s) {
    if (p->M == 0) return;
    const int64_t want = (p->M + 255) / 256;
    const int blocks = (int)std::min<int64_t>(want, std::min<int64_t>(FX_NPART, 4 * (int64_t)p->n_sm));
    y_bound_kernel<<<blocks, 256, 0, s>>>(y, p->M, p->d_fx, p->d_status);
}

}  // namespace rimo
