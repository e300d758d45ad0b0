// Application of Phi (Eq. 6), Phi^dagger and Phi^dagger Phi (Eq. 7, Eq. 8) and the PSF.
// Per w-bin p the work is a fixed sequence of launches on the caller's stream:
//   F Z_p        : forward rows pass, forward cols pass          (fft.cu)
//   G_p / G_p^H  : uv-tile de-grid / grid / fused G^H G           (grid.cu)
//   Z_p^H F^H    : inverse cols pass, inverse rows pass (+ accumulate over p)
#include <algorithm>
#include <memory>

#include "internal.h"

namespace rimo {

static cudaEvent_t prof_event(rimo_plan* p) {
    if (!p->prof_pool.empty()) {
        cudaEvent_t e = p->prof_pool.back();
        p->prof_pool.pop_back();
        return e;
    }
    cudaEvent_t e;
    RIMO_CUDA(cudaEventCreate(&e));
    return e;
}

void prof_begin(rimo_plan* p, int stage, cudaStream_t s) {
    if (!p->prof_on) return;
    p->prof_open_stage = stage;
    p->prof_open_event = prof_event(p);
    RIMO_CUDA(cudaEventRecord(p->prof_open_event, s));
}

void prof_end(rimo_plan* p, int launches, cudaStream_t s) {
    if (!p->prof_on || p->prof_open_stage < 0) return;
    cudaEvent_t b = prof_event(p);
    RIMO_CUDA(cudaEventRecord(b, s));
    p->prof_pending.push_back({p->prof_open_stage, launches, p->prof_open_event, b});
    p->prof_open_stage = -1;
    p->prof_open_event = nullptr;
}

static void prof_collect(rimo_plan* p) {
    for (auto& m : p->prof_pending) {
        RIMO_CUDA(cudaEventSynchronize(m.b));
        float ms = 0.f;
        RIMO_CUDA(cudaEventElapsedTime(&ms, m.a, m.b));
        p->prof_ms[m.stage] += ms;
        p->prof_launches[m.stage] += m.launches;
        p->prof_pool.push_back(m.a);
        p->prof_pool.push_back(m.b);
    }
    p->prof_pending.clear();
}

static int gtg_launches(const rimo_plan* p, int b) { return p->bins[b].t1 > p->bins[b].t0 ? 1 : 0; }

static void check_plan(rimo_plan* p) {
    if (!p) fail(RIMO_ERR_INVALID_ARG, "null plan");
}

static bool bin_empty(const rimo_plan* p, int b) { return p->bins[b].ve == p->bins[b].vb; }

static void zero_image(rimo_plan* p, rimo_cfloat* out, cudaStream_t s) {
    RIMO_CUDA(cudaMemsetAsync(out, 0, (size_t)p->nx * p->ny * sizeof(float2), s));
}

static void fwd(rimo_plan* p, int b, const float2* x, cudaStream_t s) {
    prof_begin(p, ST_FWD_ROWS, s);
    launch_fwd_rows(p, b, x, p->d_AB, s);
    prof_end(p, 1, s);
    prof_begin(p, ST_FWD_COLS, s);
    launch_fwd_cols(p, b, p->d_AB, p->d_X, s);
    prof_end(p, 1, s);
}

static void reset_schedulers(rimo_plan* p, cudaStream_t s) {
    RIMO_CUDA(cudaMemsetAsync(p->d_counter, 0, (size_t)p->P * sizeof(int32_t), s));
}

static void inv(rimo_plan* p, int b, float2* out, bool first, int real_only, cudaStream_t s, bool holo = false) {
    prof_begin(p, ST_INV_COLS, s);
    launch_inv_cols_from(p, b, holo, p->d_AB, s);
    prof_end(p, p->bins[b].n1 > p->bins[b].n0 ? 2 : 1, s);
    prof_begin(p, ST_INV_ROWS, s);
    launch_inv_rows(p, b, p->d_AB, out, first ? 0 : 1, real_only, s);
    prof_end(p, 1, s);
}

// Plans without stored G: the tiles of bins [b0, b1] into the tap scratch.  Their largest tap raises
// the plan's bound before the grid step of any of them, so a bin's fixed-point scale may be coarser
// than by itself by the ratio of its largest tap to the run's (2^-36 of the bound instead of 2^-37).
static void generate(rimo_plan* p, int b0, int b1, cudaStream_t s) {
    const int64_t v0 = p->bins[b0].vb, n = p->bins[b1].ve - v0;
    if (p->mode == RIMO_MODE_SURROGATE) {
        prof_begin(p, ST_MLP, s);
        prof_end(p, surrogate_generate(p, v0, n, s), s);
    } else if (p->mode == RIMO_MODE_ONTHEFLY || p->mode == RIMO_MODE_HOLOGRAPHIC) {
        prof_begin(p, ST_GBUILD, s);
        launch_gbuild_range(p, v0, n, s);  // exact tiles
        prof_end(p, 1, s);
    }
}

static void gtg(rimo_plan* p, int b, int mode, const float2* y_in, float2* y_out, cudaStream_t s) {
    generate(p, b, b, s);
    prof_begin(p, ST_GTG, s);
    launch_gtg(p, b, mode, y_in, y_out, s);
    const bool merge = mode != 0 && p->bins[b].m1 > p->bins[b].m0;
    prof_end(p, gtg_launches(p, b) + (merge ? 1 : 0), s);
}

// ---- the bins of a plan in groups
// A pass over one bin of a small image does not fill the GPU: its grid is nx ny / 4096 blocks,
// 304 of which are resident at once, and 4 bins of 256^2 took 27 launches of 4 to 10 us.  Plans
// of several bins, two of which have at most STAGE_BLOCKS blocks in a pass, therefore run as many
// bins at a time as have about that many, every pass one launch over a table of (bin) jobs with a
// grid, half transforms and patches of their own.  The kernels and the order of every sum are those
// of one bin at a time, so with stored G and with H the results are the same bit for bit; generated
// tiles share the bound of their run of bins (see generate), so that the fixed-point scale, hence
// the last bits, may depend on whether memory allowed a run.  The scratch of a group is at most
// STAGE_BYTES.  The line lies between 2048 x 1024 (512 blocks a bin; 20k visibilities, 6 bins,
// groups of three 0.656 ms, one by one 0.706; 5M, 8 bins 2.99 and 3.06) and 2048^2 (1024 blocks; 2k
// visibilities, 4 bins, two by two 0.677 and 0.677 ms for 512 MiB).
// Plans that generate their tiles do so for as many bins of a group as fit STAGE_TAPS (at
// 1024^2/1M/16 bins, generation and grid step of four bins instead of one at a time: tabulated
// kernels 0.82 -> 0.56 and 0.96 -> 0.87 ms per apply, the network 1.03 -> 0.80 ms).
// Measured, us per call, this change alone: Phi^dagger Phi and an update at 256^2/20k/4 bins 200 -> 100, Phi at
// 512x256/100k/3 bins 108 -> 60, Phi and Phi^dagger at 1024^2/2M/16 bins 1269 -> 1062 and
// 2010 -> 1854.
constexpr int STAGE_BLOCKS = 1216;                       // four waves of two blocks per SM
constexpr int64_t STAGE_BYTES = (int64_t)512 << 20;
constexpr int64_t STAGE_TAPS = (int64_t)1 << 30;

void PlanStage::drop_holographic() {
    for (Group& g : groups) {
        if (g.hfft) wide_fft_destroy(g.hfft);
        if (g.h) wide_h_destroy(g.h);
        g.hfft = nullptr;
        g.h = nullptr;
    }
    cudaFree(hpatch);
    hpatch = nullptr;
}

PlanStage::~PlanStage() {
    drop_holographic();
    for (Group& g : groups) {
        if (g.fft) wide_fft_destroy(g.fft);
        for (Run& r : g.runs) wide_gtg_destroy(r.gtg);
    }
    cudaFree(scratch);
}

static int64_t al256(int64_t x) { return (x + 255) & ~(int64_t)255; }
// scratch of one bin: half transforms, grid, patches
struct BinScratch {
    int64_t ab, gx, pt;
    explicit BinScratch(const rimo_plan* p)
        : ab(al256((int64_t)2 * p->nx * p->ny * 8)), gx(al256((int64_t)p->gx * p->gy * 8)),
          pt(al256((int64_t)std::max(1, p->max_tiles_bin) * p->PW * p->PW * 8)) {}
    int64_t total() const { return ab + gx + pt; }
};

void stage_bins(rimo_plan* p, bool share_taps) {
    int nb = 0;
    for (int b = 0; b < p->P; ++b) nb += p->bins[b].t1 > p->bins[b].t0;
    const int per_bin = std::max(1, p->nx * p->ny / 4096);
    const int64_t most =
        2 * per_bin > STAGE_BLOCKS ? 1 : std::min<int64_t>({(int64_t)nb, (STAGE_BLOCKS + per_bin - 1) / per_bin,
                                                            STAGE_BYTES / BinScratch(p).total()});
    // groups of nearly equal size
    const int64_t ng = most < 2 ? nb : (nb + most - 1) / most;
    p->stage_each = ng > 0 ? (int)((nb + ng - 1) / ng) : 1;
    // generated tiles: runs of a group's bins that share the tap scratch
    p->tap_run.assign((size_t)nb, 1);
    if (p->mode == RIMO_MODE_STORED_G) {
        for (int i = 0; i < nb; ++i) p->tap_run[i] = i % p->stage_each == 0;
    } else if (share_taps) {
        int64_t sum = 0;
        for (int i = 0; i < nb; ++i) {
            p->tap_run[i] = i % p->stage_each == 0 || sum + p->block_bytes[i] > STAGE_TAPS;
            sum = (p->tap_run[i] ? 0 : sum) + p->block_bytes[i];
        }
    }
}

// Scratch and tables of the plan's groups (an allocation that fails throws; what is made so far goes
// with `st`).
static void make_groups(rimo_plan* p, PlanStage* st, cudaStream_t s) {
    std::vector<int> bins;
    for (int b = 0; b < p->P; ++b)
        if (p->bins[b].t1 > p->bins[b].t0) bins.push_back(b);
    const BinScratch sc(p);
    const int64_t each = p->stage_each;
    RIMO_CUDA(device_malloc(&st->scratch, (size_t)(each * sc.total())));
    st->scratch_bytes = each * sc.total();
    char* base = static_cast<char*>(st->scratch);
    int runs = 0;
    for (size_t i = 0; i < bins.size(); i += (size_t)each) {
        PlanStage::Group g;
        for (size_t k = i; k < std::min(bins.size(), i + (size_t)each); ++k) {
            char* q = base + (int64_t)(k - i) * sc.total();
            g.jobs.push_back(WideJob{p, bins[k], 0, reinterpret_cast<float2*>(q), reinterpret_cast<float2*>(q + sc.ab),
                                     reinterpret_cast<float2*>(q + sc.ab + sc.gx)});
        }
        st->groups.push_back(g);
        PlanStage::Group& h = st->groups.back();
        h.fft = wide_fft_create(h.jobs, {nullptr}, {nullptr}, s);
        for (size_t k = 0; k < h.jobs.size(); ++k) {
            if (!p->tap_run[i + k]) continue;
            size_t e = k + 1;
            while (e < h.jobs.size() && !p->tap_run[i + e]) ++e;
            PlanStage::Run r{h.jobs[k].bin, h.jobs[e - 1].bin, nullptr};
            // (the counters are cleared at the start of every apply; there are at most P runs)
            r.gtg = wide_gtg_create(std::vector<WideJob>(h.jobs.begin() + (long)k, h.jobs.begin() + (long)e),
                                    p->d_counter + runs++, s);
            h.runs.push_back(r);
        }
    }
}

void stage_plan(rimo_plan* p, cudaStream_t s) {
    if (p->stage_each < 2) return;
    // only from memory that is plentiful: what a caller allocates next fits as it did without groups
    size_t room = 0, total = 0;
    RIMO_CUDA(cudaMemGetInfo(&room, &total));
    if (room < (size_t)(4 * p->stage_each * BinScratch(p).total())) return;
    auto st = std::make_unique<PlanStage>();
    try {
        make_groups(p, st.get(), s);
    } catch (const Error& e) {
        if (e.status == RIMO_ERR_CUDA) throw;
        return;  // no room for the scratch or the tables: one bin at a time, which needs neither
    }
    p->info.scratch_bytes += st->scratch_bytes;
    p->stage = st.release();  // freed with the plan
}

// `holo`: Phi^dagger Phi through H
static bool staged(const rimo_plan* p, bool holo) {
    return p->stage && !p->bin_by_bin && (!holo || p->stage->hpatch);
}

// One group: F Z_p x (mode 0 and 2), the grid step (`holo`: H), and the image (mode 1 and 2;
// `first`: written, else added to).
static void apply_group(rimo_plan* p, const PlanStage::Group& g, int mode, bool holo, const float2* x,
                        const float2* y_in, float2* y_out, float2* out, bool first, int real_only, cudaStream_t s) {
    const WideFft* fft = holo ? g.hfft : g.fft;
    if (mode != 1) {
        prof_begin(p, ST_FWD_ROWS, s);
        wide_fwd_rows(fft, x, s);
        prof_end(p, 1, s);
        prof_begin(p, ST_FWD_COLS, s);
        wide_fwd_cols(fft, s);
        prof_end(p, 1, s);
    }
    if (holo) {
        prof_begin(p, ST_HAPPLY, s);
        wide_happly(g.h, s);
        prof_end(p, 1, s);
    } else {
        for (const PlanStage::Run& r : g.runs) {
            // (its bins are neighbours but for empty ones: one range of visibilities)
            generate(p, r.bin0, r.bin1, s);
            prof_begin(p, ST_GTG, s);
            const int nl = wide_gtg(r.gtg, mode, y_in, y_out, s);
            prof_end(p, nl, s);
        }
    }
    if (mode == 0) return;
    prof_begin(p, ST_INV_COLS, s);
    wide_inv_cols(fft, s);
    prof_end(p, 2, s);
    prof_begin(p, ST_INV_ROWS, s);
    wide_inv_rows(fft, out, first ? 0 : 1, real_only, s);
    prof_end(p, 1, s);
}

static void begin_apply(rimo_plan* p, cudaStream_t s) {
    reset_schedulers(p, s);
    if (p->mode == RIMO_MODE_SURROGATE && !p->sur)
        fail(RIMO_ERR_STATE, "surrogate plan without a surrogate (rimo_plan_set_surrogate)");
    if (p->mode != RIMO_MODE_STORED_G) reset_surrogate_bounds(p, s);  // tap bounds of generated tiles
}

void apply_phi(rimo_plan* p, const float2* x, float2* y, cudaStream_t s) {
    begin_apply(p, s);
    if (staged(p, false)) {
        for (const auto& g : p->stage->groups) apply_group(p, g, 0, false, x, nullptr, y, nullptr, false, 0, s);
        return;
    }
    for (int b = 0; b < p->P; ++b) {
        if (bin_empty(p, b)) continue;
        fwd(p, b, x, s);
        gtg(p, b, 0, nullptr, y, s);
    }
}

void apply_phi_adj(rimo_plan* p, const float2* y, float2* x, cudaStream_t s) {
    bool first = true;
    begin_apply(p, s);
    prof_begin(p, ST_BOUND, s);
    launch_y_bound(p, y, s);
    prof_end(p, p->M > 0 ? 1 : 0, s);
    if (staged(p, false)) {
        for (const auto& g : p->stage->groups) {
            apply_group(p, g, 1, false, nullptr, y, nullptr, x, first, 0, s);
            first = false;
        }
        if (first) zero_image(p, (rimo_cfloat*)x, s);
        return;
    }
    for (int b = 0; b < p->P; ++b) {
        if (bin_empty(p, b)) continue;
        gtg(p, b, 1, y, nullptr, s);
        inv(p, b, x, first, 0, s);
        first = false;
    }
    if (first) zero_image(p, (rimo_cfloat*)x, s);
}

void apply_phi_adj_phi(rimo_plan* p, const float2* x, float2* out, int real_only, cudaStream_t s) {
    apply_phi_adj_phi_bins(p, x, out, real_only, nullptr, s);
}

void apply_phi_adj_phi_bins(rimo_plan* p, const float2* x, float2* out, int real_only, const uint8_t* mask,
                            cudaStream_t s) {
    bool first = true;
    begin_apply(p, s);
    prof_begin(p, ST_BOUND, s);
    launch_image_bound(p, x, s);
    prof_end(p, 1, s);
    if (!mask && staged(p, p->h_built)) {
        for (const auto& g : p->stage->groups) {
            apply_group(p, g, 2, p->h_built, x, nullptr, nullptr, out, first, real_only, s);
            first = false;
        }
        if (first) zero_image(p, (rimo_cfloat*)out, s);
        return;
    }
    for (int b = 0; b < p->P; ++b) {
        if (bin_empty(p, b) || (mask && !mask[b])) continue;
        fwd(p, b, x, s);
        if (p->h_built) {
            // H_p in place of G_p^dagger G_p (Section 3.3)
            prof_begin(p, ST_HAPPLY, s);
            launch_happly(p, b, s);
            prof_end(p, p->bins[b].n1 > p->bins[b].n0 ? 1 : 0, s);
        } else {
            gtg(p, b, 2, nullptr, nullptr, s);
        }
        inv(p, b, out, first, real_only, s, p->h_built);
        first = false;
    }
    if (first) zero_image(p, (rimo_cfloat*)out, s);
}

}  // namespace rimo

using namespace rimo;


extern "C" {

rimo_status rimo_apply_phi(rimo_plan_t p, const rimo_cfloat* x, rimo_cfloat* y, void* stream) {
    RIMO_API_BEGIN
    check_plan(p);
    if (!x || !y) fail(RIMO_ERR_INVALID_ARG, "null buffer");
    apply_phi(p, (const float2*)x, (float2*)y, (cudaStream_t)stream);
    RIMO_CUDA(cudaGetLastError());
    RIMO_API_END
}

rimo_status rimo_apply_phi_adj(rimo_plan_t p, const rimo_cfloat* y, rimo_cfloat* x, void* stream) {
    RIMO_API_BEGIN
    check_plan(p);
    if (!x || !y) fail(RIMO_ERR_INVALID_ARG, "null buffer");
    apply_phi_adj(p, (const float2*)y, (float2*)x, (cudaStream_t)stream);
    RIMO_CUDA(cudaGetLastError());
    RIMO_API_END
}

rimo_status rimo_apply_phi_adj_phi(rimo_plan_t p, const rimo_cfloat* x, rimo_cfloat* out,
                                   int32_t real_part_only, void* stream) {
    RIMO_API_BEGIN
    check_plan(p);
    if (!x || !out) fail(RIMO_ERR_INVALID_ARG, "null buffer");
    if ((const void*)x == (const void*)out) fail(RIMO_ERR_INVALID_ARG, "x and out must be distinct");
    apply_phi_adj_phi(p, (const float2*)x, (float2*)out, real_part_only, (cudaStream_t)stream);
    RIMO_CUDA(cudaGetLastError());
    RIMO_API_END
}

rimo_status rimo_apply_phi_adj_phi_bins(rimo_plan_t p, const rimo_cfloat* x, rimo_cfloat* out,
                                        int32_t real_part_only, const uint8_t* bin_mask, void* stream) {
    RIMO_API_BEGIN
    check_plan(p);
    if (!x || !out) fail(RIMO_ERR_INVALID_ARG, "null buffer");
    if ((const void*)x == (const void*)out) fail(RIMO_ERR_INVALID_ARG, "x and out must be distinct");
    apply_phi_adj_phi_bins(p, (const float2*)x, (float2*)out, real_part_only, bin_mask, (cudaStream_t)stream);
    RIMO_CUDA(cudaGetLastError());
    RIMO_API_END
}

rimo_status rimo_psf(rimo_plan_t p, rimo_cfloat* out, void* stream) {
    RIMO_API_BEGIN
    check_plan(p);
    if (!out) fail(RIMO_ERR_INVALID_ARG, "null buffer");
    apply_phi_adj_phi(p, p->d_delta, (float2*)out, 0, (cudaStream_t)stream);
    RIMO_CUDA(cudaGetLastError());
    RIMO_API_END
}

rimo_status rimo_profile_enable(rimo_plan_t p, int32_t on) {
    RIMO_API_BEGIN
    check_plan(p);
    p->prof_on = on != 0;
    RIMO_API_END
}

rimo_status rimo_profile_read(rimo_plan_t p, double* ms, int64_t* launches, int32_t n,
                              int32_t reset) {
    RIMO_API_BEGIN
    check_plan(p);
    if (n < 0 || n > RIMO_N_STAGES) fail(RIMO_ERR_INVALID_ARG, "n must be in [0, RIMO_N_STAGES]");
    prof_collect(p);
    for (int i = 0; i < n; ++i) {
        if (ms) ms[i] = p->prof_ms[i];
        if (launches) launches[i] = p->prof_launches[i];
    }
    if (reset)
        for (int i = 0; i < RIMO_N_STAGES; ++i) {
            p->prof_ms[i] = 0.0;
            p->prof_launches[i] = 0;
        }
    RIMO_API_END
}

rimo_status rimo_plan_get_zlayer(rimo_plan_t p, int32_t bin, rimo_cfloat* out, void* stream) {
    RIMO_API_BEGIN
    check_plan(p);
    if (!out) fail(RIMO_ERR_INVALID_ARG, "null buffer");
    if (bin < 0 || bin >= p->P) fail(RIMO_ERR_INVALID_ARG, "bin out of range");
    launch_zlayer(p, bin, (float2*)out, (cudaStream_t)stream);
    RIMO_CUDA(cudaGetLastError());
    RIMO_API_END
}

rimo_status rimo_plan_set_wait_test(rimo_plan_t p, int32_t stall, int32_t polls) {
    RIMO_API_BEGIN
    check_plan(p);
    if (stall != 0 && stall != 1) fail(RIMO_ERR_INVALID_ARG, "stall must be 0 or 1");
    if (stall && (polls < 1 || polls > (1 << 15))) fail(RIMO_ERR_INVALID_ARG, "polls must be in [1, 32768]");
    p->test_stall = stall;
    p->test_polls = stall ? (uint32_t)polls : 0u;
    RIMO_API_END
}

rimo_status rimo_plan_status(rimo_plan_t p, void* stream) {
    RIMO_API_BEGIN
    check_plan(p);
    cudaStream_t s = (cudaStream_t)stream;
    int32_t flag = 0;
    RIMO_CUDA(cudaMemcpyAsync(&flag, p->d_status, sizeof(flag), cudaMemcpyDeviceToHost, s));
    RIMO_CUDA(cudaStreamSynchronize(s));
    if (flag != 0) {
        RIMO_CUDA(cudaMemsetAsync(p->d_status, 0, sizeof(int32_t), s));
        RIMO_CUDA(cudaStreamSynchronize(s));
        if (flag == 3) fail(RIMO_ERR_INVALID_ARG, "non-finite input values (or a fixed-point bound overflowed)");
        fail(RIMO_ERR_TIMEOUT, "a bounded device wait ran out (code " + std::to_string(flag) + ")");
    }
    RIMO_API_END
}



}  // extern "C"
