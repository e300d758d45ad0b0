"""The grid step at the edges of its work units (GPU): units of fewer visibilities than a block
has warps, of one more, and around the 32 visibilities per warp that it holds metadata for;
every tile side; both uv-tile sizes; units split over several slices; against the FP64 oracle."""
import math

import numpy as np
import pytest

from parity_util import TOL, both, rel, to_dev, to_host

pytestmark = pytest.mark.gpu

# (visibilities, kb_support, max_wsupport, uv-tile, spread in grid cells)
CASES = [
    (1, 7, 9, 32, 4), (7, 7, 9, 32, 4), (8, 7, 9, 32, 4), (9, 7, 9, 32, 4), (13, 7, 9, 32, 4), (25, 7, 9, 32, 4),
    (256, 7, 9, 32, 6), (257, 7, 9, 32, 6), (385, 7, 9, 32, 6), (769, 7, 9, 32, 6),
    (300, 3, 1, 32, 40), (300, 5, 3, 32, 40), (300, 9, 1, 32, 40), (300, 11, 5, 32, 40),
    (300, 11, 7, 32, 40), (300, 11, 9, 32, 40), (300, 11, 9, 64, 60), (300, 7, 9, 64, 60), (1200, 7, 9, 64, 6),
]


@pytest.mark.parametrize("m, kb, cap, tile, spread", CASES)
def test_units_of_every_size_and_tile_side(m, kb, cap, tile, spread):
    n, fov = 64, math.radians(2.0)
    rng = np.random.default_rng(m * 31 + kb * 7 + cap)
    uvw = np.empty((m, 3))
    # a patch of `spread` cells that straddles the wrap of the grid in v
    uvw[:, 0] = (10.0 + spread * rng.random(m)) / (2.0 * fov)
    uvw[:, 1] = (spread * (rng.random(m) - 0.5)) / (2.0 * fov)
    uvw[:, 2] = 2000.0 * (rng.random(m) - 0.5)
    plan, op = both(uvw, n, n, fov, fov, n_wbins=1, kb_support=kb, max_wsupport=cap, tile_size=tile)
    x = (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))).astype(np.complex64)
    y = (rng.standard_normal(m) + 1j * rng.standard_normal(m)).astype(np.complex64)
    assert rel(to_host(plan.phi(to_dev(x))), op.phi(x)) < TOL
    assert rel(to_host(plan.phi_adj(to_dev(y))), op.phi_adj(y)) < TOL
    first = to_host(plan.phi_adj_phi(to_dev(x)))
    assert rel(first, op.phi_adj_phi(x)) < TOL
    assert np.array_equal(to_host(plan.phi_adj_phi(to_dev(x))), first)  # fixed-point sums: bit for bit
    plan.status()
    plan.close()


def row_passes(plan, call):
    """Launches of the forward row pass in a call: one per group of bins, or per bin."""
    plan.profile_read()
    plan.profile(True)
    call()
    plan.profile(False)
    return plan.profile_read()["fwd_rows"][1]


def test_no_groups_where_a_bins_passes_fill_the_gpu():
    """At 2048^2 two bins side by side are no faster than one after the other: no scratch for them."""
    import synth

    import paper_2605_26347_gb300 as pkg
    n, bins, fov = 2048, 4, math.radians(2.0)
    plan = pkg.Plan(synth.make_uvw(500, 60, 1.28e9, 11), pkg.default_params(n, n, fov, fov, n_wbins=bins))
    x = to_dev(np.ones((n, n)))
    assert row_passes(plan, lambda: plan.phi_adj_phi(x)) == bins
    # one bin's scratch: 2 n^2 half transforms, 4 n^2 grid, n^2 delta image, patches
    assert plan.info()["scratch_bytes"] < 8 * 8 * n * n
    plan.close()


@pytest.mark.parametrize("nx, ny, m, bins, kw", [
    (64, 64, 500, 2, {}), (64, 64, 40, 9, {}), (256, 64, 3000, 5, {}), (64, 256, 3000, 5, dict(tile_size=64)),
    (512, 512, 20000, 23, {}), (1024, 1024, 30000, 7, {}), (4096, 64, 3000, 3, {}), (64, 4096, 3000, 3, {}),
    (128, 128, 4000, 4, dict(mode=4, wkernel_table=64)), (128, 128, 4000, 4, dict(kb_support=11)),
    (2048, 1024, 3000, 3, {}),
])
def test_bins_in_groups_equal_one_bin_at_a_time(nx, ny, m, bins, kw):
    """Plans of small images run their bins in groups; a call that selects every bin by a mask
    takes them one at a time: the same sums in the same order, bit for bit with stored G.  With
    tiles generated per group the fixed-point scale comes from the group's tap bound, which may
    be a power of two above a bin's: 2^-36 of the bound instead of 2^-37 per contribution, far below
    an FP32 rounding."""
    import synth
    import torch

    import paper_2605_26347_gb300 as pkg
    side = max(nx, ny)
    fov_x, fov_y = math.radians(2.0) * nx / side, math.radians(2.0) * ny / side
    uvw = synth.make_uvw(m, 60, 1.28e9, 11)
    plan = pkg.Plan(uvw, pkg.default_params(nx, ny, fov_x, fov_y, n_wbins=bins, **kw))
    rng = np.random.default_rng(5)
    x = torch.from_numpy((rng.standard_normal((ny, nx)) + 1j * rng.standard_normal((ny, nx))).astype(np.complex64)).cuda()
    assert row_passes(plan, lambda: plan.phi_adj_phi(x)) < row_passes(
        plan, lambda: plan.phi_adj_phi_bins(x, np.ones(bins, np.uint8)))  # the plan has groups
    for real in (False, True):
        a = plan.phi_adj_phi(x, real_part_only=real)
        b = plan.phi_adj_phi_bins(x, np.ones(bins, np.uint8), real_part_only=real)
        if kw.get("mode") == 4:
            assert rel(to_host(a), to_host(b)) < 1e-7
        else:
            assert torch.equal(torch.view_as_real(a), torch.view_as_real(b))
    # Phi^dagger Phi x = Phi^dagger (Phi x), the two halves in groups as well
    c = plan.phi_adj(plan.phi(x))
    a = plan.phi_adj_phi(x)
    assert rel(to_host(c), to_host(a)) < 2e-6  # each within 1e-6 of 64 bits
    plan.status()
    plan.close()


@pytest.mark.parametrize("m, kb, cap, tile, dense", [
    (300, 7, 9, 32, False), (300, 7, 9, 64, False), (60000, 7, 9, 32, True), (60000, 7, 9, 64, True),
    (300, 3, 1, 32, False), (60000, 3, 1, 32, True), (60000, 5, 1, 32, True), (60000, 5, 3, 32, True),
    (60000, 9, 1, 32, True), (60000, 11, 1, 32, True), (60000, 11, 3, 32, True), (60000, 11, 7, 32, True),
    (60000, 11, 9, 32, True), (400, 11, 9, 64, False), (1, 7, 9, 32, False),
])
def test_holographic_apply_of_every_tile_side(m, kb, cap, tile, dense):
    """H against G^dagger G of the same plan, rows kept dense (a visibility or more per cell) and
    compressed, for every tile side; with bins in groups and one at a time."""
    import torch

    import paper_2605_26347_gb300 as pkg
    n, fov = 64, math.radians(2.0)
    rng = np.random.default_rng(m + kb + cap)
    uvw = (rng.random((m, 3)) - 0.5) * np.array([2 * n / (2 * fov), 2 * n / (2 * fov), 3000.0])
    bins = 1 if m < 2 else 2
    plan = pkg.Plan(uvw, pkg.default_params(n, n, fov, fov, n_wbins=bins, kb_support=kb, max_wsupport=cap,
                                            tile_size=tile))
    x = to_dev((rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))))
    g = to_host(plan.phi_adj_phi(x))
    plan.build_holographic()
    i = plan.info()
    if dense:
        assert i["h_nonzero"] > 0.8 * i["h_entries"]
    a = plan.phi_adj_phi(x)
    assert rel(to_host(a), g) < TOL  # both within a few 1e-7 of the operator
    b = plan.phi_adj_phi_bins(x, np.ones(bins, np.uint8))
    assert torch.equal(torch.view_as_real(a), torch.view_as_real(b))
    plan.status()
    plan.close()


@pytest.mark.parametrize("n, tile", [(64, 32), (64, 64), (128, 32), (256, 32), (256, 64), (512, 64), (1024, 32),
                                     (2048, 64)])
def test_needed_tiles_of_the_column_passes(n, tile):
    """Few visibilities, scattered over the whole grid and its edges: most tiles are not needed, so
    the column passes' marks (per warp, or in shared memory below 256) decide what is stored and read."""
    fov = math.radians(2.0)
    rng = np.random.default_rng(n + tile)
    m = 40
    uvw = np.empty((m, 3))
    uvw[:, :2] = (rng.random((m, 2)) - 0.5) * (2 * n - 1) / (2.0 * fov)
    uvw[:2, :2] = [[0.4999 * n / fov, 0.0], [0.0, -0.4999 * n / fov]]
    uvw[:, 2] = 100.0 * (rng.random(m) - 0.5)
    plan, op = both(uvw, n, n, fov, fov, n_wbins=2, tile_size=tile)
    x = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    assert rel(to_host(plan.phi(to_dev(x))), op.phi(x.astype(np.complex64).astype(np.complex128))) < TOL
    assert rel(to_host(plan.phi_adj_phi(to_dev(x))), op.phi_adj_phi(x.astype(np.complex64).astype(np.complex128))) < TOL
    plan.close()


@pytest.mark.parametrize("bins", [[1, 2], [16, 15], [16, 16], [16, 17], [32, 32, 1], [32, 32, 31, 4]])
def test_staged_batch_of_many_jobs(bins):
    """A block finds its (plan, bin) job 32 candidates at a time: job counts on both sides of 32 and
    beyond 64, against each plan's own apply bit for bit."""
    import synth
    import torch

    import paper_2605_26347_gb300 as pkg
    n, fov = 64, math.radians(2.0)
    chans = synth.wideband_channels(n_chan=len(bins), m_lo=2000, m_hi=3000, seed=43)
    plans = [pkg.Plan(uvw, pkg.default_params(n, n, fov, fov, n_wbins=b)) for (_, uvw), b in zip(chans, bins)]
    batch = pkg.Batch(plans, form=pkg.BATCH_STAGED)
    assert batch.layout()["jobs"] > 0.9 * sum(bins)
    rng = np.random.default_rng(sum(bins))
    x = torch.stack([to_dev(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))) for _ in bins])
    out = batch.phi_adj_phi(x)
    for k, p in enumerate(plans):
        assert torch.equal(torch.view_as_real(out[k].contiguous()),
                           torch.view_as_real(p.phi_adj_phi(x[k].contiguous())))


@pytest.mark.parametrize("kb, op", [(3, "phi_adj"), (3, "phi_adj_phi"), (7, "phi_adj_phi")])
def test_scaling_by_powers_of_two_is_exact_up_to_the_largest_numbers(kb, op):
    """The fixed-point scale of a unit is a power of two that follows its bound, so inputs times 2^k
    give outputs times 2^k bit for bit, also where the bound is within a doubling or two of the
    largest FP32 number."""
    import torch

    import paper_2605_26347_gb300 as pkg
    n, m, fov = 64, 4 if kb == 3 else 1, math.radians(2.0)  # (wider tiles of several visibilities sum up to overflow)
    rng = np.random.default_rng(kb)
    uvw = np.zeros((m, 3))
    uvw[:, :2] = (10.0 + 3.0 * rng.random((m, 2))) / (2.0 * fov)
    plan = pkg.Plan(uvw, pkg.default_params(n, n, fov, fov, n_wbins=1, kb_support=kb, max_wsupport=1))
    size = [np.abs(t.real) + np.abs(t.imag) for t in plan.tiles(np.arange(m))[3]]
    tmax, t1 = max(s.max() for s in size), max(s.sum() for s in size)
    if op == "phi_adj":
        v = (rng.standard_normal(m) + 1j * rng.standard_normal(m)) * np.array([1.0, 1e-2, 1e-4, 1e-6])
        bound = 2 * tmax * (np.abs(v.real) + np.abs(v.imag)).max()
    else:
        # a point source beside faint ones: |X| over the grid is that of the point source at the
        # image centre to a few per cent, |Re X| + |Im X| between it and sqrt(2) times it
        v = np.zeros((n, n), np.complex128)
        v[30:33, 20:28] = 1e-4 * rng.standard_normal((3, 8))
        v[n // 2, n // 2] = 1.0
        bound = 4 * tmax * t1 * float(to_host(plan.zlayer(0))[n // 2, n // 2].real) * math.sqrt(2.0)
    v = torch.view_as_real(to_dev(v * 1.6 / bound))
    apply = getattr(plan, op)

    def scaled(k):
        out = torch.view_as_real(apply(torch.view_as_complex(v * 2.0**k)))
        plan.status()
        assert torch.isfinite(out).all()
        return out.double() * 2.0**-k

    ref = scaled(0)
    for k in (-60, 20, 125, 126):  # the bound 1.1 to 1.6 times 2^k, 1.1 of it with the phases of X
        assert torch.equal(scaled(k), ref), k
    plan.close()


def test_plans_of_other_shapes_in_other_threads():
    """The grid step's kernel for run-time strides serves plans of 13 x 13 and of 19 x 19 tiles, whose
    blocks need different shared memory: launches from two threads do not disturb each other."""
    import threading

    import torch

    import paper_2605_26347_gb300 as pkg
    n, fov, m = 64, math.radians(2.0), 300
    rng = np.random.default_rng(2)
    uvw = (rng.random((m, 3)) - 0.5) * np.array([2 * n / (2 * fov), 2 * n / (2 * fov), 3000.0])
    x = to_dev(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    work = []
    for kb in (5, 11):
        plan = pkg.Plan(uvw, pkg.default_params(n, n, fov, fov, n_wbins=1, kb_support=kb))
        work.append((plan, torch.cuda.Stream(), plan.phi_adj_phi(x), torch.empty_like(x)))
    torch.cuda.synchronize()
    failed = []

    def run(plan, stream, ref, out):
        try:
            for _ in range(400):
                plan.phi_adj_phi(x, out=out, stream=stream)
            stream.synchronize()
            if not torch.equal(torch.view_as_real(out), torch.view_as_real(ref)):
                failed.append("result")
        except Exception as e:
            failed.append(e)

    threads = [threading.Thread(target=run, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    for plan, *_ in work:
        plan.status()
        plan.close()
