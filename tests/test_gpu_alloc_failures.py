"""Device allocations that fail (rimo_set_alloc_test makes them, on the host): what was there
before stays usable, and what needs no more memory goes on without it."""
import ctypes as C
import math

import numpy as np
import pytest

from oracle import mlp as omlp
from parity_util import to_dev, to_host
from test_gpu_surrogate import batch, rel

OOM = 2


def fail_alloc(n):
    """The nth device allocation from now on fails; returns what was left of the last count."""
    import paper_2605_26347_gb300 as pkg
    left = C.c_int64()
    pkg._lib.check(pkg._lib.load().rimo_set_alloc_test(n, C.byref(left)))
    return left.value


def test_the_count_is_set_read_and_ended(rimo_lib):
    import paper_2605_26347_gb300 as pkg
    assert fail_alloc(3) == 0
    assert fail_alloc(0) == 3
    assert fail_alloc(0) == 0
    with pytest.raises(pkg.RimoError) as e:
        fail_alloc(-1)
    assert e.value.status == 1


@pytest.mark.gpu
def test_a_batch_that_does_not_fit_leaves_the_surrogate_as_it_was():
    import paper_2605_26347_gb300 as pkg
    s = pkg.Surrogate(seed=0)
    p = {k: v.astype(np.float64) for k, v in pkg.unpack_params(s.get_params()).items()}
    s.gradients(*batch(256, 1))
    for call in (s.gradients, lambda x, t: s.forward(x)):
        fail_alloc(1)
        with pytest.raises(pkg.RimoError) as e:
            call(*batch(4096, 2))
        assert e.value.status == OOM and fail_alloc(0) == 0
    # larger than the buffers that are there, smaller than the batch that failed
    for B in (1408, 256, 4096):
        x, t = batch(B, B)
        ref_loss, ref = omlp.loss_and_grads(p, x.astype(np.float64), t.astype(np.float64), bf=True)
        loss, g = s.gradients(x, t)
        assert abs(loss - ref_loss) < 1e-4 * ref_loss
        gd = pkg.unpack_params(g)
        for k in ("W3", "b3", "W2", "b2", "W1", "b1"):
            assert rel(gd[k], ref[k]) < 2e-3, (B, k)  # bf16 flips, as in test_gpu_surrogate


@pytest.mark.gpu
def test_a_larger_batch_gives_back_the_smaller_ones_memory():
    import torch

    import paper_2605_26347_gb300 as pkg
    s = pkg.Surrogate(seed=0)
    x = torch.zeros((65536, 3), device="cuda")
    y = torch.empty((65536, 450), device="cuda")

    def free(B):  # MiB left on the device after a batch of B
        pkg._lib.check(s._lib.rimo_surrogate_forward(s._h, x.data_ptr(), B, y.data_ptr(), 0))
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0] / 2**20

    start = free(128)  # (kernels loaded)
    per = 6976 / 2**20  # bytes of a sample's activations
    half, full = start - free(32768), start - free(65536)
    assert abs(half - 32768 * per) < 16
    assert abs(full - 65536 * per) < 16, (half, full)


def applies(plan, x, y):
    """Phi x, Phi^dagger y and Phi^dagger Phi x, and the launches of forward row passes of the last:
    one per group of bins, or per bin."""
    out = [to_host(plan.phi(x)), to_host(plan.phi_adj(y))]
    plan.profile_read()
    plan.profile(True)
    out.append(to_host(plan.phi_adj_phi(x)))
    plan.profile(False)
    launches = plan.profile_read()["fwd_rows"][1]
    plan.status()
    return out, launches


def small_plan(bins=3, n=64, m=500, **kw):
    import synth

    import paper_2605_26347_gb300 as pkg
    fov = math.radians(2.0)
    return pkg.Plan(synth.make_uvw(m, 60, 1.28e9, 11), pkg.default_params(n, n, fov, fov, n_wbins=bins, **kw))


@pytest.mark.gpu
@pytest.mark.parametrize("kw, optional", [
    ({}, 3),                                # the groups' scratch, transform tables, unit list
    (dict(mode=4, wkernel_table=64), 4),    # and the taps of several bins at a time
])
def test_plan_creation_goes_on_without_groups(kw, optional):
    """Whichever allocation of plan creation fails: either creation reports it, or the plan takes
    one bin at a time, with the results of the bins in a group bit for bit (generated tiles: to the
    scale of the fixed-point sums, 2^-36 of their bound)."""
    bins = 3
    rng = np.random.default_rng(3)
    x = to_dev(rng.standard_normal((64, 64)) + 1j * rng.standard_normal((64, 64)))
    y = to_dev(rng.standard_normal(500) + 1j * rng.standard_normal(500))
    plan = small_plan(bins, **kw)
    ref, launches = applies(plan, x, y)
    assert launches == 1  # one group
    plan.close()
    survived = 0
    for nth in range(1, 200):
        fail_alloc(nth)
        try:
            plan = small_plan(bins, **kw)
        except Exception as e:
            assert getattr(e, "status", None) == OOM and fail_alloc(0) == 0
            continue
        if fail_alloc(0) != 0:  # more than creation makes
            plan.close()
            break
        survived += 1
        got, launches = applies(plan, x, y)
        for a, b in zip(got, ref):
            assert rel(a, b) < 1e-7 if kw else np.array_equal(a, b)
        if not kw:
            assert launches == bins
        plan.close()
    assert nth > 10 and survived == optional


@pytest.mark.gpu
def test_the_holographic_build_goes_on_without_groups():
    """Whichever allocation of the build of H fails: either it reports it and a second build
    succeeds, or H is there and applied one bin at a time, bit for bit as in groups."""
    bins = 3
    rng = np.random.default_rng(4)
    x = to_dev(rng.standard_normal((64, 64)) + 1j * rng.standard_normal((64, 64)))

    def normal(plan):
        plan.profile_read()
        plan.profile(True)
        out = to_host(plan.phi_adj_phi(x))
        plan.profile(False)
        return out, plan.profile_read()["h_apply"][1]

    plan = small_plan(bins)
    plan.build_holographic()
    ref, launches = normal(plan)
    assert launches == 1  # one group
    plan.close()
    survived = 0
    for nth in range(1, 200):
        plan = small_plan(bins)
        fail_alloc(nth)
        try:
            plan.build_holographic()
        except Exception as e:
            assert getattr(e, "status", None) == OOM and fail_alloc(0) == 0
            left = 0
            plan.build_holographic()
            got, launches = normal(plan)
            assert launches == 1
        else:
            left = fail_alloc(0)
            got, launches = normal(plan)
            if left == 0:
                survived += 1
                assert launches == bins
        assert np.array_equal(got, ref)
        h_bytes = plan.info()["h_bytes"]
        plan.build_holographic()  # built already: nothing to do
        assert plan.info()["h_bytes"] == h_bytes > 0
        plan.close()
        if left > 0:  # more than the build makes
            break
    assert survived == 4  # the groups' patches, transform tables, and the apply's jobs and their first blocks
