"""cis_turn (csrc/phase.cuh), compiled for the host, against 64 bits over a turn."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2605_26347_gb300 import _build

SOURCE = """
#include "phase.cuh"
extern "C" void cis(const float* r, float* out, long n) {
    for (long i = 0; i < n; ++i) {
        const float2 v = rimo::cis_turn(r[i]);
        out[2 * i] = v.x;
        out[2 * i + 1] = v.y;
    }
}
"""


@pytest.fixture(scope="module")
def cis(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("phase")
    (d / "cis.cpp").write_text(SOURCE)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build.nvcc()))), "include")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", cuda, "-I", _build.CSRC,
                    str(d / "cis.cpp"), "-o", str(d / "cis.so")], check=True)
    lib = C.CDLL(str(d / "cis.so"))
    lib.cis.argtypes = [C.c_void_p, C.c_void_p, C.c_long]

    def run(r):
        r = np.ascontiguousarray(r, np.float32)
        out = np.empty((r.size, 2), np.float32)
        lib.cis(r.ctypes.data, out.ctypes.data, r.size)
        return out.astype(np.float64)
    return run


def test_within_one_ulp_of_64_bits(cis):
    """sincospif's bound is 1 ulp; the function that takes its place may not be further off."""
    rng = np.random.default_rng(1)
    r = np.concatenate([np.linspace(-0.5, 0.5, 2_000_001), rng.uniform(-0.5, 0.5, 500_000),
                        rng.uniform(-1, 1, 100_000) * 2.0 ** -rng.integers(2, 40, 100_000)]).astype(np.float32)
    a = 2 * np.pi * r.astype(np.float64)
    ref = np.stack([np.cos(a), np.sin(a)], 1)
    err = np.abs(cis(r) - ref)
    assert err.max() < 5.4e-8
    big = np.abs(ref) > 1e-9  # (at the zeros the angle itself is rounded: sin(pi) of 64 bits is not 0)
    ulp = np.spacing(np.abs(ref).astype(np.float32)).astype(np.float64)
    assert (err[big] / ulp[big]).max() < 1.0
    assert np.sqrt((err**2).mean()) < 1.53e-8


def test_quarter_turns_are_exact(cis):
    r = np.array([0.0, 0.25, 0.5, -0.25, -0.5, 0.125])
    assert np.array_equal(cis(r)[:5], [[1, 0], [0, 1], [-1, 0], [0, -1], [-1, 0]])
    assert np.abs(cis(r)[5] - np.sqrt(0.5)).max() < 3e-8
