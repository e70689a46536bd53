"""Device helpers whose accuracy other tests only see through whole time steps, each against plain
arithmetic: the reciprocal of the FP64 collision, scaling by powers of two through the exponent, the
widening of floats by their bits; and the launch helper's error handling."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_1710_10569_gb300 import build as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def helpers(tmp_path_factory):
    import os
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    out = str(tmp_path_factory.mktemp("helpers") / "helpers.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "device_helpers.cu")
    r = subprocess.run([B.nvcc(), "-shared", "-cudart", "static", src, "-o", out] + B._flags(), capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(out)


def doubles(helpers, x):
    x = np.ascontiguousarray(x, dtype=np.float64)
    out = np.empty((4, x.size))
    assert helpers.helpers_doubles(x.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p), x.size) == 0
    return out


def samples():
    rng = np.random.default_rng(0)
    m = np.concatenate([1.0 + rng.random(200000), 2.0 - 2.0 ** -rng.uniform(1, 52, 20000), 1.0 + 2.0 ** -rng.uniform(1, 52, 20000)])
    rho = rng.uniform(0.5, 2.0, 200000)
    wide = np.ldexp(m, rng.integers(-1000, 1000, m.size)) * rng.choice([-1.0, 1.0], m.size)
    return np.concatenate([m, rho, wide])


def test_reciprocal_within_one_unit_of_the_last_place(helpers):
    """rcp.approx.ftz.f64 is right to about 2^-20, and one step of the third order leaves the cube of its
    error: half a unit of the last place for the rounding and a small part of one, so within one."""
    x = samples()
    got = doubles(helpers, x)[0]
    assert np.max(np.abs(got.view(np.int64) - (1.0 / x).view(np.int64))) <= 1


def test_scaling_by_the_exponent(helpers):
    tiny = np.finfo(np.float64).tiny
    x = np.concatenate([samples(), [0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -1e-310, tiny, 2 * tiny, -4 * tiny, 8 * tiny,
                                    np.ldexp(1.0, 1022), -np.ldexp(1.5, 1023)]])
    _, half, quarter, twice = doubles(helpers, x)
    for n, got in ((1, half), (2, quarter)):
        exp = x * 2.0 ** -n
        exp = np.where(np.abs(exp) < tiny, np.copysign(0.0, x), exp)  # below the normal numbers: a signed zero
        assert np.array_equal(got.view(np.int64)[~np.isnan(x)], exp.view(np.int64)[~np.isnan(x)]) and np.isnan(got[np.isnan(x)]).all()
    exp = np.where(np.abs(x) < tiny, np.copysign(0.0, x), np.where(np.abs(x) >= np.ldexp(1.0, 1023), x, 2.0 * x))
    assert np.array_equal(twice.view(np.int64)[~np.isnan(x)], exp.view(np.int64)[~np.isnan(x)]) and np.isnan(twice[np.isnan(x)]).all()


def test_floats_widened_by_their_bits(helpers):
    rng = np.random.default_rng(1)
    bits = np.concatenate([rng.integers(0, 2 ** 32, 500000, dtype=np.uint64).astype(np.uint32), np.arange(0, 1000, dtype=np.uint32),
                           np.array([0x80000000, 0x7f800000, 0xff800000, 0x7fc00000, 0x00800000, 0x007fffff, 0x807fffff], dtype=np.uint32)])
    x = bits.view(np.float32)
    out = np.empty(x.size)
    assert helpers.helpers_floats(x.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p), x.size) == 0
    exp = x.astype(np.float64)
    num = ~np.isnan(x)
    assert np.array_equal(out.view(np.int64)[num], exp.view(np.int64)[num]) and np.isnan(out[~num]).all()


def test_refused_launch_leaves_no_error_behind(helpers):
    """A launch that the runtime refuses is reported by the call that made it, and not again by the next."""
    refused, left = ctypes.c_int(), ctypes.c_int()
    helpers.helpers_refused_launch(ctypes.byref(refused), ctypes.byref(left))
    assert refused.value != 0 and left.value == 0
