"""Scalar device helpers of the stage kernels (csrc/rlb_device_math.cuh) on the GPU: a double-float joined to one double
by integer operations, the refined reciprocal square root, square root and quotient, and the split of values beyond
FP32's range.

Tolerances: df_join rounds lo once to the double's last place (half a unit) after the exact placement of hi, so it is
within one unit of hi + lo; the Newton steps leave a few roundings of FP64 (the correction steps of sqrt and the
quotient one), held to 4 and 2 units."""
import ctypes
import os
import shutil
import subprocess
import tempfile

import numpy as np
import pytest

from paper_1608_03004_gb300 import build as B

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
ULP = 2.0**-52


@pytest.fixture(scope="module")
def shim():
    out = os.path.join(tempfile.mkdtemp(prefix="rlb_ds_"), "libds.so")
    subprocess.run([B.nvcc(), B.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-o", out,
                    os.path.join(HERE, "gpu_src", "device_scalar_check.cu")], check=True)
    lib = ctypes.CDLL(out)
    lib.ds_eval.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 3 + [ctypes.c_int]

    def run(which, a, b=None):
        a = np.ascontiguousarray(a, dtype=np.float64)
        b = np.zeros_like(a) if b is None else np.ascontiguousarray(b, dtype=np.float64)
        y = np.empty_like(a)
        assert lib.ds_eval(which, a.ctypes.data, b.ctypes.data, y.ctypes.data, a.size) == 0
        return y

    yield run
    shutil.rmtree(os.path.dirname(out), ignore_errors=True)


def test_join_of_normalised_pairs(shim):
    rng = np.random.default_rng(3)
    v = np.concatenate([rng.normal(size=200000) * 10.0 ** rng.uniform(-18, 18, 200000),
                        # around powers of two, where hi and the sum lie in different binades
                        *[s * 2.0**k * (1.0 + d * 2.0**-e) for k in (-60, -20, -1, 0, 1, 40) for s in (1.0, -1.0)
                          for e in (25, 26, 30, 47, 52) for d in (np.array([-1.0]), np.array([0.0]), np.array([1.0]))]])
    hi = v.astype(np.float32)
    lo = (v - hi.astype(np.float64)).astype(np.float32)
    ref = hi.astype(np.float64) + lo.astype(np.float64)
    got = shim(0, hi, lo)
    assert np.all(np.abs(got - ref) <= ULP * np.abs(ref)), np.max(np.abs(got - ref) / np.abs(ref)) / ULP
    # lo at exactly half a unit of hi, both signs
    h = np.array([1.0, 1.5, 2.0, -1.0, -1.5, -4.0])
    half = np.spacing(np.abs(h).astype(np.float32)).astype(np.float64) / 2
    for s, f in ((1.0, 1.0), (-1.0, 0.5)):  # half a unit below a power of two is a quarter of the unit above it
        l = s * np.sign(h) * half * f
        np.testing.assert_array_equal(shim(0, h, l), h + l)


def test_join_of_special_values(shim):
    h = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 2.0**-100, -(2.0**-126), 2.0**-149])
    got = shim(0, h, np.zeros_like(h))
    assert got[0] == 0.0 and got[1] == 0.0 and got[2] == np.inf and got[3] == -np.inf and np.isnan(got[4])
    assert got[5] == h[5] and got[6] == h[6] and got[7] == 0.0


def test_roots_and_quotient(shim):
    rng = np.random.default_rng(4)
    x = np.exp(rng.uniform(-150, 150, 1 << 18))
    y = np.exp(rng.uniform(-60, 60, x.size)) * rng.choice([-1.0, 1.0], x.size)
    assert np.max(np.abs(shim(1, x) * np.sqrt(x) - 1.0)) <= 4 * ULP
    assert np.max(np.abs(shim(2, x) / np.sqrt(x) - 1.0)) <= 2 * ULP
    assert np.max(np.abs(shim(3, y, x) / (y / x) - 1.0)) <= 2 * ULP
    assert shim(2, np.zeros(4)).max() == 0.0 and np.isnan(shim(2, -np.ones(4))).all()


def test_split_beyond_the_fp32_range(shim):
    v = np.array([2.0**128, -(2.0**200), np.inf, -np.inf, np.nan, 2.0**-127, 2.0**-126])
    got = shim(4, v)
    assert got[0] == np.inf and got[1] == -np.inf and got[2] == np.inf and got[3] == -np.inf and np.isnan(got[4])
    assert got[5] == 0.0 and got[6] == v[6]
