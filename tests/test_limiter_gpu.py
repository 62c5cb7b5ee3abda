"""The FP64 kernels' limiter code on the GPU where its two users differ from one interface at a time: the packed
double-float limiter with different stencils in its two halves (one of them with indicator ratios beyond 1e19, where the
quotient's denominator underflows and the smoothest stencil's value is taken), and the adjoint's gradient of the interface
value against the complex step of the textbook formula in extended precision.

Tolerances: each half of a packed operation is rounded on its own, so a pair of interfaces gives the bits of each alone.
The gradient: every indicator's quadratic form has a condition number below 60 (4x^2 - 11xy + 10y^2 and its mirror image
are definite with eigenvalues 0.74 and 13.3; absolute terms against the form: (13.3 + 11/2)/0.74 < 26), so v_k is good to
60 x 4 x 2^-53, the weights and z_k to three of these; each partial then carries 1e-13 of the sum of its terms' magnitudes."""
import ctypes
import os
import shutil
import subprocess
import tempfile

import numpy as np
import pytest

import oracle
from paper_1608_03004_gb300 import build as B

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
EPS = 1e-6


@pytest.fixture(scope="module")
def shim():
    out = os.path.join(tempfile.mkdtemp(prefix="rlb_lm_"), "liblm.so")
    subprocess.run([B.nvcc(), B.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-o", out,
                    os.path.join(HERE, "gpu_src", "limiter_check.cu")], check=True)
    lib = ctypes.CDLL(out)
    lib.lm_eval.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 3 + [ctypes.c_int]

    def run(which, v, w):
        v, w = (np.ascontiguousarray(a, dtype=np.float64) for a in (v, w))
        y = np.empty((len(v), 2 if which == 0 else 5))
        assert lib.lm_eval(which, v.ctypes.data, w.ctypes.data, y.ctypes.data, len(v)) == 0
        return y

    yield run
    shutil.rmtree(os.path.dirname(out), ignore_errors=True)


def samples(rng, n):
    """Rough, smooth, stepped and nearly constant stencils."""
    rough = rng.normal(size=(n, 5)) * 10.0 ** rng.uniform(-4, 1, (n, 1))
    smooth = 1 + 1e-3 * np.cumsum(rng.normal(size=(n, 5)), axis=1)
    step = np.where(np.arange(5) >= rng.integers(1, 5, size=(n, 1)), 1.0, 0.1) + 1e-6 * rng.normal(size=(n, 5))
    flat = 1 + 1e-9 * rng.normal(size=(n, 5))
    return np.concatenate([rough, smooth, step, flat])


def test_halves_of_the_packed_limiter_are_independent(shim):
    rng = np.random.default_rng(21)
    v = samples(rng, 4000)
    # jumps so high against the epsilon term that two of the three weights vanish in FP32's range
    far = np.where(np.arange(5) >= rng.integers(1, 5, size=(4000, 1)), 10.0 ** rng.uniform(8, 12, (4000, 1)), 0.0)
    v = np.concatenate([v, far])
    w = v[rng.permutation(len(v))]
    got = shim(0, v, w)
    np.testing.assert_array_equal(got[:, 0], shim(0, v, v)[:, 0])
    np.testing.assert_array_equal(got[:, 1], shim(0, w, w)[:, 1])
    np.testing.assert_array_equal(shim(0, v, v)[:, 0], shim(0, v, v)[:, 1])


def textbook(v):
    """Jiang and Shu's interface value between the third and the fourth sample, and what each partial is a sum of."""
    q = [(2 * v[0] - 7 * v[1] + 11 * v[2]) / 6, (-v[1] + 5 * v[2] + 2 * v[3]) / 6, (2 * v[2] + 5 * v[3] - v[4]) / 6]
    b = [np.longdouble(13) / 12 * (v[0] - 2 * v[1] + v[2]) ** 2 + (v[0] - 4 * v[1] + 3 * v[2]) ** 2 / 4,
         np.longdouble(13) / 12 * (v[1] - 2 * v[2] + v[3]) ** 2 + (v[1] - v[3]) ** 2 / 4,
         np.longdouble(13) / 12 * (v[2] - 2 * v[3] + v[4]) ** 2 + (3 * v[2] - 4 * v[3] + v[4]) ** 2 / 4]
    a = [d / (np.longdouble(EPS) + x) ** 2 for d, x in zip((np.longdouble(1) / 10, np.longdouble(6) / 10, np.longdouble(3) / 10), b)]
    s = a[0] + a[1] + a[2]
    return sum(x * y for x, y in zip(a, q)) / s, [x / s for x in a], q, b


def test_gradient_of_the_interface_value(shim):
    rng = np.random.default_rng(22)
    v = samples(rng, 2000)
    got = shim(1, v, v)
    x = v.T.astype(np.clongdouble)
    h = np.longdouble(1e-30)
    Phi, w, q, b = textbook(v.T.astype(np.longdouble))
    # magnitude of the terms: the candidates' coefficients (below 2) and 2 w_k |q_k - Phi| / (eps + b_k) |db_k/dv|, where
    # |db_k/dv| <= 8 sqrt(b_k) (13/6 |second difference| x 2 + 1/2 |first| x 4, each bounded through b_k)
    size = 2 + sum(2 * wk * abs(qk - Phi) / (EPS + bk) * 8 * np.sqrt(bk) for wk, qk, bk in zip(w, q, b))
    for m in range(5):
        y = x.copy()
        y[m] += 1j * h
        ref = (textbook(y)[0].imag / h).astype(np.float64)
        err = np.abs(got[:, m] - ref) / size.astype(np.float64)
        assert err.max() <= 1e-13, (m, err.max())


def test_packed_limiter_matches_the_oracle_in_both_halves(shim):
    """As the bound of the limiter at one interface (6e-14 of the samples' scale), here for two different ones at once."""
    rng = np.random.default_rng(23)
    v = samples(rng, 1500)
    w = v[rng.permutation(len(v))]
    got = shim(0, v, w)
    for s, g in ((v, got[:, 0]), (w, got[:, 1])):
        ref = np.array([oracle.weno5(*row) for row in s])
        assert np.max(np.abs(g - ref) / np.max(np.abs(s), axis=1)) <= 6e-14
