"""Thin gas: values below the normal range of FP32 keep what FP32's subnormals hold, and FP64 ones below theirs.

The rounding to FP32 (round_f32, integer operations) is compared bit for bit with numpy's conversion. A uniform gas off
equilibrium, scaled by a power of two, relaxes as the unscaled gas does: the scaling is exact except where a result
falls below 2^-126 and is rounded to the storage's fixed spacing q (2^-149 for FP32, 2^-133 for BF16) or, in FP32
arithmetic, to 2^-149. Tolerance: per stage a population collects at most half a q from the store and 16 units of 2^-149
from the equilibrium's coefficients (Nv + 1 of them, |w P_k| < 1), its sum, the combination and the sums of the moments;
a moment weighs the populations with at most max(pbar, pbar^2), and a stage does not amplify them (the rates stay below
1 per stage), so 3 (N + 1) W (q/2 + 16 x 2^-149) with W the sum of those weights
over the velocities (the last 3 for the state that the run starts from, rounded twice and multiplied by 1.5 between)."""
import ctypes
import os
import shutil
import subprocess
import tempfile

import numpy as np
import pytest

from paper_1608_03004_gb300 import binding as rb
from paper_1608_03004_gb300 import build as B

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def shim():
    out = os.path.join(tempfile.mkdtemp(prefix="rlb_sv_"), "libsv.so")
    subprocess.run([B.nvcc(), B.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-o", out,
                    os.path.join(HERE, "gpu_src", "small_values_check.cu")], check=True)
    lib = ctypes.CDLL(out)
    lib.sv_eval.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 3 + [ctypes.c_int]

    def run(which, a, b=None):
        a = np.ascontiguousarray(a, dtype=np.float64)
        b = np.zeros_like(a) if b is None else np.ascontiguousarray(b, dtype=np.float64)
        y = np.empty_like(a)
        assert lib.sv_eval(which, a.ctypes.data, b.ctypes.data, y.ctypes.data, a.size) == 0
        return y

    yield run
    shutil.rmtree(os.path.dirname(out), ignore_errors=True)


def test_rounding_to_fp32_is_numpys(shim):
    rng = np.random.default_rng(7)
    x = [rng.choice([-1.0, 1.0], 200000) * rng.uniform(1, 2, 200000) * 2.0 ** rng.integers(-155, 130, 200000)]
    for e in range(-152, 129):  # ties, their neighbours, carries into the next binade, the ends of the range
        m = np.array([1.0, 1.5, 2.0 - 2.0**-23, 2.0 - 2.0**-24, 2.0 - 2.0**-25, 1.0 + 2.0**-24, 1.0 + 3 * 2.0**-24])
        if e < -126:
            u = np.arange(1, 9) * 2.0 ** (-150 - e)
            m = np.concatenate([m, u])
        v = m * 2.0**e
        x += [v, -v, np.nextafter(v, np.inf), np.nextafter(v, 0)]
    x.append(np.array([0.0, -0.0, np.inf, -np.inf, 5e-324, -5e-324, 1e308, -1e308]))
    x = np.concatenate(x)
    with np.errstate(over="ignore", under="ignore"):
        ref = x.astype(np.float32)
    got = shim(0, x).astype(np.float32)
    np.testing.assert_array_equal(got.view(np.uint32), ref.view(np.uint32))
    assert np.isnan(shim(0, np.array([np.nan]))).all()


def relax(storage, Qp, scale, v=0.3, nsteps=3, tau=1.0):
    """Moments of a uniform periodic gas after some steps from a state off equilibrium, divided by the scale, and the
    tolerance of the scaled run."""
    Qxi, Nx = 8, 8
    t = rb.Tube(Qp, Qxi, Qp - 1, 5, Nx, 100.0, 0.5 * tau, tau, rb.BC_PERIODIC, storage)
    one = np.ones(Nx)
    with rb.rlb_init([t], scale * one, scale * one, v * one) as h:
        F = rb.rlb_get_state(h).reshape(Qp * Qxi, Nx)
        # off equilibrium by exact factors, so that the scaled and the unscaled populations agree
        F *= np.where(np.arange(Qp * Qxi) % 3 == 0, 1.5, 1.0)[:, None]
        rb.rlb_set_state(h, F.ravel())
        rb.rlb_step(h, nsteps)
        M = rb.rlb_moments(h)
    pb = rb.rlb_quadrature(Qp, Qxi)[0]
    W = Qxi * np.maximum(pb, pb * pb).sum()
    q = {rb.STORAGE_F32: 2.0**-149, rb.STORAGE_BF16: 2.0**-133}[storage]
    return M[:5, 0] / scale, 3 * (nsteps + 1) * W * (q / 2 + 16 * 2.0**-149) / scale


@pytest.mark.parametrize("storage,Qp,exp,v", [
    (rb.STORAGE_F32, 3, -116, 0.0), (rb.STORAGE_F32, 3, -116, 0.3), (rb.STORAGE_F32, 3, -120, 0.3),
    (rb.STORAGE_F32, 4, -120, 0.3), (rb.STORAGE_BF16, 4, -110, 0.0), (rb.STORAGE_BF16, 4, -110, 0.3),
    (rb.STORAGE_BF16, 4, -112, 0.0), (rb.STORAGE_BF16, 4, -112, 0.3)])
def test_thin_gas_relaxes_to_its_equilibrium(storage, Qp, exp, v):
    got, tol = relax(storage, Qp, 2.0**exp, v)
    ref, _ = relax(storage, Qp, 1.0, v)
    assert np.all(np.abs(got - ref) <= tol), (got, ref, tol)


def test_sum_of_a_double_float_keeps_subnormals(shim):
    """hi + lo, exact in FP64: within its last place for a normal high part, exact below 2^-126."""
    rng = np.random.default_rng(8)
    u = rng.integers(-(2**23), 2**23, 20000) * 2.0**-149  # subnormal, and zero
    hi = np.concatenate([u, [0.0, -0.0, 2.0**-149, -(2.0**-149), 2.0**-126 - 2.0**-149], 2.0**-126 * rng.uniform(1, 4, 5000)])
    hi = hi.astype(np.float32).astype(np.float64)
    lo = rng.integers(-4, 5, hi.size) * 2.0**-149
    np.testing.assert_allclose(shim(1, hi, lo), hi + lo, rtol=2.0**-52, atol=0)


@pytest.mark.parametrize("Qp,exp,v", [(3, -128, 0.0), (3, -128, 0.3), (3, -124, 0.02), (3, -120, 0.0), (4, -120, 0.0)])
def test_moments_below_the_normal_range(Qp, exp, v):
    """The moments that a step leaves for the next one (N^0 below 2^-126, or the N^x and T^0x of a slow gas)."""
    got, tol = relax(rb.STORAGE_F32, Qp, 2.0**exp, v)
    ref, _ = relax(rb.STORAGE_F32, Qp, 1.0, v)
    assert np.all(np.abs(got - ref) <= tol), (got, ref, tol)


def test_square_root_of_subnormals(shim):
    rng = np.random.default_rng(9)
    x = np.concatenate([rng.uniform(1, 2, 20000) * 2.0 ** rng.integers(-1074, -1000, 20000), [5e-324, 2.0**-1022]])
    assert np.max(np.abs(shim(2, x) / np.sqrt(x) - 1.0)) <= 2 * 2.0**-52


@pytest.mark.parametrize("v", [0.3, -0.9])
def test_moving_fp64_gas_whose_squared_moments_are_subnormal(v):
    """(T^00 + T^xx)^2 - 4 (T^0x)^2 near 2^-1026 is held to 2^-1075: about 2^-48 relative, a half of it in e, and 9
    stages of it with gamma^2 = 5.3 at most stay below 1e-12."""
    Qxi, Nx = 8, 8
    t = rb.Tube(3, Qxi, 2, 5, Nx, 100.0, 0.1, 1.0, rb.BC_PERIODIC, rb.STORAGE_F64)
    out = []
    for s in (1.0, 2.0**-515):
        with rb.rlb_init([t], np.full(Nx, s), np.full(Nx, s), np.full(Nx, v)) as h:
            rb.rlb_step(h, 3)
            out.append(rb.rlb_get_state(h) / s)
    assert np.max(np.abs(out[1] - out[0])) <= 1e-12 * np.max(np.abs(out[0]))
