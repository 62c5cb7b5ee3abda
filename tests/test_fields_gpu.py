"""Fields (rlb_moments) of states with special values, and at the edges of the kernel's tiles and mirror pairs, for every
storage type: NaN and infinite populations are reported as non-physical; subnormal FP32 populations are summed, not
dropped; the five moments match the quadrature sums of the stored state (numpy, extended precision) to the rounding of at
most 264 FP64 additions of positive terms, 264 x 2^-53 x 4 < 2e-13."""
import math

import numpy as np
import pytest

from paper_1608_03004_gb300 import binding as rb

pytestmark = pytest.mark.gpu
STORAGES = [rb.STORAGE_F64, rb.STORAGE_F32, rb.STORAGE_BF16]


def handle(storage, Nx=130, Qxi=9, Qp=3, tau=math.inf, scale=1.0):
    x = (np.arange(Nx) + 0.5) / Nx * 2 * np.pi
    t = rb.Tube(Qp, Qxi, Qp - 1, 5, Nx, 1.0 / Nx, 1e-4, tau, rb.BC_OPEN, storage)
    return rb.rlb_init([t], scale * (1 + 0.3 * np.sin(x)), scale * (1 + 0.2 * np.cos(x)), 0.4 * np.sin(x + 1))


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("tau", [math.inf, 0.05])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_special_values_are_reported(storage, tau, bad):
    with handle(storage, tau=tau) as h:
        F = rb.rlb_get_state(h)
        F[7 * 130 + 61] = bad
        with pytest.raises(rb.RlbError) as e:
            rb.rlb_set_state(h, F)
            rb.rlb_moments(h)
        assert e.value.status == rb.ENONPHYS


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("Nx,Qxi,Qp", [(1, 4, 3), (59, 5, 4), (60, 8, 3), (61, 66, 4), (121, 7, 3)])
@pytest.mark.parametrize("scale", [1.0, 1e-36])
def test_moments_are_the_sums_of_the_state(storage, Nx, Qxi, Qp, scale):
    if scale != 1.0 and storage == rb.STORAGE_F64:
        pytest.skip("FP64 has no subnormal populations at this scale")
    pb, _, xi, _ = (a.astype(np.longdouble) for a in rb.rlb_quadrature(Qp, Qxi))
    with handle(storage, Nx, Qxi, Qp, scale=scale) as h:
        F = rb.rlb_get_state(h).reshape(Qp, Qxi, Nx).astype(np.longdouble)
        got = rb.rlb_moments(h)[:5]
    a, b = np.einsum("ijx,i->jx", F, pb), np.einsum("ijx,i->jx", F, pb * pb)
    aa, bb = np.einsum("ijx,i->jx", abs(F), pb), np.einsum("ijx,i->jx", abs(F), pb * pb)
    ref = [a.sum(0), xi @ a, b.sum(0), xi @ b, (xi * xi) @ b]
    for k in range(5):
        size = aa.sum(0) if k < 2 else bb.sum(0)
        assert np.all(abs(got[k] - ref[k]) <= 2e-13 * size), k
