"""The FP64 stage kernel's own equilibrium at speed: a uniform gas in equilibrium does not change in a step, whichever basis the
kernel evaluates F^eq in (the default orders a polynomial in xi, the generic ones Legendre polynomials, rlb_init always
the latter), from rest to the documented speed limit in both directions.

Tolerance, normwise per cell, for one step at dt gamma (1 + |v|) / tau = 0.25. The Landau frame loses digits near the speed of
light: (T^00 + T^xx)^2 - 4 (T^0x)^2 = (4P)^2 is left of terms of 16 gamma^4 P^2, so a unit 2^-53 in the moments, of which
their sums leave up to 8, becomes up to 8 gamma^4 in e, and F^eq takes it in powers up to the fourth: 256 gamma^4 2^-53; the
coefficients add at most 34 x 2^-52."""
import numpy as np
import pytest

from paper_1608_03004_gb300 import binding as rb

pytestmark = pytest.mark.gpu

SPEEDS = [0.0, 1e-300, 1e-9, 0.02, 0.3, 0.58, 0.7, 0.85, 0.9, 0.95, 0.97, 0.99, 0.9949]


@pytest.mark.parametrize("Qp,Qxi,Np,Nv", [(3, 8, 2, 5), (4, 9, 2, 5), (4, 7, 3, 8), (3, 6, 2, 8)])
def test_uniform_equilibrium_stays(Qp, Qxi, Np, Nv):
    v = np.array([s * b for b in SPEEDS for s in (1.0, -1.0)])
    g = 1 / np.sqrt(1 - v**2)
    Nx, dt = 4, 1e-3
    rng = np.random.default_rng(31)
    P, n = rng.uniform(0.1, 2.0, v.size), rng.uniform(0.1, 2.0, v.size)
    tubes = [rb.Tube(Qp, Qxi, Np, Nv, Nx, 1.0, dt, dt * k * (1 + abs(b)) / 0.25, rb.BC_PERIODIC, rb.STORAGE_F64)
             for b, k in zip(v, g)]
    with rb.rlb_init(tubes, np.repeat(P, Nx), np.repeat(n, Nx), np.repeat(v, Nx)) as h:
        F0 = rb.rlb_get_state(h).reshape(v.size, Qp * Qxi, Nx)
        rb.rlb_step(h, 1)
        F1 = rb.rlb_get_state(h).reshape(F0.shape)
    err = np.max(np.abs(F1 - F0), axis=(1, 2)) / np.max(np.abs(F0), axis=(1, 2))
    assert np.all(err <= 2.0**-53 * (256 * g**4 + 68)), (v, err / 2.0**-53 / g**4)
