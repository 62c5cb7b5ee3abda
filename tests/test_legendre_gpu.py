"""The Legendre coefficients of (1 - beta xi)^-m on the GPU (backward recurrence in the order, raising in m) against
the oracle's term-by-term series, through the equilibrium that rlb_init writes: speeds from rest to the documented
limit, both signs, for the default orders and for the generic kernel path.

Tolerance, normwise per cell: each coefficient carries a few units of FP64 rounding, and its relative error grows with
the conditioning of 1 - beta^2 (gamma^2 units at most); the three or four terms of the radial sum alternate in sign
with an amplification below 10. 2^-52 x 10 x (8 + gamma^2) x 4 stays below 1e-13 gamma^2 + 1e-13."""
import numpy as np
import pytest

import oracle
from paper_1608_03004_gb300 import binding as rb

pytestmark = pytest.mark.gpu

SPEEDS = [0.0, 1e-300, 1e-12, 1e-5, 0.02, 0.11, 0.3, 0.45, 0.58, 0.7, 0.85, 0.9, 0.95, 0.97, 0.99, 0.9949]


@pytest.mark.parametrize("Qp,Qxi,Np,Nv", [(3, 8, 2, 5), (4, 9, 2, 5), (4, 7, 3, 8), (3, 6, 2, 8), (4, 5, 3, 2)])
def test_equilibrium_matches_oracle_at_every_speed(Qp, Qxi, Np, Nv):
    v = np.array([s * b for b in SPEEDS for s in (1.0, -1.0)])
    rng = np.random.default_rng(5)
    P, n = rng.uniform(0.1, 2.0, v.size), rng.uniform(0.1, 2.0, v.size)
    t = rb.Tube(Qp, Qxi, Np, Nv, v.size, 1.0 / v.size, 1e-4, 1.0, rb.BC_OPEN, rb.STORAGE_F64)
    with rb.rlb_init([t], P, n, v) as h:
        F = rb.rlb_get_state(h).reshape(Qp * Qxi, v.size)
    for c in range(v.size):
        ref = oracle.feq_cell(Qp, Qxi, Np, Nv, n[c], P[c] / n[c], v[c])
        err = np.max(np.abs(F[:, c] - ref)) / np.max(np.abs(ref))
        assert err <= 1e-13 * (1.0 + 1.0 / (1.0 - v[c] ** 2)), (v[c], err)


def test_speed_limit_of_the_generic_orders():
    """Np = 3 takes one power more, so its documented limit lies lower than that of Np = 2 (0.9955)."""
    for v0, ok in ((0.99502, True), (0.99503, False), (np.nan, False)):
        t = rb.Tube(4, 7, 3, 8, 40, 1.0 / 40, 1e-4, 1.0, rb.BC_OPEN, rb.STORAGE_F64)
        make = lambda: rb.rlb_init([t], np.ones(40), np.ones(40), np.full(40, v0))  # noqa: E731
        if ok:
            make().__exit__()
        else:
            with pytest.raises(rb.RlbError):
                make()
