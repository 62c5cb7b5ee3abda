"""The collision keeps N^0 and T^00, so on a periodic tube the gradient in log(tau) of their sums is zero. What the
adjoint returns instead is the error of its equilibrium in the two moments, summed over cells and stages: gradients in
log(tau) are sums whose terms cancel, and a bias of that equilibrium is what is left of them.

Tolerance on the mean relative error of a moment per collision: the radial constants meet the moment conditions to
7.5e-18 (sum over their orders), the polar weights sum to 2 with an error that is taken from the rule itself, and the
rounding of one equilibrium, at most 6e-16 in a moment, averages over 4096 cells and 30 stages to 1.7e-18, 5 times of it
taken: 7.5e-18 + 8.5e-18 < 2e-17. With constants rounded one by one the bias was 5e-17 (Qp = 3) to 2e-16 (Qp = 4)."""
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_1608_03004_gb300 import binding as rb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Qp,Np,Nv,Qxi", [(3, 2, 5, 32), (3, 2, 5, 9), (3, 2, 8, 8), (4, 2, 5, 16), (4, 3, 8, 8)])
def test_equilibrium_of_the_adjoint_keeps_the_moments(Qp, Np, Nv, Qxi):
    Nx, steps, tau = 4096, 10, 5e-2
    x = np.arange(Nx) / Nx * 2 * np.pi
    dt = 0.5 / Nx
    t = rb.Tube(Qp, Qxi, Np, Nv, Nx, 1.0 / Nx, dt, tau, rb.BC_PERIODIC, rb.STORAGE_F64)
    weights = rb.rlb_quadrature(Qp, Qxi)[3]
    polar = abs(float(sum(Fraction(float(w)) for w in weights) / 2 - 1))
    with rb.rlb_init([t], 1 + 0.4 * np.sin(x), 1 + 0.3 * np.cos(2 * x), 0.3 * np.sin(x + 1)) as h:
        M = rb.rlb_moments(h)
        F0 = rb.rlb_get_state(h)
        for k in (0, 2):  # N^0, T^00
            rb.rlb_set_state(h, F0)
            rb.rlb_record(h, steps, steps)
            g = torch.zeros((5, Nx), dtype=torch.float64, device="cuda")
            g[k] = 1.0
            seed = torch.empty(h.state_size, dtype=torch.float64, device="cuda")
            rb.rlb_moments_vjp(h, g, seed)
            _, glt = rb.rlb_backward(h, seed, torch.empty_like(seed))
            # the stages of a step weigh 1/6, 1/6 and 2/3
            bias = glt[0] / (M[k].sum() * steps * dt / tau)
            assert abs(bias) <= 2e-17 + polar, (k, bias, polar)
