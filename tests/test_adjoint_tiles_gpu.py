"""The adjoint's two kernels at the edges of their tiles (60 cells per row tile, 16 per per-cell tile) and of their
mirror pairs: tubes of 3 to 121 cells, odd and even Qxi, three and four radial nodes, both orders of the kernels,
open and periodic, with and without collisions, one and several tubes in a handle (which changes the split).

One step from a smooth state; L = sum of seeded weights times the fields. The reverse sweep's directional derivative
along a smooth change of (P, n, v) and of log(tau) must match the fourth-order central difference of the GPU forward
at h = 1e-4: truncation ~h^4 times the fifth derivative (1e-16 x at most 1e4) and rounding ~1e-15 |L| / h = 1e-11 |L|,
so 1e-8 relative to the sum of the terms' magnitudes."""
import math

import numpy as np
import pytest
import torch

from paper_1608_03004_gb300 import binding as rb

pytestmark = pytest.mark.gpu

CASES = [  # Nx, Qxi, Qp, Np, Nv, bc, tau
    (3, 4, 3, 2, 5, rb.BC_PERIODIC, 0.05), (7, 5, 3, 2, 5, rb.BC_OPEN, 0.05), (16, 8, 3, 2, 5, rb.BC_OPEN, 0.02),
    (17, 9, 4, 3, 8, rb.BC_PERIODIC, 0.05), (59, 4, 3, 2, 5, rb.BC_PERIODIC, 0.1), (60, 33, 3, 2, 5, rb.BC_OPEN, 0.05),
    (61, 6, 4, 2, 5, rb.BC_OPEN, math.inf), (64, 7, 3, 2, 8, rb.BC_PERIODIC, 0.03), (120, 11, 4, 3, 6, rb.BC_OPEN, 0.05),
    (121, 16, 3, 2, 5, rb.BC_PERIODIC, math.inf),
]


def problem(cases):
    P, n, v, d = [], [], [], []
    for k, c in enumerate(cases):
        x = (np.arange(c[0]) + 0.5) / c[0] * 2 * np.pi
        P.append(1.0 + 0.2 * np.sin(x + k))
        n.append(1.0 + 0.2 * np.cos(x + 0.5 * k))
        v.append(0.3 * np.sin(x + 1.0 + k))
        d.append(np.stack([0.3 * np.cos(x), 0.2 * np.sin(x + 2.0), 0.25 * np.cos(x - 1.0)]))
    return [np.concatenate(a) for a in (P, n, v)], np.concatenate(d, axis=1)


def tubes_of(cases, dlt=0.0):
    return [rb.Tube(Qp, Qxi, Np, Nv, Nx, 1.0 / Nx, min(0.4 / Nx, 0.4 * tau), tau * math.exp(dlt), bc, rb.STORAGE_F64)
            for Nx, Qxi, Qp, Np, Nv, bc, tau in cases]


@pytest.mark.parametrize("cases", [[c] for c in CASES] + [CASES], ids=[f"{c[0]}x{c[1]}" for c in CASES] + ["all"])
def test_directional_derivative(cases):
    (P, n, v), d = problem(cases)
    nx = P.size
    R = np.random.default_rng(9).normal(size=(rb.NFIELDS, nx))

    def L(h):
        with rb.rlb_init(tubes_of(cases, h), P + h * d[0], n + h * d[1], v + h * d[2]) as hd:
            rb.rlb_step(hd, 1)
            return float(np.sum(R * rb.rlb_moments(hd)))

    h = 1e-4
    fd = (8 * (L(h) - L(-h)) - (L(2 * h) - L(-2 * h))) / (12 * h)
    dev = lambda a: torch.tensor(a, device="cuda")  # noqa: E731
    with rb.rlb_init(tubes_of(cases), P, n, v) as hd:
        rb.rlb_record(hd, 1, 1)
        seed = torch.empty(hd.state_size, dtype=torch.float64, device="cuda")
        rb.rlb_fields_vjp(hd, dev(R), seed)
        gF, glt = rb.rlb_backward(hd, seed, torch.empty_like(seed))
        g = [torch.empty(nx, dtype=torch.float64, device="cuda") for _ in range(3)]
        rb.rlb_init_vjp(hd, dev(P), dev(n), dev(v), gF, *g)
    terms = np.concatenate([(a.cpu().numpy() * b) for a, b in zip(g, d)])
    assert all(t == 0.0 for t, c in zip(glt, cases) if math.isinf(c[6]))
    got, scale = terms.sum() + glt.sum(), np.abs(terms).sum() + np.abs(glt).sum()
    assert abs(got - fd) <= 1e-8 * scale, (got, fd, scale)
