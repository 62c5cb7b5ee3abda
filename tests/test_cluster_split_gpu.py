"""Every split of the FP64 stage kernel against one item per tile, bit for bit. With the one-CTA-per-tile schedule the
items of a tile share its cells: 30 and 20 cells each (splits 2 and 3), 15 to 9 (4 to 7, the last share shorter at 7) and
8 (split 8, where the coefficients are built one per thread). Tubes of both kernel paths (default orders, polynomial
equilibrium; generic orders, Legendre basis), odd and even Qxi, a ballistic one, sizes off the tile width of 60."""
import math

import numpy as np
import pytest

from paper_1608_03004_gb300 import binding as rb

pytestmark = pytest.mark.gpu

TUBES = [  # Nx, Qxi, Qp, Np, Nv, bc, tau
    (131, 8, 3, 2, 5, rb.BC_OPEN, 2e-2), (60, 9, 3, 2, 5, rb.BC_PERIODIC, 5e-2), (77, 7, 4, 3, 8, rb.BC_OPEN, 5e-2),
    (121, 12, 4, 2, 8, rb.BC_PERIODIC, 3e-2), (61, 10, 4, 2, 5, rb.BC_OPEN, math.inf), (3, 5, 3, 2, 5, rb.BC_PERIODIC, 5e-2),
]


def run(tubes, shape, steps=5):
    P, n, v, ts = [], [], [], []
    for k, (Nx, Qxi, Qp, Np, Nv, bc, tau) in enumerate(tubes):
        x = (np.arange(Nx) + 0.5) / Nx * 2 * np.pi
        P.append(1 + 0.3 * np.sin(x + k))
        n.append(1 + 0.2 * np.cos(x + 0.3 * k))
        v.append(0.6 * np.sin(x + 1 + k))
        ts.append(rb.Tube(Qp, Qxi, Np, Nv, Nx, 1.0 / Nx, min(0.3 / Nx, 0.3 * tau), tau, bc, rb.STORAGE_F64))
    with rb.rlb_init(ts, np.concatenate(P), np.concatenate(n), np.concatenate(v)) as h:
        rb.rlb_set_launch(h, shape)
        rb.rlb_step(h, steps)
        return rb.rlb_get_state(h)


@pytest.mark.parametrize("tubes", [TUBES, TUBES[2:3], TUBES[:1]], ids=["all", "generic", "default"])
def test_every_split_is_bit_identical(tubes):
    shape = dict(schedule=rb.SCHED_TILE, ctas_per_sm=0, graph_steps=0, order=rb.ORDER_COST, split=1)
    ref = run(tubes, shape)
    for split in range(2, 9):
        np.testing.assert_array_equal(run(tubes, dict(shape, split=split)), ref, err_msg=f"tile {split}")
        np.testing.assert_array_equal(run(tubes, dict(shape, schedule=rb.SCHED_COUNTER, split=split)), ref,
                                      err_msg=f"counter {split}")
    np.testing.assert_array_equal(run(tubes, dict(shape, split=7, graph_steps=2)), ref, err_msg="graph 7")
