"""Automatic split of the FP64 stage kernel by schedule. The one-CTA-per-tile launch shares a tile's per-cell work among
its CTAs, the persistent ones repeat it for every work item: with more tiles than resident CTAs their automatic choice
must not cost more than one item per tile. Times are the smaller of several alternating runs on one handle; the allowed
difference, 5 %, is ten times the spread of such runs (0.5 %), a repeated moment pass costs 25 % and more."""
import numpy as np
import pytest
import torch

from paper_1608_03004_gb300 import binding as rb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("schedule", [rb.SCHED_STRIDE, rb.SCHED_COUNTER], ids=["stride", "counter"])
@pytest.mark.parametrize("ntiles,Qxi", [(500, 128), (1000, 32)])
def test_persistent_schedules_are_not_split_when_the_tiles_fill_the_gpu(schedule, ntiles, Qxi):
    Nx = 60 * ntiles
    x = np.arange(Nx) / Nx * 2 * np.pi
    t = rb.Tube(3, Qxi, 2, 5, Nx, 1.0 / Nx, 0.4 / Nx, 1e-2, rb.BC_PERIODIC, rb.STORAGE_F64)
    with rb.rlb_init([t], 1 + 0.2 * np.sin(x), 1 + 0.2 * np.cos(x), 0.3 * np.sin(x)) as h:
        best = [np.inf, np.inf]
        for k in range(12):
            rb.rlb_set_launch(h, dict(schedule=schedule, ctas_per_sm=0, graph_steps=0, order=0, split=k % 2))
            rb.rlb_step(h, 1)
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            rb.rlb_step(h, 4)
            e[1].record()
            torch.cuda.synchronize()
            best[k % 2] = min(best[k % 2], e[0].elapsed_time(e[1]))
    assert best[0] <= 1.05 * best[1], best
