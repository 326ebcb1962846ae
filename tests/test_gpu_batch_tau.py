"""Batches of boxes with different relaxation times: each box takes the
collision that it takes alone, also a tau = 1 box among others (outgoing
populations equal to the equilibrium, not the blend with it). Bitwise against
the boxes stepped alone, in tiles and on the staged kernel (FP32, tau != 1,
above 1.5 M cells)."""
import numpy as np
import pytest

import inputs
from paper_1708_01613_gb300 import Batch, Simulation, make_config

pytestmark = pytest.mark.gpu

RL, RG = inputs.RHO_LIQ_G55, inputs.RHO_GAS_G55
SMALL = [(256, 64, 1.0), (131, 77, 0.8), (250, 100, 1.0), (12, 40, 1.3), (13, 41, 1.0)]
LARGE = SMALL + [(1301, 700, 1.0), (777, 801, 0.8)]


def boxes(sizes, storage, barrier):
    out = []
    for i, (nx, ny, tau) in enumerate(sizes):
        sim = Simulation(make_config(nx, ny, storage=storage, tau=tau, barrier=barrier, relabel_every=3, rho_ref=RL))
        r = 0.22 * min(nx, ny)  # two bubbles 3 cells apart
        sim.init_bubbles([[nx / 2 - 0.3, ny / 2 - r - 1.5, r], [nx / 2 + 0.2, ny / 2 + r + 1.5, r]], RL, RG, 4.0)
        out.append(sim)
    return out


@pytest.mark.parametrize("barrier", [False, True])
@pytest.mark.parametrize("sizes,storage", [(SMALL, "f32"), (SMALL, "f16"), (SMALL, "bf16"), (LARGE, "f32")])
def test_boxes_of_several_tau(sizes, storage, barrier):
    cells = sum(nx * ny for nx, ny, _ in sizes)
    assert (cells > 1500000) == (sizes is LARGE)
    alone, batched = boxes(sizes, storage, barrier), boxes(sizes, storage, barrier)
    b = Batch(batched)
    b.step(4)
    counts = [3 + i % 3 for i in range(len(sizes))]
    b.step_each(counts)
    b.sync()
    b.close()
    blocked = 0
    for s, a, n in zip(batched, alone, counts):
        a.step(4 + n)
        got, ref = s.read("pops", "mask"), a.read("pops", "mask")
        assert np.array_equal(got["pops"], ref["pops"]), (s.nx, s.ny, s.cfg.tau)
        assert np.array_equal(got["mask"], ref["mask"])
        blocked += int(np.count_nonzero(got["mask"]))
    assert (blocked > 0) == barrier
