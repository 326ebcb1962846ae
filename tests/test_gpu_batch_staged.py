"""Batches above the tile kernel's range: the two-cell staged kernel over work
items of all boxes (16-bit storage above 30 M cells, FP32 with tau != 1 above 1.5
M), with a box narrower than it takes, in graphs and without, at several item
sizes, multi-rate steps, a box switched off and the tuner. Bitwise against each
box alone on the plain-load step."""
import numpy as np
import pytest

import inputs
from paper_1708_01613_gb300 import Batch, Simulation, make_config

pytestmark = pytest.mark.gpu

RL, RG = inputs.RHO_LIQ_G55, inputs.RHO_GAS_G55
SMALL = [(250, 100), (131, 77), (512, 33), (13, 41)]


def make_boxes(sizes, storage, barrier, tau):
    out = []
    for i, (nx, ny) in enumerate(sizes):
        sim = Simulation(make_config(nx, ny, storage=storage, tau=tau, barrier=barrier, relabel_every=3, rho_ref=RL))
        rng = np.random.default_rng(i)
        r = 0.2 * min(nx, ny, 150)
        x, y = (rng.random((2, 1 + 40 * (nx > 1000))) * [[nx], [ny]])  # pairs of bubbles 3 cells apart
        sim.init_bubbles(np.concatenate([np.stack([x, y, 0 * x + r], 1),
                                         np.stack([x, (y + 2 * r + 3) % ny, 0 * x + r], 1)]), RL, RG, 4.0)
        out.append(sim)
    return out


@pytest.mark.parametrize("storage,tau,large", [("f16", 1.0, (5501, 5460)), ("bf16", 1.0, (5501, 5460)),
                                               ("f32", 0.8, (1301, 1163))])
@pytest.mark.parametrize("barrier", [False, True])
@pytest.mark.parametrize("graph", [False, True])
def test_staged_batch_matches_boxes_alone(storage, tau, large, barrier, graph):
    sizes = SMALL[:2] + [large] + SMALL[2:]
    assert sum(nx * ny for nx, ny in sizes) > (1500000 if storage == "f32" else 30000000)
    batched, alone = make_boxes(sizes, storage, barrier, tau), make_boxes(sizes, storage, barrier, tau)
    done = np.zeros(len(sizes), int)
    b = Batch(batched)
    b.use_graph(graph)
    b.step(7)
    done += 7
    for strip, rows in ((256, 16), (512, 40)):
        b.set_tiles(strip, rows)
        counts = [(2 * i + strip // 256) % 5 for i in range(len(sizes))]
        b.step_each(counts)
        b.step(4)
        done += np.array(counts) + 4
    b.set_active(1, False)
    b.step(5)
    b.set_active(1, True)
    done += np.array([5, 0, 5, 5, 5])
    b.tune(trial_steps=1)
    done += 20  # ten candidates x (1 + 1) steps
    b.sync()
    b.close()
    blocked = 0
    for s, a, n in zip(batched, alone, done):
        a.set_step_variant(1)
        a.step(int(n))
        assert s.steps_done == n
        got, ref = s.read("pops", "mask", device=True), a.read("pops", "mask", device=True)
        assert got["pops"].equal(ref["pops"]), (s.nx, s.ny)
        assert got["mask"].equal(ref["mask"])
        blocked += int((got["mask"] != 0).sum())
    assert (blocked > 0) == barrier
