"""Steps of a small box in one launch (a cluster's shared memory) against one
launch per step, bitwise: boxes at the edges of the rows a CTA holds (16 CTAs;
fewer rows than CTAs, a CTA with fewer rows, idle CTAs), of one and two pairs
per thread and of the largest size taken; odd widths; every storage; tau = 1
and not; films between relabels; and runs of fewer steps than the launch takes."""
import numpy as np
import pytest

import inputs
from paper_1708_01613_gb300 import Simulation, make_config

pytestmark = pytest.mark.gpu

RL, RG = inputs.RHO_LIQ_G55, inputs.RHO_GAS_G55


def make(variant, nx, ny, bubbles=None, **kw):
    sim = Simulation(make_config(nx, ny, barrier=bubbles is not None, rho_ref=RL if bubbles is not None else 0.7, **kw))
    if bubbles is not None:
        sim.init_bubbles(bubbles, RL, RG, 4.0)
    else:
        sim.init_density(inputs.noise_density(nx, ny, seed=5, amp=0.05))
    sim.set_step_variant(variant)
    return sim


@pytest.mark.parametrize("storage,tau", [("f32", 1.0), ("f32", 0.8), ("f16", 1.0), ("bf16", 0.8)])
@pytest.mark.parametrize("nx,ny", [(4, 4), (5, 15), (7, 16), (33, 17), (16, 31), (127, 129), (128, 128), (1000, 16), (311, 100),
                                   (64, 511), (256, 128)])
def test_many_steps_match_single_steps(nx, ny, storage, tau):
    a, b, c = (make(v, nx, ny, storage=storage, tau=tau) for v in (0, 1, 0))
    before = a.kernel_launches
    a.step(24)
    a.step(5)
    b.step(29)
    for k in (3, 3, 3, 20):  # short calls take a launch per step
        c.step(k)
    for s in (a, b, c):
        s.sync()
    want = b.read("pops")["pops"]
    assert np.array_equal(a.read("pops")["pops"], want) and np.array_equal(c.read("pops")["pops"], want)
    assert a.steps_done == 29
    if (nx, ny) == (128, 128):
        assert a.kernel_launches - before == 2  # the box is one that the launch takes


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("nx,ny,cx,cy", [(121, 62, 60.0, 31.0), (121, 62, 0.5, 31.0), (65, 100, 32.0, 0.2)])
def test_films_between_relabels(storage, nx, ny, cx, cy):
    """A film of two cells, inside, across the seam, and along the strips."""
    r = 14.0
    bub = [[(cx - r - 1.0) % nx, cy, r], [(cx + r + 1.0) % nx, cy, r]]
    out = []
    for v in (0, 1):
        sim = make(v, nx, ny, bubbles=bub, storage=storage, relabel_every=6, rupture_eps=-1.0)
        for k in (8, 7, 9):
            sim.step(k)
        sim.sync()
        out.append(sim.read("pops", "mask", "owner"))
    assert out[0]["mask"].any()
    for f in ("mask", "owner", "pops"):
        assert np.array_equal(out[0][f], out[1][f])
