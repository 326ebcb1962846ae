"""The tile step (the automatic variant) against the plain-load step: bitwise
the same populations on boxes at the edges of its tiles (60 and 120 columns,
6 and 10 rows; one row or column more and less; the narrowest boxes), for every
storage, tau = 1 and not, with its small and its large tile; and with films,
where its pull does the bounce-back between relabels that the plain-load step
leaves to a kernel of its own."""
import numpy as np
import pytest

import inputs
from paper_1708_01613_gb300 import Batch, Simulation, make_config

pytestmark = pytest.mark.gpu

RL, RG = inputs.RHO_LIQ_G55, inputs.RHO_GAS_G55


def run(variant, nx, ny, steps, calls=1, bubbles=None, **kw):
    sim = Simulation(make_config(nx, ny, barrier=bubbles is not None, rho_ref=RL if bubbles is not None else 0.7, **kw))
    if bubbles is not None:
        sim.init_bubbles(bubbles, RL, RG, 4.0)
    else:
        sim.init_density(inputs.noise_density(nx, ny, seed=3, amp=0.05))
    sim.set_step_variant(variant)
    for _ in range(calls):
        sim.step(steps)
    sim.sync()
    return sim


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("tau", [1.0, 0.8])
@pytest.mark.parametrize("nx,ny", [(4, 4), (5, 7), (59, 6), (60, 5), (61, 12), (62, 13), (120, 4), (121, 11), (182, 19),
                                   (1099, 1101)])
def test_tile_step_matches_plain_step(storage, tau, nx, ny):
    steps = 7 if nx > 1000 else 23
    a = run(0, nx, ny, steps, storage=storage, tau=tau).read("pops")["pops"]
    b = run(1, nx, ny, steps, storage=storage, tau=tau).read("pops")["pops"]
    assert np.array_equal(a, b)


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("nx,ny,cx", [(121, 62, 60.0), (121, 62, 0.5), (1103, 1091, 1102.0)])
def test_pull_bounces_back_across_films(storage, nx, ny, cx):
    """A film of two cells (wider bubbles merge slower than the run) inside a
    tile, and across the periodic seam, where the mask's and the populations'
    ghosts carry it; calls of 7 steps against a relabel period of 5."""
    r = 14.0
    bub = [[cx - r - 1.0, ny / 2, r], [(cx + r + 1.0) % nx, ny / 2, r]]
    bub = [[b[0] % nx, b[1], b[2]] for b in bub]
    out = [run(v, nx, ny, 7, calls=3, bubbles=bub, storage=storage, relabel_every=5, rupture_eps=-1.0).read("pops", "mask")
           for v in (0, 1)]
    assert out[0]["mask"].any()
    assert np.array_equal(out[0]["mask"], out[1]["mask"]) and np.array_equal(out[0]["pops"], out[1]["pops"])


def test_batch_items_of_ragged_boxes():
    """Tiles of a batch: boxes at tile edges, different relabel phases, rates."""
    sizes = [(61, 12), (120, 23), (181, 31), (40, 40)]
    bub = [[[s[0] / 2, s[1] / 2, min(s) / 4]] for s in sizes]
    ref = [run(1, *s, n, bubbles=b, relabel_every=4, storage="f16") for s, b, n in zip(sizes, bub, (9, 12, 5, 7))]
    boxes = [run(0, *s, 0, bubbles=b, relabel_every=4, storage="f16") for s, b in zip(sizes, bub)]
    batch = Batch(boxes)
    batch.step_each([4, 7, 0, 2])
    batch.step(5)
    batch.sync()
    batch.close()
    for a, b in zip(boxes, ref):
        assert a.steps_done == b.steps_done
        assert np.array_equal(a.read("pops")["pops"], b.read("pops")["pops"])
