"""The tiled relabel (32 x 8 tiles) against the oracle's labels, owners and
masks, all equal, on rough gas: patches of noise whose pieces wind through
many tiles and around the box, boxes at the edges of tiles and at the smallest
size of a zone radius, every path of the owner search (R = 4, smaller,
larger, 16), with and without cells opened in the same relabel."""
import numpy as np
import pytest

import oracle as O
from paper_1708_01613_gb300 import Simulation, make_config

pytestmark = pytest.mark.gpu


def rough(nx, ny, seed, fill):
    """A density of 0.2 where smoothed noise is low (a share `fill`), else 2."""
    rng = np.random.default_rng(seed)
    a = rng.random((ny, nx))
    for ax in (0, 1):
        a = a + np.roll(a, 1, ax) + np.roll(a, -1, ax)
    return np.where(a < np.quantile(a, fill), 0.2, 2.0)


@pytest.mark.parametrize("nx,ny,R", [(10, 10, 4), (10, 41, 4), (33, 10, 4), (65, 12, 3), (32, 8, 3), (96, 64, 4), (130, 67, 1),
                                     (131, 95, 15), (67, 35, 16), (515, 301, 4)])
@pytest.mark.parametrize("fill", [0.04, 0.45])
@pytest.mark.parametrize("eps", [-1.0, 0.5])
def test_relabel_of_rough_gas(nx, ny, R, fill, eps):
    rho = rough(nx, ny, nx + R, fill)
    sim = Simulation(make_config(nx, ny, barrier=True, zone_radius=R, rupture_eps=eps, relabel_every=1))
    sim.init_density(rho)
    label = sim.read("label")["label"]  # of the density now, by the diagnostics' kernels
    sim.step(1)
    got = sim.read("owner", "mask", "open")
    P = O.make_params(nx, ny, barrier=True, zone_radius=R)
    assert (rho < P.gas_threshold).any() and (rho >= P.gas_threshold).any()
    lab = O.label(P, rho)
    own = O.owner(P, lab)
    assert np.array_equal(label, lab)
    assert np.array_equal(got["owner"], own)  # at gas cells: the label
    if eps < 0:
        assert not got["open"].any()
    assert np.array_equal(got["mask"], O.mask(P, own, got["open"]))


def test_relabel_of_moving_gas():
    """Labels of a tile whose gas has gone since the previous relabel are
    cleared."""
    nx, ny = 97, 45
    sim = Simulation(make_config(nx, ny, barrier=True, relabel_every=1, rupture_eps=-1.0))
    sim.init_bubbles([[30.3, 20.2, 9.0], [70.0, 25.0, 3.0]], 2.306865, 0.104158, 4.0)  # the small one dissolves
    P = O.make_params(nx, ny, barrier=True)
    seen = []
    for _ in range(80):
        before = sim.read("rho")["rho"]
        sim.step(1)
        got = sim.read("owner", "mask", "open")
        clear = np.abs(before - P.gas_threshold).min() > 1e-5
        seen.append(len(np.unique(got["owner"])))
        if clear:
            lab = O.label(P, before.astype(np.float64))
            own = O.owner(P, lab)
            assert np.array_equal(got["owner"], own)
            assert np.array_equal(got["mask"], O.mask(P, own, got["open"]))
    assert max(seen) > min(seen)
