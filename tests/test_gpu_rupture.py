"""The rupture test of the relabel against the oracle's, cell by cell: which
cells open for a small |D2| (Eq. 41) and, at a second relabel of another state,
for a sign that turned; the mask that the oracle's opened cells leave. Rough gas
in boxes at the edges of tiles and across their seams, every path of the owner
search, the untiled relabel (R = 18) and the three storages.

The oracle takes the densities that the GPU read out. Cells whose opening
differs between thresholds 3e-6 below and above eps are left out: four FP32
pressures of magnitude 1 are off by less."""
import numpy as np
import pytest

import oracle as O
from paper_1708_01613_gb300 import Simulation, make_config

pytestmark = pytest.mark.gpu

EPS, MARGIN = 1e-3, 3e-6


def density(gas, seed):
    """0.2 in the gas; in the liquid smoothed noise around 2."""
    a = np.random.default_rng(seed).standard_normal(gas.shape)
    a = a + np.roll(a, 1, 0) + np.roll(a, 1, 1)
    return np.where(gas, 0.2, 2.0 + 0.01 * a)


def populations(rho):
    w = np.array([4 / 9] + 4 * [1 / 9] + 4 * [1 / 36])[:, None, None]
    return (w * rho).astype(np.float32)


@pytest.mark.parametrize("nx,ny,R", [(10, 10, 4), (33, 10, 4), (96, 64, 4), (131, 95, 15), (67, 35, 16), (515, 301, 4),
                                     (130, 67, 2), (90, 61, 18)])
@pytest.mark.parametrize("fill", [0.06, 0.45])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_opened_cells(nx, ny, R, fill, storage):
    rng = np.random.default_rng(nx + R)
    a = rng.random((ny, nx))
    a = a + np.roll(a, 1, 0) + np.roll(a, 1, 1)
    gas = a < np.quantile(a, fill)
    sim = Simulation(make_config(nx, ny, storage=storage, barrier=True, zone_radius=R, rupture_eps=EPS, relabel_every=1,
                                 rho_ref=2.0))
    sim.init_density(density(gas, 1))
    params = [O.make_params(nx, ny, barrier=True, zone_radius=R, rupture_eps=EPS + d) for d in (-MARGIN, 0.0, MARGIN)]
    sgn = [np.zeros((ny, nx), np.int8) for _ in params]
    opened = [np.zeros((ny, nx), np.uint8) for _ in params]
    film, before = 0, 0
    for k in (1, 2):
        rho = sim.read("rho")["rho"].astype(np.float64)
        own = O.owner(params[1], O.label(params[1], rho))
        for p, s, o in zip(params, sgn, opened):
            O.rupture(p, rho, own, s, o)
        film += int(np.count_nonzero(sgn[1]))
        sim.step(1)
        got = sim.read("owner", "open", "mask")
        assert np.array_equal(got["owner"], own)
        sure = opened[0] == opened[2]
        assert np.count_nonzero(~sure) <= 0.01 * film + 2
        assert np.array_equal(got["open"][sure], opened[1][sure]), k
        assert np.array_equal(got["mask"], O.mask(params[1], own, np.where(sure, opened[1], got["open"])))
        if film > 100:  # some cells open, and at the second relabel more of them
            assert before < np.count_nonzero(opened[1]) < film
        before = np.count_nonzero(opened[1])
        sim.load_populations(populations(density(gas, 2)))  # labels, signs and opened cells stay
