"""The FP64 mass (lbm_mass and the statistics') against the exactly rounded sum
of the populations: no value is lost beside larger ones, sums beyond the FP32
range are finite, and infinities and NaN come out as FP64 adds give them.

Tolerance: a value passes through at most 40 FP64 additions (chunks of a thread,
the tree over a block, the partial sums), each within 2^-53."""
import math

import numpy as np
import pytest

from paper_1708_01613_gb300 import Simulation, make_config

pytestmark = pytest.mark.gpu

TOL = 40 * 2.0**-53
SMALL = 2.0**-25 * (1 + 2.0**-23)  # below half an ulp of 1, with all 24 bits


def populations(kind, nx, ny, seed):
    rng = np.random.default_rng(seed)
    if kind == "beside":
        f = np.where(rng.random((9, ny, nx)) < 1 / 32, 1.0, SMALL)
    elif kind == "spread":
        f = 10.0 ** rng.uniform(-12, 0, (9, ny, nx)) * rng.choice([-0.25, 1.0], (9, ny, nx))
    else:  # "huge": FP32 sums overflow, FP64 sums do not
        f = 3e38 * rng.random((9, ny, nx))
    return f.astype(np.float32)


def masses(sim):
    return sim.mass(), sim.stats()["mass"]


@pytest.mark.parametrize("nx,ny", [(4, 4), (37, 13), (256, 64), (2051, 33)])
@pytest.mark.parametrize("kind,storage", [("beside", "f32"), ("spread", "f32"), ("huge", "f32"), ("spread", "f16"),
                                          ("spread", "bf16")])
def test_mass_is_the_sum_in_fp64(nx, ny, kind, storage):
    sim = Simulation(make_config(nx, ny, storage=storage, rho_ref=0.3))
    sim.load_populations(populations(kind, nx, ny, nx))
    f = sim.read("pops")["pops"].astype(np.float64).ravel()
    exact, scale = math.fsum(f), math.fsum(np.abs(f))
    for got in masses(sim):
        assert abs(got - exact) <= TOL * scale, (got, exact)


@pytest.mark.parametrize("nx,ny", [(37, 13), (2051, 33)])
@pytest.mark.parametrize("values", [[np.inf], [-np.inf], [np.nan], [np.inf, -np.inf], [np.inf, 3e38]])
def test_mass_of_infinities(nx, ny, values):
    f = populations("spread", nx, ny, 1)
    f[4, ny // 2, 5:5 + len(values)] = values
    sim = Simulation(make_config(nx, ny))
    sim.load_populations(f)
    with np.errstate(invalid="ignore"):
        want = np.sum(np.asarray(values, np.float64))
    for got in masses(sim):
        assert got == want or (np.isnan(got) and np.isnan(want)), (got, want)
