"""A field's value does not depend on which others are read with it."""
import itertools

import numpy as np
import pytest

import inputs
from paper_1708_01613_gb300 import Simulation, make_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,barrier,comps", [("f32", True, 1), ("f32", False, 1), ("f16", True, 1), ("bf16", False, 1),
                                                   ("f32", True, 2)])
def test_fields_read_alone_and_together(storage, barrier, comps):
    nx, ny = 121, 52
    sim = Simulation(make_config(nx, ny, storage=storage, barrier=barrier, components=comps, G=-5.5 if comps == 1 else -1.0,
                                 G_mg=2.5 if comps == 2 else 0.0, rho_ref=inputs.RHO_LIQ_G55))
    if comps == 2:
        sim.init_density(inputs.noise_density(nx, ny, seed=1), inputs.noise_density(nx, ny, seed=2, rho_mean=0.6))
    else:
        sim.init_bubbles([[48.0, 25.0, 11.0], [73.0, 25.5, 11.0]], inputs.RHO_LIQ_G55, inputs.RHO_GAS_G55, 4.0)
    sim.step(30)
    names = ["rho", "ux", "uy", "p", "rho_gas", "label"]
    together = sim.read(*names)
    assert np.abs(together["ux"]).max() > 1e-4 and np.abs(together["uy"]).max() > 1e-4
    for n in (1, 2):
        for chosen in itertools.combinations(names, n):
            got = sim.read(*chosen)
            for k in chosen:
                assert np.array_equal(got[k], together[k]), (chosen, k)
