"""The batched tile step with its boxes as a kernel argument (up to 40) and
from tables (more): every box as when stepped alone, bitwise; all boxes
together and with step counts of their own (a shrinking prefix of the boxes)."""
import numpy as np
import pytest

import inputs
from paper_1708_01613_gb300 import Batch, Simulation, make_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 40, 41])
@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_boxes_step_as_alone(n, storage):
    sizes = [(40 + 13 * k % 97, 30 + 7 * k % 41) for k in range(n)]

    def make():
        sims = []
        for k, (nx, ny) in enumerate(sizes):
            s = Simulation(make_config(nx, ny, storage=storage, rho_ref=0.7))
            s.init_density(inputs.noise_density(nx, ny, seed=k, amp=0.05))
            sims.append(s)
        return sims

    together, alone = make(), make()
    each = [3 + k % 5 for k in range(n)]
    b = Batch(together)
    b.step(7)
    b.step_each(each)
    b.sync()
    for k in range(n):
        alone[k].set_step_variant(1)
        alone[k].step(7 + each[k])
        alone[k].sync()
        assert np.array_equal(together[k].read("pops")["pops"], alone[k].read("pops")["pops"]), k
