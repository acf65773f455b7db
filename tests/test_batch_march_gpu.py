"""Row march over a batch too large for several-step launches, bitwise
against each instance's own handle on the tile kernel: every edge kind, dry
strips, Dirichlet columns, ragged widths, an instance switched off."""
import numpy as np
import pytest

import inputs
from inputs import BOUNCEBACK, PERIODIC, SPECULAR

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def cases():
    return [
        inputs.dish_lake(450, seed=1),
        inputs.bump_channel(801, 333, seed=2),
        inputs.bump_channel(241, 70, seed=7),  # the last column alone past a multiple of 60
        inputs.random_case(517, 301, 3, edges=(PERIODIC, PERIODIC, SPECULAR, SPECULAR), dirichlet=False),
        inputs.random_case(61, 9, 4, edges=(BOUNCEBACK,) * 4, dirichlet=False),
        inputs.random_case(200, 7, 5, edges=(SPECULAR, SPECULAR, PERIODIC, PERIODIC), dirichlet=False),
        inputs.random_case(3, 130, 6, edges=(SPECULAR,) * 4, solids=False, dirichlet=False),
    ]


def test_equals_handles():
    from paper_1902_02999_gb300 import Batch, Simulation
    cs = cases()
    batch = Batch(cs, precision="f32")
    batch.set_graph_steps(8)
    batch.step(11)
    batch.set_active([1, 1, 1, 0, 1, 1, 1])
    batch.step(4)
    batch.set_active([1] * 7)
    batch.step(1)
    res = batch.residual()
    for i, c in enumerate(cs):
        sim = Simulation.from_case(c, precision="f32")
        sim.set_step_kernel("tile")
        sim.step(12 if i == 3 else 16)
        for a, b in zip(batch.get_state(i), sim.get_state()):
            assert np.array_equal(a, b), i
        r, m, u = sim.residual()
        # same terms, summed in another order
        assert abs(res[i, 0] - r) <= 1e-12 * r and abs(res[i, 1] - m) <= 1e-12 * m and res[i, 2] == u
        sim.close()
