"""Memory of the several-step path's lists: room for the nodes with a
bounce-back link that a window holds, not for all its nodes."""
import numpy as np
import pytest

import inputs
from inputs import BOUNCEBACK, PERIODIC, SPECULAR

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make", [
    lambda: inputs.dish_lake(256, seed=1),
    lambda: inputs.random_case(1001, 333, 3, edges=(BOUNCEBACK,) * 4, dirichlet=False),
    lambda: inputs.random_case(600, 500, 4, edges=(PERIODIC, PERIODIC, SPECULAR, SPECULAR)),
], ids=["lake", "walls", "blocks"])
def test_bytes(make):
    from paper_1902_02999_gb300 import Simulation
    case = make()
    sim = Simulation.from_case(case, precision="f32")
    nodes = case.nx * case.ny
    # two states, depths, types and transfers: 61 a node; the path's scratch
    # state 12; its windows' units 16 each for at most two nodes, with up to
    # four times the nodes in overlapping windows 32; 15 for the rest
    assert sim.info["device_bytes"] <= (61 + 12 + 32 + 15) * nodes * 1.03 + (1 << 20)
    sim.close()


@pytest.mark.parametrize("nx,ny,edges", [
    (23, 41, (PERIODIC,) * 4),               # windows wrap more than once
    (150, 31, (PERIODIC, PERIODIC, BOUNCEBACK, BOUNCEBACK)),
    (31, 150, (BOUNCEBACK, SPECULAR, PERIODIC, PERIODIC)),
    (201, 180, (BOUNCEBACK,) * 4),
    (12, 12, (BOUNCEBACK,) * 4),
])
def test_walls_everywhere(nx, ny, edges):
    """Solid nodes on a lattice: nearly every node has such a link."""
    from paper_1902_02999_gb300 import Batch, Simulation
    case = inputs.random_case(nx, ny, 7, edges=edges, solids=False, dirichlet=False)
    yy, xx = np.mgrid[0:ny, 0:nx]
    solid = (xx % 3 == 1) & (yy % 4 == 2)
    case.mask[solid] = inputs.SOLID
    for q in (case.h0, case.u0, case.v0):
        q[solid] = 0.0
    sims = [Simulation.from_case(case, precision="f32") for _ in range(2)]
    sims[1].set_step_kernel("tile")
    batch = Batch([case, case], precision="f32")
    for s in sims + [batch]:
        s.step(16)
        s.step(3)
    for a, b, c, d in zip(sims[0].get_state(), sims[1].get_state(), batch.get_state(0), batch.get_state(1)):
        assert np.array_equal(a, b) and np.array_equal(b, c) and np.array_equal(b, d)
