"""Several steps per launch (the default on small grids and batches) against
one launch of the tile kernel per step, bitwise: both take the same
operations per node in the same order."""
import numpy as np
import pytest

import inputs
import oracle
from inputs import BOUNCEBACK, PERIODIC, SPECULAR

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EDGES = [
    (BOUNCEBACK, BOUNCEBACK, SPECULAR, SPECULAR),
    (PERIODIC, PERIODIC, SPECULAR, SPECULAR),
    (SPECULAR, SPECULAR, BOUNCEBACK, SPECULAR),
    (PERIODIC, PERIODIC, PERIODIC, PERIODIC),
    (BOUNCEBACK, SPECULAR, PERIODIC, PERIODIC),
]
# one node, one row, one column, two and three rows, odd sizes, sizes around
# a tile and a window, a grid of many tiles
SIZES = [(1, 1), (1, 37), (64, 1), (2, 2), (5, 3), (400, 3), (63, 33), (131, 97), (258, 130), (517, 301)]


def both(case, precision, steps, graph_steps=64):
    from paper_1902_02999_gb300 import Simulation
    out = []
    for kernel in (None, "tile"):
        sim = Simulation.from_case(case, precision=precision)
        sim.set_graph_steps(graph_steps)
        if kernel:
            sim.set_step_kernel(kernel)
        states = []
        for n in steps:
            sim.step(n)
            states.append(sim.get_state() + sim.residual())
        assert sim.time()[1] == sum(steps)
        out.append(states)
        sim.close()
    for a, b in zip(*out):
        for x, y in zip(a, b):
            assert np.array_equal(x, y, equal_nan=True)


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("edges", EDGES)
@pytest.mark.parametrize("nx,ny", SIZES)
def test_equals_tile_kernel(nx, ny, edges, precision):
    dirichlet = nx >= 8 and edges[0] != PERIODIC
    rows = dirichlet and ny >= 8 and edges[2] != PERIODIC and edges[3] != PERIODIC
    case = inputs.random_case(nx, ny, 11 + nx + ny, edges=edges, dirichlet=dirichlet, dirichlet_sn=rows)
    # one step, two, a launch's worth and its neighbours, many
    both(case, precision, (1, 2, 3, 7, 16, 17, 40))


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_graph_replay_and_walls(precision):
    both(inputs.dish_lake(70, seed=3), precision, (64, 1, 130, 2))
    both(inputs.bump_channel(130, 66, seed=4), precision, (1, 65, 64))
    both(inputs.bump_channel(130, 66, seed=4), precision, (129, 3), graph_steps=0)


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_tidal_strip_against_oracle(precision):
    case = inputs.tidal_strip(201, 3)
    from paper_1902_02999_gb300 import Simulation
    sim = Simulation.from_case(case, precision=precision)
    sim.step(301)
    h, u, v = sim.get_state()
    want = oracle.run(case, 301)
    # the FP64 bound of the parity tests on h; FP32 theirs
    assert np.abs(h - want[0]).max() <= (1e-12 if precision == "f64" else 2e-5) * np.abs(want[0]).max()


def test_chosen_kernel_and_mark():
    """A chosen step kernel takes every step; the interval residual agrees."""
    from paper_1902_02999_gb300 import Simulation
    case = inputs.dish_lake(96, seed=5)
    r = []
    for kernel in (None, "march"):
        sim = Simulation.from_case(case, precision="f32")
        if kernel:
            sim.set_step_kernel(kernel)
        sim.step(3)
        sim.mark()
        sim.step(50)
        r.append(sim.residual_since_mark())
        sim.close()
    assert r[0] == r[1]


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_batch_equals_handles(precision):
    """Instances of one batch on this path against handles on the tile kernel,
    with one switched off in between."""
    from paper_1902_02999_gb300 import Batch, Simulation
    cases = [inputs.dish_lake(50, seed=1), inputs.bump_channel(130, 40, seed=2),
             inputs.random_case(33, 65, 4, edges=(PERIODIC, PERIODIC, SPECULAR, SPECULAR), dirichlet=False),
             inputs.random_case(9, 7, 5, edges=(SPECULAR,) * 4, solids=False, dirichlet=False)]
    batch = Batch(cases, precision=precision)
    batch.set_graph_steps(16)
    batch.step(21)
    batch.set_active([1, 0, 1, 1])
    batch.step(5)
    batch.set_active([1, 1, 1, 1])
    batch.step(1)
    for i, c in enumerate(cases):
        sim = Simulation.from_case(c, precision=precision)
        sim.set_step_kernel("tile")
        sim.step(22 if i == 1 else 27)
        for a, b in zip(batch.get_state(i), sim.get_state()):
            assert np.array_equal(a, b), i
        sim.close()
