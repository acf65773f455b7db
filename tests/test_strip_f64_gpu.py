"""The warp-strip kernel in FP64 against the tile kernel (bitwise) over every
edge kind, and its rows per strip, which change nothing."""
import numpy as np
import pytest

import inputs
import oracle
from inputs import BOUNCEBACK, PERIODIC, SPECULAR

from test_parity_gpu import compare

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EDGES = [
    (BOUNCEBACK, BOUNCEBACK, SPECULAR, SPECULAR),
    (PERIODIC, PERIODIC, SPECULAR, SPECULAR),
    (SPECULAR,) * 4,
    (PERIODIC,) * 4,
    (BOUNCEBACK,) * 4,
    (BOUNCEBACK, SPECULAR, PERIODIC, PERIODIC),
]


def sim_of(case, kernel, precision="f64", rows=None):
    from paper_1902_02999_gb300 import Simulation
    sim = Simulation.from_case(case, precision=precision)
    sim.set_step_kernel(kernel)
    if rows:
        sim.set_tile_rows(rows)
    return sim


@pytest.mark.parametrize("nx,ny", [(131, 97), (31, 40), (517, 61)])
@pytest.mark.parametrize("edges", EDGES)
def test_strip_and_march_equal_tile(nx, ny, edges):
    rows = ny >= 8 and PERIODIC not in edges[2:]
    case = inputs.random_case(nx, ny, 5 + nx, edges=edges, dirichlet_sn=rows)
    out = []
    for kernel in ("tile", "strip", "march"):
        sim = sim_of(case, kernel)
        sim.step(60)
        out.append(sim.get_state())
        sim.close()
    for other in out[1:]:
        for a, b in zip(out[0], other):
            assert np.array_equal(a, b)


def test_strip_against_oracle():
    case = inputs.random_case(131, 97, 1)
    sim = sim_of(case, "strip")
    sim.step(300)
    compare(case, sim.get_state(), oracle.run(case, 300), "f64", "strip")


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("rows", [1, 3, 8, 1000])
def test_rows_per_strip(rows, precision):
    case = inputs.random_case(131, 50, 9)
    ref, sim = sim_of(case, "tile", precision), sim_of(case, "strip", precision, rows)
    for s in (ref, sim):
        s.step(50)
    for a, b in zip(ref.get_state(), sim.get_state()):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_several_steps_tidal_strip_speeds(precision):
    """u and v of the strip after several-step launches, against the oracle at
    the parity tolerances (FP64: against max(speed, g h / e), as there)."""
    case = inputs.tidal_strip(201, 3)
    from paper_1902_02999_gb300 import Simulation
    sim = Simulation.from_case(case, precision=precision)
    sim.step(301)
    compare(case, sim.get_state(), oracle.run(case, 301), precision, "several steps", conditioned=True)
