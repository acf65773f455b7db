"""Calls of a few steps on grids whose window costs more to load than single
steps take: single-step launches, longer calls several steps per launch, both
in any order with the same results."""
import numpy as np
import pytest

import inputs
from inputs import PERIODIC, SPECULAR

from launches import kernels

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make,steps,want", [
    (lambda: inputs.random_case(809, 809, 3, edges=(PERIODIC,) * 4), 1, "step_march_kernel"),
    (lambda: inputs.random_case(809, 809, 3, edges=(PERIODIC,) * 4), 16, "step_window_kernel"),
    (lambda: inputs.random_case(30000, 20, 3, edges=(SPECULAR,) * 4, dirichlet=False), 2, "step_march_kernel"),
    (lambda: inputs.dish_lake(128, seed=1), 1, "step_window_kernel"),
    (lambda: inputs.dish_lake(128, seed=1), 8, "step_window_kernel"),
])
def test_handle_route(make, steps, want):
    from paper_1902_02999_gb300 import Simulation
    stream = torch.cuda.Stream()
    sim = Simulation.from_case(make(), precision="f32", stream=stream)
    names = kernels(lambda: sim.step(steps), stream)
    assert names and all(want in k for k in names), names
    assert len(names) == (steps if want == "step_march_kernel" else len(names)) <= steps
    sim.close()


@pytest.mark.parametrize("steps,want", [(1, "step_batch_kernel"), (16, "step_window_kernel")])
def test_batch_route(steps, want):
    from paper_1902_02999_gb300 import Batch
    stream = torch.cuda.Stream()
    cases = [inputs.random_case(256, 256, 2, edges=(PERIODIC,) * 4, solids=False)] * 4
    batch = Batch(cases, precision="f32", stream=stream)
    names = kernels(lambda: batch.step(steps), stream)
    assert names and any(want in k for k in names), names
    assert not any("window" in k for k in names) or want == "step_window_kernel"
    batch.close()


def test_any_order_of_calls():
    """Short and long calls in turn, residuals between them, graph replay of
    short blocks, against the tile kernel."""
    from paper_1902_02999_gb300 import Batch, Simulation
    case = inputs.random_case(809, 703, 3, edges=(PERIODIC, PERIODIC, SPECULAR, SPECULAR))
    sims = [Simulation.from_case(case, precision="f32") for _ in range(2)]
    sims[1].set_step_kernel("tile")
    sims[0].set_graph_steps(2)
    for n in (1, 17, 1, 2, 33, 3, 1, 1, 64, 5):
        if n == 33:
            sims[0].set_graph_steps(64)
        out = []
        for s in sims:
            s.step(n)
            out.append((s.residual(), s.get_state(), s.time()))
        assert out[0][0] == out[1][0] and out[0][2] == out[1][2]
        for a, b in zip(out[0][1], out[1][1]):
            assert np.array_equal(a, b), n
    cases = [inputs.random_case(256, 256, k, edges=(PERIODIC,) * 4) for k in (1, 2, 3, 4)]
    batch = Batch(cases, precision="f32")
    ref = [Simulation.from_case(c, precision="f32") for c in cases]
    for s in ref:
        s.set_step_kernel("tile")
    for n in (1, 16, 2, 1, 20, 64, 1):
        batch.step(n)
        res = batch.residual()
        for i, s in enumerate(ref):
            s.step(n)
            assert abs(res[i, 0] - s.residual()[0]) <= 1e-12 * res[i, 0]
            for a, b in zip(batch.get_state(i), s.get_state()):
                assert np.array_equal(a, b), (n, i)
