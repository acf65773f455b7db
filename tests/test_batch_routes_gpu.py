"""Which kernel steps an FP32 batch, and that each of them gives what the
instances' own handles give on the tile kernel (bitwise) and the oracle."""
import numpy as np
import pytest

import inputs
import oracle
from inputs import BOUNCEBACK, PERIODIC, SPECULAR

from launches import kernels
from test_parity_gpu import compare
from test_paths_oracle_gpu import steady

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def odd():
    """Small instances of every edge kind, ragged and narrow widths, a width
    of 60 n + 1 (shifted strips), Dirichlet columns."""
    return [
        inputs.bump_channel(241, 70, seed=7),
        inputs.random_case(181, 61, 8, edges=(SPECULAR,) * 4, dirichlet=False),
        inputs.random_case(61, 9, 4, edges=(BOUNCEBACK,) * 4, dirichlet=False),
        inputs.random_case(200, 35, 5, edges=(SPECULAR, SPECULAR, PERIODIC, PERIODIC), dirichlet=False),
        inputs.random_case(150, 47, 9, edges=(PERIODIC,) * 4),
        inputs.random_case(3, 130, 6, edges=(SPECULAR,) * 4, solids=False, dirichlet=False),
        inputs.random_case(130, 50, 10, edges=(PERIODIC, PERIODIC, SPECULAR, SPECULAR), dirichlet=False),
    ]


def lakes(count):
    return [inputs.dish_lake(450 + i % 3, seed=i % 4) for i in range(count)]


def rows_apart():
    """A row of Dirichlet nodes whose strip block holds no other row."""
    return steady(inputs.random_case(97, 17, 11, edges=(SPECULAR,) * 4, dirichlet_sn=True))


def rows_together():
    """Rows of Dirichlet nodes in one strip block with their inward rows."""
    return steady(inputs.random_case(97, 51, 11, edges=(SPECULAR,) * 4, dirichlet_sn=True))


def walled():
    """Dirichlet nodes whose inward node has a bounce-back link."""
    return steady(inputs.random_case(70, 40, 3, edges=(BOUNCEBACK,) * 4))


BATCHES = {
    "march": (lambda: odd() + lakes(12), "step_march_batch_kernel"),
    "rows_together": (lambda: odd() + [rows_together()] + lakes(12), "step_march_batch_kernel"),
    "rows_apart": (lambda: odd() + [rows_apart()] + lakes(12), "step_batch_kernel"),
    "walled": (lambda: odd() + [walled()] + lakes(12), "step_batch_kernel"),
    "narrow": (lambda: odd() + [inputs.random_case(64, 64, 1 + i % 2, edges=(SPECULAR,) * 4, solids=False, dirichlet=False)
                                for i in range(366)], "step_batch_kernel"),
    "million": (lambda: odd() + lakes(2) + [inputs.random_case(256, 256, 2, edges=(PERIODIC,) * 4)] * 8, "step_batch_kernel"),
    "small": (lambda: odd() + [walled()], "step_window_kernel"),
}


@pytest.mark.parametrize("name", sorted(BATCHES))
def test_route_and_results(name):
    from paper_1902_02999_gb300 import Batch, Simulation
    make, want = BATCHES[name]
    cases = make()
    stream = torch.cuda.Stream()
    probe = Batch(cases, precision="f32", stream=stream)
    names = kernels(lambda: probe.step(16), stream)
    assert all(want in k or "batch_dirichlet_kernel" in k or "batch_general_kernel" in k for k in names), names
    assert sum(want in k for k in names) >= 2
    probe.close()
    batch = Batch(cases, precision="f32")
    batch.set_graph_steps(8)
    batch.step(19)
    off = [i % 3 != 1 for i in range(len(cases))]
    batch.set_active(off)
    batch.step(9)
    batch.set_active([1] * len(cases))
    batch.step(1)
    shown = list(range(min(len(cases), 9))) + [len(cases) - 1]
    for i in shown:
        sim = Simulation.from_case(cases[i], precision="f32")
        sim.set_step_kernel("tile")
        sim.step(29 if off[i] else 20)
        for a, b in zip(batch.get_state(i), sim.get_state()):
            assert np.array_equal(a, b), i
        sim.close()


def test_row_march_against_oracle():
    from paper_1902_02999_gb300 import Batch
    cases = odd() + lakes(12)
    batch = Batch(cases, precision="f32")
    batch.step(200)
    for i in list(range(len(odd()))) + [len(cases) - 1]:
        compare(cases[i], batch.get_state(i), oracle.run(cases[i], 200), "f32", ("batch march", i))
