"""Device memory at its limit: what the faster paths hold on top is optional.
A handle or batch is created without it, steps on the next path and gives the
same results."""
import numpy as np
import pytest

import inputs
import paper_1902_02999_gb300 as maclab

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class Allocator(maclab._TorchAllocator):
    """torch's memory up to `limit` bytes in all; `log` keeps the sizes given."""

    limit = None
    log: list = []

    def __init__(self, device, stream):
        super().__init__(device, stream)
        cls, give, take, held = type(self), self._alloc, self._release, {}

        def alloc(nbytes, ctx):
            if cls.limit is not None and sum(held.values()) + nbytes > cls.limit:
                return None
            p = give(nbytes, ctx)
            if p:
                held[p] = nbytes
                cls.log.append(nbytes)
            return p

        def release(p, ctx):
            held.pop(p, None)
            take(p, ctx)

        self._keep = (give, take)
        self._alloc = maclab._abi.ALLOC_FN(alloc)
        self._release = maclab._abi.RELEASE_FN(release)
        self.struct = maclab._abi.Allocator(self._alloc, self._release, None)


@pytest.fixture
def allocator(monkeypatch):
    monkeypatch.setattr(maclab, "_TorchAllocator", Allocator)
    Allocator.limit, Allocator.log = None, []
    yield Allocator
    Allocator.limit = None


HANDLES = [
    (lambda: inputs.dish_lake(128, seed=1), "f32"),
    (lambda: inputs.dish_lake(128, seed=1), "f64"),
    (lambda: inputs.bump_channel(640, 200, seed=1), "f32"),
    (lambda: inputs.tidal_strip(201, 3), "f64"),
]


@pytest.mark.parametrize("make,precision", HANDLES)
def test_handle_without_the_window_path(allocator, make, precision):
    case, out = make(), []
    for limited in (False, True):
        if limited:
            allocator.limit = sum(allocator.log) - 1   # the last request is refused
        sim = maclab.Simulation.from_case(case, precision=precision)
        for n in (1, 20, 70):
            sim.step(n)
        out.append((sim.get_state(), sim.residual(), sim.info["device_bytes"]))
        sim.close()
    for a, b in zip(out[0][0], out[1][0]):
        assert np.array_equal(a, b)
    assert out[0][1] == out[1][1] and out[1][2] < out[0][2]


@pytest.mark.parametrize("precision,big", [("f32", False), ("f64", False), ("f32", True)])
def test_batch_without_window_or_march(allocator, precision, big):
    cases = [inputs.dish_lake(50, seed=1), inputs.bump_channel(130, 40, seed=2)]
    if big:
        cases += [inputs.dish_lake(450, seed=i) for i in range(12)]
    out = []
    for limited in (False, True):
        if limited:
            allocator.limit = sum(allocator.log) - 1
        batch = maclab.Batch(cases, precision=precision)
        for n in (1, 20, 70):
            batch.step(n)
        out.append([batch.get_state(i) for i in range(len(cases))])
        batch.close()
    for a, b in zip(*out):
        for x, y in zip(a, b):
            assert np.array_equal(x, y)
