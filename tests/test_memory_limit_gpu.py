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
    """torch's memory up to `limit` bytes in all; `peak` is the most held."""

    limit = None
    peak = 0

    def __init__(self, device, stream):
        super().__init__(device, stream)
        cls, give, take, held = type(self), self._alloc, self._release, {}

        def alloc(nbytes, ctx):
            if cls.limit is not None and sum(held.values()) + nbytes > cls.limit:
                return None
            p = give(nbytes, ctx)
            if p:
                held[p] = nbytes
                cls.peak = max(cls.peak, sum(held.values()))
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
    Allocator.limit, Allocator.peak = None, 0
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
            allocator.limit = peak - 1   # one request is refused
        sim = maclab.Simulation.from_case(case, precision=precision)
        peak = allocator.peak            # (of the creation)
        for n in (1, 20, 70):
            sim.step(n)
        out.append((sim.get_state(), sim.residual(), sim.info["device_bytes"]))
        sim.mark()     # still fits
        sim.close()
    for a, b in zip(out[0][0], out[1][0]):
        assert np.array_equal(a, b)
    assert out[0][1] == out[1][1] and out[1][2] < out[0][2]


@pytest.mark.parametrize("precision,persistent", [("f32", 0), ("f64", 0), ("f64", 1)])
@pytest.mark.parametrize("big", [False, True])
def test_batch_without_its_options(allocator, precision, persistent, big):
    """Several-step path, row march (FP32) and stencils of the depth (FP64)."""
    cases = [inputs.dish_lake(50, seed=1), inputs.bump_channel(130, 40, seed=2),
             inputs.random_case(97, 51, 11, edges=(inputs.SPECULAR,) * 4, dirichlet=False),
             inputs.random_case(66, 35, 12, edges=(inputs.PERIODIC,) * 4)]
    if big:
        cases += [inputs.dish_lake(450, seed=i) for i in range(12)]
    out = []
    for limited in (False, True):
        if limited:
            allocator.limit = peak - 1
        batch = maclab.Batch(cases, precision=precision)
        peak = allocator.peak            # (of the creation)
        batch.set_persistent(persistent)
        for n in (1, 20, 70):
            batch.step(n)
        batch.mark()   # still fits
        out.append([batch.get_state(i) for i in range(len(cases))])
        batch.close()
    for a, b in zip(*out):
        for x, y in zip(a, b):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("kernel", ["tile", "strip", "march"])
@pytest.mark.parametrize("nx,ny,edges", [(512, 1024, (inputs.PERIODIC,) * 4), (1001, 701, (inputs.SPECULAR,) * 4),
                                         (30001, 3, (inputs.PERIODIC, inputs.PERIODIC, inputs.SPECULAR, inputs.SPECULAR)),
                                         (37, 300, (inputs.BOUNCEBACK,) * 4)])
def test_fp64_grid_fits_where_it_did(allocator, nx, ny, edges, kernel):
    """Memory for two states, two arrays of depths, types, three doubles a
    node for transfers (and a little for lists) holds the handle, without the
    stencils of the depth; with a marked state's size on top also that; and
    with the distributions' size the distribution form."""
    solids = edges[0] == inputs.BOUNCEBACK
    case = inputs.random_case(nx, ny, 3, edges=edges, solids=solids, dirichlet=False)
    padded = (nx + 63) // 64 * 64 * ny
    former = 65 * padded + 24 * nx * ny + (1 << 19)
    limits = [None, former, former + 24 * padded] + ([] if solids else [former + 144 * padded])
    out, size = [], []
    for limit in limits:
        allocator.limit = limit
        sim = maclab.Simulation.from_case(case, precision="f64")
        sim.set_step_kernel(kernel)
        size.append(sim.info["device_bytes"])
        sim.step(5)
        out.append(list(sim.get_state()))
        if limit == former + 24 * padded:
            sim.mark()
        if not solids and limit in (None, former + 144 * padded):
            sim.set_relaxation(0.8)
            sim.step(4)
            out[-1] += sim.get_state()
            sim.set_relaxation(1.0)
            sim.step(3)
            out[-1] += sim.get_state()
        sim.close()
    for other in out[1:]:
        for a, b in zip(out[0], other):   # (as many as both have)
            assert np.array_equal(a, b)
    assert size[1] <= former < size[0] or padded < 20000
