"""Simulation.device_state on the CPU: every call makes its own tensors and
names the handle's GPU, whatever device is current."""
import types

import pytest

torch = pytest.importorskip("torch")

import paper_1902_02999_gb300 as maclab  # noqa: E402


class FakeLibrary:
    """Two buffers per quantity, the current one swapped by step()."""

    def __init__(self):
        self.cur = 0

    def maclab_device_state(self, handle, *out):
        for q, p in enumerate(out):
            p._obj.value = 4096 * (1 + q + 3 * self.cur)
        return 0


@pytest.mark.parametrize("precision,size", [("f32", 4), ("f64", 8)])
def test_names_its_device_and_keeps_nothing(monkeypatch, precision, size):
    calls = []

    def as_tensor(data, device=None):
        calls.append((data.__cuda_array_interface__, device))
        return types.SimpleNamespace(number=len(calls))

    monkeypatch.setattr(torch, "as_tensor", as_tensor)
    sim = maclab.Simulation.__new__(maclab.Simulation)
    sim._lib, sim._h = FakeLibrary(), 1
    sim.nx, sim.ny, sim.device, sim.precision, sim.info = 70, 5, 1, precision, {"pitch": 128}
    seen = []
    for cur in (0, 1, 0, 0):
        sim._lib.cur = cur
        seen += [t.number for t in sim.device_state()]
    sim._h = None
    assert seen == list(range(1, 13))                      # no tensor handed out twice
    for k, (array, device) in enumerate(calls):
        assert torch.device(device) == torch.device("cuda", 1)
        assert array["data"] == (4096 * (1 + k % 3 + 3 * (0, 1, 0, 0)[k // 3]), False)
        assert array["shape"] == (5, 70) and array["strides"] == (128 * size, size)
