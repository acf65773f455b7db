"""Simulation.device_state: views of the handle's own buffers that carry
nothing over from the call before (autograd modes, history, writes)."""
import numpy as np
import pytest

import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("n", [64, 37])
def test_views_follow_the_state(precision, n):
    from paper_1902_02999_gb300 import Simulation
    case = inputs.dish_lake(n, seed=2)
    sim = Simulation.from_case(case, precision=precision)
    for steps in (0, 1, 2, 9, 1):
        sim.step(steps)
        eta, u, v = sim.device_state()
        want = sim.get_state()
        assert eta.shape == (n, n) and eta.device.index == sim.device and not eta.requires_grad
        assert eta.stride() == (sim.info["pitch"], 1)
        assert np.array_equal(u.double().cpu().numpy(), want[1]) and np.array_equal(v.double().cpu().numpy(), want[2])
    eta.fill_(0.125)  # writes reach the handle
    live = case.mask != inputs.SOLID
    assert np.array_equal(sim.get_state()[0][live], (case.h_ref - case.zb + 0.125)[live])


def test_nothing_carried_between_calls():
    from paper_1902_02999_gb300 import Simulation
    sim = Simulation.from_case(inputs.dish_lake(40, seed=3), precision="f64")
    with torch.inference_mode():
        first = sim.device_state()
        sim.step(1)
        first = sim.device_state()
    w = torch.ones(40, 40, dtype=torch.float64, device="cuda", requires_grad=True)
    eta, u, v = sim.device_state()
    assert not any(t.is_inference() for t in (eta, u, v)) and eta.data_ptr() == first[0].data_ptr()
    (eta * w).sum().backward()                # saved for backward
    assert torch.equal(w.grad, eta)
    u.add_(1.0)                               # in-place work outside inference mode
    v.copy_(w)                                # history stays with this tensor
    assert v.requires_grad
    assert not any(t.requires_grad for t in sim.device_state())
