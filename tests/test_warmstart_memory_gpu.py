"""The network at the memory limit: the rectified activation copies are
optional, and the layers that would read them rectify as they stage."""
import numpy as np
import pytest

from test_warmstart_gpu import make, random_setup, rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

C, DIL, BATCH = 128, (1, 2, 4, 8, 1, 2, 4, 8, 1, 2, 4, 8), 192
COPIES = (len(DIL) + 1) * BATCH * 64 * 64 * C * 2


def test_without_rectified_copies():
    theta, out, filler = None, [], None
    dev = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")  # noqa: E731
    for limited in (False, True):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        before = torch.cuda.mem_get_info()[0]
        if limited:  # leave room for the network without the copies and 0.7 GB
            filler = torch.empty(before - (used - COPIES) - 700 * (1 << 20), dtype=torch.uint8, device="cuda")
        net = make(C, DIL, BATCH)
        if not limited:
            used = before - torch.cuda.mem_get_info()[0]
            assert used > 2 * COPIES
            theta, X, T, w = random_setup(net, C, DIL, 2, 5)
        net.set_params(theta)
        y = net.forward(dev(X)).cpu().numpy()
        loss, grad = net.gradients(dev(X), dev(T), dev(w))
        out.append((y, grad, loss))
        net.close()
        del filler
        filler = None
    torch.cuda.empty_cache()
    assert rel(out[1][0], out[0][0]) <= 1e-2, rel(out[1][0], out[0][0])
    assert rel(out[1][1], out[0][1]) <= 2e-2, rel(out[1][1], out[0][1])
    assert abs(out[1][2] - out[0][2]) <= 1e-2 * abs(out[0][2])
