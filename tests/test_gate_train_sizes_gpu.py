"""Loss and gradient of the gate at the edges of the kernel's tiles (32 samples, and more
tiles than blocks) and with a gradient array that is not 16-byte aligned, against float64
backpropagation.  Tolerance: the one of the minibatch test, 1e-4 relative with a floor of
1e-2 of the largest gradient."""

import numpy as np
import pytest

from oracle import gate as ogate
from test_gate_gpu import _weights

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2501_05520_gb300 as pt  # noqa: E402


@pytest.mark.parametrize("n", [1, 31, 32, 33, 4095, 9729, 20001])
@pytest.mark.parametrize("shift", [0, 1])
def test_loss_and_gradient(n, shift):
    rng = np.random.default_rng(n)
    X = rng.normal(0, 1, (n, 12)).astype(np.float32)
    y = (rng.random(n) < 0.3).astype(np.float32)
    w = _weights(5)
    L, G = ogate.loss_and_grad(w.astype(np.float64), X, y)
    room = torch.full((5057 + 8,), 7.0, device="cuda")
    grad = room[shift:shift + 5057]
    loss = torch.full((1,), 3.0, device="cuda")
    for _ in range(2):  # overwritten, not added to
        pt.pt_gate_loss_grad(torch.from_numpy(w).cuda(), torch.from_numpy(X).cuda(),
                             torch.from_numpy(y).cuda(), grad, loss)
    g = grad.cpu().numpy().astype(np.float64)
    assert float(loss.item()) == pytest.approx(L, rel=1e-5)
    assert np.all(np.abs(g - G) <= 1e-4 * np.maximum(np.abs(G), 1e-2 * np.abs(G).max()))
    assert torch.all(room[:shift] == 7.0) and torch.all(room[shift + 5057:] == 7.0)
