"""Gate scoring at the edges of its 128-row tiles and from feature arrays that are not
16-byte aligned: a row's score does not depend on where it lies (bitwise), and matches the
oracle with the gate's score tolerance."""

import numpy as np
import pytest

from oracle import gate as ogate
from test_gate_gpu import SCORE_ATOL, SCORE_RTOL, _weights

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2501_05520_gb300 as pt  # noqa: E402

CAP = dict(max_events=1, max_hits=64, max_cells=64, max_links=200_000, max_ntuplets=64,
           phi_bins=64, reserved=0)


@pytest.mark.parametrize("n", [1, 127, 128, 129, 116_737])
def test_rows(n):
    rng = np.random.default_rng(n)
    X = rng.normal(0, 1, (n, 12)).astype(np.float32)
    w = _weights(6)
    x = torch.from_numpy(X).cuda()
    room = torch.zeros(n * 12 + 3, device="cuda")
    room[1:1 + n * 12] = x.flatten()
    out = [torch.full((n + 4,), 9.0, device="cuda") for _ in range(2)]
    with pt.Context(capacity=CAP) as ctx:
        ctx.pt_set_gate(w, 0.0)
        ctx.pt_gate_score(x, out[0][:n])
        ctx.pt_gate_score(room[1:1 + n * 12].view(n, 12), out[1][:n])
    assert torch.equal(out[0], out[1]) and torch.all(out[0][n:] == 9.0)
    s = ogate.forward(w, X, bf16=True)
    got = out[0][:n].cpu().numpy()
    assert np.all(np.abs(got - s) <= SCORE_ATOL + SCORE_RTOL * np.abs(s))
