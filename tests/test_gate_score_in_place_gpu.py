"""Standalone gate scoring into memory that its own feature rows occupy: scores as with arrays of
their own, whichever part of the rows they replace; the rest of the memory is left alone."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2501_05520_gb300 as pt  # noqa: E402

ROWS = 300_001


@pytest.mark.parametrize("n,start", [(1, 0), (129, 0), (129, 12 * 128), (ROWS, 0), (ROWS, 5),
                                     (ROWS, 6 * ROWS), (ROWS, 12 * ROWS - 1), (ROWS, 12 * ROWS)])
def test_scores_over_rows(n, start):
    """start: of the scores, in floats from the first row (the last case shares nothing)."""
    rng = np.random.default_rng(5)
    rows = torch.from_numpy(rng.normal(size=(n, 12)).astype(np.float32)).cuda()
    memory = torch.zeros(13 * n, device="cuda")
    memory[:12 * n] = rows.view(-1)
    want = torch.empty(n, device="cuda")
    cap = pt.default_capacity(max_events=1, links_per_event=ROWS)
    with pt.Context(capacity=cap) as ctx:
        ctx.pt_set_gate(*pt.default_gate())
        torch.cuda.synchronize()
        ctx.pt_gate_score(rows, want)
        ctx.pt_gate_score(memory[:12 * n].view(n, 12), memory[start:start + n])
    assert torch.equal(memory[start:start + n], want)
    rest = torch.cat([memory[:start], memory[start + n:]])
    before = torch.cat([rows.view(-1), torch.zeros(n, device="cuda")])
    assert torch.equal(rest, torch.cat([before[:start], before[start + n:]]))
