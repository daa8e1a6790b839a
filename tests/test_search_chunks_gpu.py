"""The doublet and link searches hand out chunks of 1 to 8 sorted hits depending on the
batch's hits and the warps of the launch.  Batches on both sides of the chunk sizes (one
event, and thousands of copies of a few events) give every event its oracle ntuplets, and
the cell and link slots keep no hole inside a small event."""

import numpy as np
import pytest

import oracle
import sim

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2501_05520_gb300 as pt  # noqa: E402

DISTINCT = 5


@pytest.fixture(scope="module")
def events(cuts):
    ev = [sim.generate(sim.SINGLE_MUON_LIKE, 1100 + i) for i in range(DISTINCT)]
    return ev, [oracle.survivors_hits(oracle.reconstruct(e.x, e.y, e.z, e.layer, cuts)) for e in ev]


# 1216 warps with one search block per SM, 4864 in the link search: 200-hit events cross
# two hits a chunk at 195 (doublets) and 779 (links) events, eight at 779 and 3114
@pytest.mark.parametrize("n_events,blocks", [(1, 5), (1, 1), (190, 1), (400, 1), (790, 1), (3300, 1),
                                             (3300, 8)])
def test_every_event_of_a_batch(cuts, events, n_events, blocks):
    ev, ref = events
    batch = [ev[i % DISTINCT] for i in range(n_events)]
    off, x, y, z, layer = sim.concat(batch)
    cap = pt.default_capacity(max_events=n_events, hits_per_event=256, cells_per_event=1024,
                              links_per_event=1024, ntuplets_per_event=512, phi_bins=64)
    with pt.Context(cuts=cuts, capacity=cap) as ctx:
        ctx.pt_set_launch(4, blocks)
        hits, _, _, evoff = ctx.pt_reconstruct_batch(off, x, y, z, layer)
        want = np.concatenate([ref[i % DISTINCT] for i in range(n_events)])
        sizes = [len(ref[i % DISTINCT]) for i in range(n_events)]
        assert np.array_equal(evoff, np.concatenate([[0], np.cumsum(sizes)]))
        assert np.array_equal(hits, want)
