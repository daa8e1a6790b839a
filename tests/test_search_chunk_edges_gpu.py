"""Batches on both sides of the searches' chunk sizes: a warp first takes hits / (8 x warps) sorted
hits, at least one and at most 32, with 8 warps to a block, as many blocks per multiprocessor as
pt_set_launch says in the doublet search (one here) and four in the link search.  Copies of a few
events of about 200 hits, as many as lie just below and above chunks of 2 and of 32 hits in each
search, give every event its oracle ntuplets; a small event reserves no more cell and link slots
than it has cells and links."""

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
BLOCKS = {"doublets": 1, "links": 4}


@pytest.fixture(scope="module")
def events(cuts):
    ev = [sim.generate(sim.SINGLE_MUON_LIKE, 1120 + i) for i in range(DISTINCT)]
    return ev, [oracle.survivors_hits(oracle.reconstruct(e.x, e.y, e.z, e.layer, cuts)) for e in ev]


def _capacity(n, cells=1024, links=1024):
    return pt.default_capacity(max_events=n, hits_per_event=256, cells_per_event=cells,
                               links_per_event=links, ntuplets_per_event=512, phi_bins=32)


@pytest.mark.parametrize("side", [-1, 1])
@pytest.mark.parametrize("chunk", [2, 32])
@pytest.mark.parametrize("search", ["doublets", "links"])
def test_every_event_around_an_edge(cuts, events, search, chunk, side):
    ev, ref = events
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    edge = chunk * 8 * sms * BLOCKS[search] * 8  # hits
    per_round = sum(e.n_hits for e in ev)
    n = DISTINCT * (edge // per_round + (side > 0))
    off, x, y, z, layer = sim.concat([ev[i % DISTINCT] for i in range(n)])
    assert (len(x) >= edge) == (side > 0) and abs(len(x) - edge) <= per_round
    with pt.Context(cuts=cuts, capacity=_capacity(n)) as ctx:
        ctx.pt_set_launch(4, 1)
        hits, _, _, evoff = ctx.pt_reconstruct_batch(off, x, y, z, layer)
    sizes = [len(ref[i % DISTINCT]) for i in range(n)]
    assert np.array_equal(evoff, np.concatenate([[0], np.cumsum(sizes)]))
    assert np.array_equal(hits, np.concatenate([ref[i % DISTINCT] for i in range(n)]))


def test_a_small_event_needs_no_spare_slots(cuts, events):
    e = events[0][0]
    with pt.Context(cuts=cuts, capacity=_capacity(1)) as ctx:
        ctx.pt_load_batch(*sim.concat([e]))
        cells, links = ctx.pt_build_doublets(), ctx.pt_connect_cells()
    assert cells > 100 and links > 50
    with pt.Context(cuts=cuts, capacity=_capacity(1, cells, links)) as ctx:
        hits, _, _, _ = ctx.pt_reconstruct_batch(*sim.concat([e]))
    assert np.array_equal(hits, events[1][0])
