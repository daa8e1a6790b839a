"""The binning kernel's tiles of 256 hits: events that end on, before and after a tile's edge,
several of them inside one tile, and empty ones.  The per-layer ranges that it gathers decide
which windows the searches look at, so each event's tracks are compared with the oracle's."""

import numpy as np
import pytest

import oracle
import sim

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2501_05520_gb300 as pt  # noqa: E402


@pytest.mark.parametrize("sizes", [
    (1,), (255,), (256,), (257,),
    (0, 256, 0, 1, 255, 0, 512, 7, 0),
    (100, 60, 40, 30, 20, 3, 2, 1, 0, 500),
    (767, 257, 1, 1023, 0, 300),
    (4000, 96, 2048, 1500),
])
@pytest.mark.parametrize("where", ["host", "device"])
def test_event_edges(cuts, sizes, where):
    rng = np.random.default_rng(sum(sizes) + 31)
    parts, refs = [], []
    for i, n in enumerate(sizes):
        ev = sim.generate(sim.PU50, 4100 + i, n_particles=max(60, n // 3))
        keep = np.sort(rng.permutation(len(ev.x))[:n])
        assert len(keep) == n
        a = [v[keep] for v in (ev.x, ev.y, ev.z, ev.layer)]
        parts.append(a)
        refs.append(oracle.survivors_hits(oracle.reconstruct(*a, cuts)) if n else
                    np.zeros((0, 6), np.int32))
    off = np.cumsum([0, *sizes]).astype(np.int32)
    arrays = [np.concatenate(c) for c in zip(*parts)]
    if where == "device":
        arrays = [torch.from_numpy(a).cuda() for a in arrays]
    cap = pt.default_capacity(max_events=16, hits_per_event=4096, cells_per_event=1 << 17,
                              links_per_event=1 << 16, ntuplets_per_event=1 << 15)
    with pt.Context(cuts=cuts, capacity=cap) as ctx:
        ctx.pt_reconstruct_batch(off, *arrays)
        hits, _, o = ctx.pt_get_ntuplets()
    assert np.array_equal(o, np.cumsum([0] + [len(r) for r in refs]))
    assert np.array_equal(hits, np.concatenate(refs))
