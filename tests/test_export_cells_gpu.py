"""Cells of the loaded batch against the oracle, event by event, on batches whose segments hold one
cell or a hundred: one-track events, events of a few tracks, and a pileup event among them, on both
sides of a warp's 32 hits."""

import numpy as np
import pytest

import oracle
import sim

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2501_05520_gb300 as pt  # noqa: E402


@pytest.mark.parametrize("copies", [1, 7, 33, 500])
def test_cells(cuts, copies):
    small = [sim.generate(sim.SINGLE_MUON_LIKE, 2380 + i, n_particles=n)
             for i, n in enumerate((1, 2, 9))]
    large = sim.generate(sim.PU50, 2390, n_particles=900)
    events = small * copies + [large] + small
    refs = {id(e): oracle.reconstruct(e.x, e.y, e.z, e.layer, cuts) for e in small + [large]}
    want = {k: sorted(zip(r["cell_inner"].tolist(), r["cell_outer"].tolist()))
            for k, r in refs.items()}
    cap = pt.default_capacity(max_events=len(events), hits_per_event=256, cells_per_event=1 << 11,
                              links_per_event=1 << 10, ntuplets_per_event=1 << 9, phi_bins=32)
    cap = dict(cap, max_hits=cap["max_hits"] + 8192, max_cells=cap["max_cells"] + (1 << 19))
    with pt.Context(cuts=cuts, capacity=cap) as ctx:
        ctx.pt_load_batch(*sim.concat(events))
        n = ctx.pt_build_doublets()
        inner, outer, event = ctx.pt_get_cells()
    assert n == len(inner) == sum(len(want[id(e)]) for e in events)
    order = np.lexsort((outer, inner, event))
    got = list(zip(inner[order].tolist(), outer[order].tolist()))
    ends = np.searchsorted(event[order], np.arange(len(events) + 1))
    for e, ev in enumerate(events):
        assert got[ends[e]:ends[e + 1]] == want[id(ev)], e
