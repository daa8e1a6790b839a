"""Vertices of batches on both sides of the number of events whose counts each block adds up
itself (2048; larger batches scan them), with events on both sides of the bucket counts of the
sort (256 tracks per 1024 buckets).  A batch of copies gives every copy the vertices that its
event has alone, counted on from the events before it."""

import numpy as np
import pytest

import sim

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2501_05520_gb300 as pt  # noqa: E402

CUT = dict(min_hits=3, dz=0.05)


def _vertices(ctx, batch):
    ctx.pt_reconstruct_batch(*batch)
    n = ctx.pt_find_vertices(**CUT)
    v, off, tv = ctx.pt_get_vertices()
    assert n == len(v) == off[-1] and off[0] == 0
    return v, off, tv, ctx.pt_get_ntuplets()[2]


def _capacity(events, hits):
    return pt.default_capacity(max_events=events, hits_per_event=hits, cells_per_event=16 * hits,
                               links_per_event=16 * hits, ntuplets_per_event=4 * hits, phi_bins=64)


def _check_copies(cuts, distinct, n_events):
    alone = []
    with pt.Context(cuts=cuts, capacity=_capacity(1, 16384)) as ctx:
        for ev in distinct:
            v, _, tv, toff = _vertices(ctx, sim.concat([ev]))
            alone.append((v.copy(), tv.copy(), int(toff[-1])))
    hits = max(ev.n_hits for ev in distinct)
    with pt.Context(cuts=cuts, capacity=_capacity(n_events, hits)) as ctx:
        v, off, tv, toff = _vertices(
            ctx, sim.concat([distinct[i % len(distinct)] for i in range(n_events)]))
    counts = [len(alone[i % len(distinct)][0]) for i in range(n_events)]
    assert np.array_equal(off, np.concatenate([[0], np.cumsum(counts)])) and off[-1] > 0
    for i in range(n_events):
        av, atv, nt = alone[i % len(distinct)]
        got = v[off[i]:off[i + 1]]
        assert np.array_equal(got["z"], av["z"]) and np.array_equal(got["sum_pt2"], av["sum_pt2"])
        assert np.array_equal(got["n_tracks"], av["n_tracks"]) and np.all(got["event"] == i)
        assert toff[i + 1] - toff[i] == nt
        assert np.array_equal(tv[toff[i]:toff[i + 1]], np.where(atv >= 0, atv + off[i], -1))


@pytest.mark.parametrize("n_events", [1, 150, 1300, 2048, 2049, 5000])
def test_small_events(cuts, n_events):
    _check_copies(cuts, [sim.generate(sim.SINGLE_MUON_LIKE, 7400 + i, n_particles=n)
                         for i, n in enumerate((30, 2, 12))], n_events)


def test_sizes_around_the_bucket_counts(cuts):
    _check_copies(cuts, [sim.generate(sim.PU50, 7410 + i, n_particles=n)
                         for i, n in enumerate((150, 250, 400, 700, 1200))], 10)
