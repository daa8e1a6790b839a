"""Vertex finding recomputed from the GPU's own tracks: order, cuts and track assignment
must agree exactly (the cut is a float32 step), on events whose tracks spread over the z
buckets of the sort, crowd into a few of them (the bitonic sort) or are very few, and with
cuts that make one group of all tracks or none.  z within the rounding of a float32 sum in
any order, n 2^-24 of the sum of magnitudes, and the same for the sum of pT^2."""

import dataclasses

import numpy as np
import pytest

import sim

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2501_05520_gb300 as pt  # noqa: E402

CAP = pt.default_capacity(max_events=8, hits_per_event=32768, cells_per_event=2 << 20,
                          links_per_event=1 << 18, ntuplets_per_event=1 << 17)


def _event(z0_sigma, n, seed):
    return sim.generate(dataclasses.replace(sim.PU50, z0_sigma=z0_sigma), seed, n_particles=n)


@pytest.mark.parametrize("min_hits,dz", [(4, 0.02), (3, 0.02), (4, 50.0), (4, 1e-9)])
def test_vertices_of_the_tracks(cuts, min_hits, dz):
    events = [_event(5.0, 2500, 7300), _event(0.001, 2500, 7301), _event(0.2, 1200, 7302),
              _event(5.0, 1, 7303), _event(5.0, 40, 7304), sim.vertex_event(7305, 60)]
    with pt.Context(cuts=cuts, capacity=CAP) as ctx:
        ctx.pt_reconstruct_batch(*sim.concat(events))
        n = ctx.pt_find_vertices(min_hits=min_hits, dz=dz)
        v, off, tv = ctx.pt_get_vertices()
        tracks = ctx.pt_get_tracks()
        _, _, tr_off = ctx.pt_get_ntuplets()
    assert n == len(v) == off[-1] and off[0] == 0 and len(tv) == len(tracks)
    want = np.full(len(tracks), -1, np.int64)
    nv = 0
    for e in range(len(events)):
        t = tracks[tr_off[e]:tr_off[e + 1]]
        use = np.nonzero((t["nhits"] >= min_hits) & np.isfinite(t["z0"]))[0]
        order = use[np.lexsort((use, t["z0"][use]))]
        z = t["z0"][order]
        cut = np.nonzero(z[1:] - z[:-1] > np.float32(dz))[0] + 1
        for g in np.split(order, cut):
            if len(g) < 2:
                continue
            want[tr_off[e] + g] = nv
            assert v["n_tracks"][nv] == len(g) and v["event"][nv] == e
            z64, p2 = t["z0"][g].astype(np.float64), t["pt"][g].astype(np.float64) ** 2
            assert abs(v["z"][nv] - z64.mean()) <= (len(g) + 2) * 2.0**-24 * np.abs(z64).mean()
            assert abs(v["sum_pt2"][nv] - p2.sum()) <= (len(g) + 2) * 2.0**-24 * p2.sum()
            nv += 1
        assert off[e + 1] == nv
    assert np.array_equal(tv, want)
