"""A context's workspace does not outgrow the sizes that callers have reserved: pt_workspace_size
for capacities where one kind of array dominates, against the bytes that a caller's fixed block
held when it was laid out.  And a small batch, whose inputs pass through the workspace's place for
the sorted hits, can run through the chain more than once (pt_autotune)."""

import pytest

import paper_2501_05520_gb300 as pt
from paper_2501_05520_gb300 import build as pkg_build


@pytest.mark.parametrize("events,hits,cells,links,ntuplets,phi,room", [
    (8, 4096, 1024, 512, 512, 64, 663296),
    (1, 1, 1, 1, 1, 16, 29696),
    (1, 4096, 64, 64, 64, 16, 488448),
    (64, 4000, 100, 50, 50, 1024, 5734912),
    (2, 65536, 4096, 1024, 1024, 256, 7619328),
])
def test_fits_a_reserved_block(events, hits, cells, links, ntuplets, phi, room):
    pkg_build.build()
    cap = dict(pt.default_capacity(), max_events=events, max_hits=hits, max_cells=cells,
               max_links=links, max_ntuplets=ntuplets, phi_bins=phi)
    assert pt.pt_workspace_size(cap) <= room


@pytest.mark.gpu
@pytest.mark.parametrize("particles", [50, 900])
def test_small_batch_runs_again(cuts, particles):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import sim
    ev = sim.generate(sim.PU50, 2360, n_particles=particles)
    assert ev.n_hits <= 4096
    cap = pt.default_capacity(max_events=1, hits_per_event=4096, cells_per_event=1 << 19,
                              links_per_event=1 << 16, ntuplets_per_event=1 << 15)
    r = pt.pt_autotune([0, ev.n_hits], ev.x, ev.y, ev.z, ev.layer, cap, (256,), (4,), (4, 5),
                       reps=3, cuts=cuts)
    assert all(ms > 0 for ms in r["table"].values())
