"""Duplicate cleaning where ntuplets tie in hit count and quality: events whose hits come in
exact copies (two and three of them on some layers), so that chains through the copies have
equal q and share cells and the smaller hit tuple decides.  The whole-batch graph and the
stage calls against the oracle, plain and with the fishbone step, and after one another."""

import numpy as np
import pytest

import oracle
import sim
from test_gpu_parity import run_stages

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2501_05520_gb300 as pt  # noqa: E402

CAP = pt.default_capacity(max_events=3, hits_per_event=16384, cells_per_event=1 << 20,
                          links_per_event=1 << 17, ntuplets_per_event=1 << 17)


class Copied:
    """An event with every hit of the given layers repeated, in a random order."""

    def __init__(self, cfg, seed, copies, n=None):
        ev = sim.generate(cfg, seed, n_particles=n)
        rng = np.random.default_rng(seed)
        idx = np.repeat(np.arange(ev.n_hits), [copies.get(int(v), 1) for v in ev.layer])
        idx = rng.permutation(idx)
        self.x, self.y, self.z, self.layer = (a[idx] for a in (ev.x, ev.y, ev.z, ev.layer))
        self.n_hits = int(idx.size)


@pytest.mark.parametrize("copies", [{1: 2}, {0: 2, 3: 2}, {2: 3}, {0: 3, 1: 2, 2: 2, 4: 2}])
@pytest.mark.parametrize("fishbone", [False, True])
def test_copied_hits(cuts, copies, fishbone):
    events = [Copied(sim.SINGLE_MUON_LIKE, 1200, copies), Copied(sim.PU50, 2250, copies, 600),
              Copied(sim.SINGLE_MUON_LIKE, 1201, copies)]
    ref = [oracle.survivors_hits(oracle.reconstruct(e.x, e.y, e.z, e.layer, cuts,
                                                    fishbone=fishbone)) for e in events]
    want = np.concatenate(ref)
    off = np.cumsum([0] + [len(r) for r in ref])
    with pt.Context(cuts=cuts, capacity=CAP) as ctx:
        ctx.pt_set_fishbone(fishbone)
        for _ in range(3):  # the tied ntuplets come in another order each time
            hits, _, _, evoff = ctx.pt_reconstruct_batch(*sim.concat(events))
            assert np.array_equal(evoff, off) and np.array_equal(hits, want)
        run_stages(ctx, events)
        hits, _, evoff = ctx.pt_get_ntuplets()
        assert np.array_equal(evoff, off) and np.array_equal(hits, want)
        ctx.pt_find_ntuplets()  # again on the same links
        assert np.array_equal(ctx.pt_get_ntuplets()[0], want)
