"""Whole-batch calls with their inputs and outputs in every kind of memory: a small batch's
inputs go up with the header and its results come back in the pinned block, larger ones are
copied, device arrays are read and written in place (wherever they start).  All routes give
the same results, and an output that is too small is not written."""

import numpy as np
import pytest

import oracle
import sim

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2501_05520_gb300 as pt  # noqa: E402


def _batch(which, cuts):
    if which == "small":  # up to 4096 hits and tracks
        ev = [sim.generate(sim.SINGLE_MUON_LIKE, 1300 + i) for i in range(3)]
    elif which == "hits":  # more hits, few tracks
        ev = [sim.generate(sim.PU50, 2300, n_particles=1100)]
    else:  # more hits and tracks
        ev = [sim.generate(sim.PU50, 2301 + i) for i in range(3)]
    refs = [oracle.survivors_hits(oracle.reconstruct(e.x, e.y, e.z, e.layer, cuts)) for e in ev]
    return sim.concat(ev), np.concatenate(refs), np.cumsum([0] + [len(r) for r in refs])


def _outputs(n, e, where, shift):
    kw = dict(device="cuda") if where == "device" else dict(pin_memory=where == "pinned")

    def new(count, dtype):
        return torch.zeros(count + shift, dtype=dtype, **kw)[shift:]

    return dict(hits=new(n * 6, torch.int32).view(n, 6), nhits=new(n, torch.uint8),
                tracks=new(n * 9, torch.float32).view(n, 9), event_offsets=new(e + 1, torch.int64))


@pytest.mark.parametrize("which", ["small", "hits", "tracks"])
def test_routes(cuts, which):
    (off, *arrays), want, want_off = _batch(which, cuts)
    S, E = len(want), len(off) - 1
    cap = pt.default_capacity(max_events=4, hits_per_event=16384, cells_per_event=1 << 20,
                              links_per_event=1 << 17, ntuplets_per_event=1 << 16)
    inputs = {
        "numpy": arrays,
        "pinned": [torch.from_numpy(a).pin_memory() for a in arrays],
        "device": [torch.from_numpy(a).cuda() for a in arrays],
        "shifted": [torch.cat([torch.zeros(1, dtype=torch.from_numpy(a).dtype),
                               torch.from_numpy(a)]).cuda()[1:] for a in arrays],
    }
    tracks = None
    with pt.Context(cuts=cuts, capacity=cap) as ctx:
        for name, a in inputs.items():
            for where in ("host", "pinned", "device"):
                for n in (S, S + 100):
                    out = _outputs(n, E, where, 1 if name == "shifted" else 0)
                    ctx.pt_reconstruct_batch(off, *a, out=out)
                    assert np.array_equal(out["hits"][:S].cpu().numpy(), want), (name, where)
                    assert np.array_equal(out["event_offsets"].cpu().numpy(), want_off)
                    assert np.array_equal(out["nhits"][:S].cpu().numpy(), (want >= 0).sum(1))
                    t = out["tracks"][:S].cpu().numpy()
                    tracks = t if tracks is None else tracks
                    assert np.array_equal(t.view(np.uint32), tracks.view(np.uint32))
                    assert not out["nhits"][S:].any() and not out["hits"][S:].any()
                out = _outputs(S - 1, E, where, 0)
                with pytest.raises(pt.PtError) as err:
                    ctx.pt_reconstruct_batch(off, *a, out=out)
                assert err.value.status == pt.PT_ERR_CAPACITY
                assert not any(out[k].any() for k in ("hits", "nhits", "event_offsets"))
                # what the getters give does not depend on where the results went
                hits, _, o = ctx.pt_get_ntuplets()
                assert np.array_equal(hits, want) and np.array_equal(o, want_off)
                assert np.array_equal(ctx.pt_get_tracks().view(np.uint32).reshape(S, 9),
                                      tracks.view(np.uint32))
                x, y, z, layer, o = ctx.pt_get_hits()
                for got, exp in zip((x, y, z, layer, o), (*arrays, off)):
                    assert np.array_equal(got, exp)
        # a stage call after a whole-batch call leaves the caller's arrays alone
        out = _outputs(S, E, "device", 0)
        ctx.pt_reconstruct_batch(off, *inputs["device"], out=out)
        out["tracks"].zero_()
        ctx.pt_fit_tracks()
        assert not out["tracks"].any()
