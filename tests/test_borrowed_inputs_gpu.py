"""Inputs are borrowed for the duration of a call: a caller may overwrite them as soon as an
asynchronous call has returned, from another stream or from the host, whatever is still queued on
the context's stream."""

import numpy as np
import pytest

import oracle
import sim

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2501_05520_gb300 as pt  # noqa: E402

QUEUED = 20_000_000  # clock cycles of work ahead of the call, about 10 ms


@pytest.mark.parametrize("where", ["device", "pinned", "numpy"])
@pytest.mark.parametrize("call", ["hits", "batch", "enqueue"])
@pytest.mark.parametrize("particles", [300, 1200])  # up to and beyond the inputs sent in one copy
def test_overwritten_on_return(cuts, call, where, particles):
    ev = sim.generate(sim.PU50, 2340, n_particles=particles)
    want = oracle.survivors_hits(oracle.reconstruct(ev.x, ev.y, ev.z, ev.layer, cuts))
    off, *arrays = sim.concat([ev])
    assert (arrays[0].size <= 4096) == (particles == 300) and len(want) > 100
    if where == "numpy":
        data = [a.copy() for a in arrays]
    else:
        data = [torch.from_numpy(a.copy()) for a in arrays]
        data = [t.cuda() if where == "device" else t.pin_memory() for t in data]
    cap = pt.default_capacity(max_events=1, hits_per_event=16384, cells_per_event=1 << 20,
                              links_per_event=1 << 17, ntuplets_per_event=1 << 16)
    stream, other = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with pt.Context(cuts=cuts, capacity=cap, stream=stream) as ctx:
        ctx.pt_reconstruct_batch(off, *arrays)  # the graph exists from here on
        with torch.cuda.stream(stream):
            torch.cuda._sleep(QUEUED)
        if call == "hits":
            ctx.pt_load_hits(*data)
        else:
            (ctx.pt_load_batch if call == "batch" else ctx.pt_enqueue_batch)(off, *data)
        with torch.cuda.stream(other):
            for a in data:
                a.fill(0) if where == "numpy" else a.zero_()
        other.synchronize()
        if call != "enqueue":
            ctx.pt_build_doublets()
            ctx.pt_connect_cells()
            ctx.pt_find_ntuplets()
        assert np.array_equal(ctx.pt_get_ntuplets()[0], want)
