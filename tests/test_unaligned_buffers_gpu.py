"""Device arrays at odd byte addresses: a copy takes any address, a kernel's load or store of a
float does not, so such inputs and outputs go through copies.  The arrays are raw pointers of the
C interface, shifted by 1 to 7 bytes."""

import ctypes

import numpy as np
import pytest

import oracle
import sim

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2501_05520_gb300 as pt  # noqa: E402


def _device(data, shift):
    """A device copy of the array's bytes at an address of `shift` modulo 256."""
    raw = torch.zeros(data.nbytes + 256 + shift, dtype=torch.uint8, device="cuda")
    start = -raw.data_ptr() % 256 + shift
    raw[start:start + data.nbytes] = torch.from_numpy(data.view(np.uint8).copy()).cuda()
    return raw, start, data.nbytes


def _at(buf):
    return ctypes.c_void_p(buf[0].data_ptr() + buf[1])


def _bytes(buf):
    return buf[0][buf[1]:buf[1] + buf[2]].cpu().numpy()


@pytest.mark.parametrize("shifts", [(1, 0, 0, 0, 0), (0, 2, 3, 1, 0), (0, 0, 0, 0, 4), (3, 1, 2, 5, 7)])
def test_odd_addresses(cuts, shifts):
    """shifts: of the inputs, of the hit tuples, the hit counts, the tracks and the offsets."""
    ev = [sim.generate(sim.PU50, 2320 + i, n_particles=600) for i in range(2)]
    want = [oracle.survivors_hits(oracle.reconstruct(e.x, e.y, e.z, e.layer, cuts)) for e in ev]
    off, *arrays = sim.concat(ev)
    cap = pt.default_capacity(max_events=2, hits_per_event=16384, cells_per_event=1 << 20,
                              links_per_event=1 << 17, ntuplets_per_event=1 << 16)
    S, room = sum(len(w) for w in want), 2 * sum(len(w) for w in want)
    ins = [_device(a, shifts[0]) for a in arrays]
    outs = [_device(np.zeros(n, np.uint8), s)
            for n, s in zip((room * 24, room, room * 36, 24), shifts[1:])]
    with pt.Context(cuts=cuts, capacity=cap) as ctx:
        _, _, tracks, _ = ctx.pt_reconstruct_batch(off, *arrays)
        n = ctypes.c_int64(0)
        torch.cuda.synchronize()
        status = pt.lib().pt_reconstruct_batch(
            ctx.handle, 2, off.ctypes.data_as(ctypes.c_void_p), *(_at(b) for b in ins), 1,
            *(_at(b) for b in outs), room, ctypes.byref(n), 1)
        assert status == pt.PT_OK and n.value == S
        hits, nhits, got, offsets = (_bytes(b) for b in outs)
        assert np.array_equal(hits.view(np.int32).reshape(-1, 6)[:S], np.concatenate(want))
        assert np.array_equal(nhits[:S], (np.concatenate(want) >= 0).sum(1))
        assert np.array_equal(got[:S * 36], tracks.view(np.uint8).reshape(-1))
        assert np.array_equal(offsets.view(np.int64), [0, len(want[0]), S])
        assert not nhits[S:].any() and not hits[S * 24:].any() and not got[S * 36:].any()
