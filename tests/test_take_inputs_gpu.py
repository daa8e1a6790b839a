"""Device inputs of pt_enqueue_batch pass through one copying launch of four hits per thread: the
context's hits equal the inputs at sizes around a block, around one and around four hits for every
thread of the launch."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2501_05520_gb300 as pt  # noqa: E402

THREADS = 8 * 256  # per multiprocessor


@pytest.mark.parametrize("rounds,more", [(0, 1), (0, 255), (0, 257), (1, -1), (1, 0), (1, 1),
                                         (4, -1), (4, 1), (9, 77)])
def test_hits_arrive(rounds, more):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = rounds * THREADS * sms + more
    rng = np.random.default_rng(3)
    x, y, z = (rng.normal(size=n).astype(np.float32) for _ in range(3))
    layer = rng.integers(0, 10, n).astype(np.uint8)
    off = np.arange(0, n + 1, dtype=np.int64) if n < 2 else \
        np.unique(np.concatenate([[0, n], np.arange(0, n, 40)])).astype(np.int64)
    cap = dict(pt.default_capacity(max_events=len(off), phi_bins=16), max_hits=n,
               max_cells=64, max_links=64, max_ntuplets=64)
    cuts = dict(pt.default_cuts(), z0max=1e-9)  # next to no doublets
    data = [torch.from_numpy(a).cuda() for a in (x, y, z, layer)]
    with pt.Context(cuts=cuts, capacity=cap) as ctx:
        ctx.pt_enqueue_batch(off, *data)
        got = ctx.pt_get_hits()
    for a, b in zip(got, (x, y, z, layer, off)):
        assert np.array_equal(a, b)
