"""Module runs around the sizes where the clustering changes hands: 224 digis (a warp, then a
block), 512 (one step of the block, then two) and 1024 (the most), against the oracle.  Hits in
the oracle's order, positions within the 2e-5 cm that float32 rounding leaves."""

import numpy as np
import pytest

from oracle import pixels as opix

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2501_05520_gb300 as pt  # noqa: E402
from paper_2501_05520_gb300 import pixels as ppix  # noqa: E402
from test_raw_gpu import _sparse_run  # noqa: E402


@pytest.mark.parametrize("sizes", [(31, 32, 33, 223, 224), (225, 224, 1), (511, 512, 513),
                                   (1023, 1024, 224, 225)])
def test_sizes(cuts, sizes):
    rng = np.random.default_rng(sum(sizes))
    table = opix.modules(ppix.PARAMS)
    mods = [3, 40, 500, 1000, 1100][:len(sizes)]
    words = np.concatenate([_sparse_run(rng, m, n, int(table[m, 8]), int(table[m, 7]))
                            for m, n in zip(mods, sizes)])
    rx, ry, rz, rl, _ = opix.reconstruct(words, table)
    off = np.array([0, len(words)], np.int64)
    cap = pt.default_capacity(max_events=1, hits_per_event=65536, cells_per_event=1024,
                              links_per_event=1024, ntuplets_per_event=1024)
    with pt.Context(cuts=cuts, capacity=cap) as ctx:
        ctx.pt_set_modules()
        n = ctx.pt_load_raw(off, words)
        x, y, z, layer, _ = ctx.pt_get_hits()
    assert n == rx.size > 0 and np.array_equal(layer, rl.astype(np.uint8))
    for got, exp in ((x, rx), (y, ry), (z, rz)):
        assert np.max(np.abs(got.astype(np.float64) - exp)) <= 2e-5
