"""Broken-line refit with next to no material: the kinks outweigh the hits by 1e7 (pairs of
floats) and by 1e11 and more (float64), and the fit goes over into one circle and one line.
Against the float64 oracle with the fit's tolerances."""

import numpy as np
import pytest

import sim
from test_brokenline_gpu import CAP, _assert_chi2_close, _chain, _oracle_refits
from test_gpu_parity import assert_fits_close

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2501_05520_gb300 as pt  # noqa: E402


@pytest.mark.parametrize("x0", [1e-6, 1e-9, 3e-13])
def test_little_material(cuts, x0):
    ev = sim.generate(sim.PU50, 2110, n_particles=1200)
    with pt.Context(cuts=cuts, capacity=CAP) as ctx:
        _chain(ctx, [ev])
        ctx.pt_refit_broken_line(x0, x0)
        tracks = ctx.pt_get_tracks()
    _, _, _, exp = _oracle_refits(ev, cuts, x0, x0)
    assert tracks.shape[0] == exp.shape[0] > 500
    assert_fits_close(tracks, exp)
    _assert_chi2_close(tracks, exp)
