"""The searches' azimuthal windows and their quick form of the doublet cuts: tracks whose
curvature lies on the curvature cut (within 1e-8 to 1e-2 of it, either side) and whose hits sit
on bin edges and around the azimuth's wrap, with windows from less than a bin to a half plane,
and at radii where the quick form has to give way.  Cells and links are the oracle's, which
evaluates the cuts' fixed float32 form on every pair."""

import numpy as np
import pytest

import oracle
from parity import cell_set, oracle_link_triples

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2501_05520_gb300 as pt  # noqa: E402


def _event(kmax, scale, n, bins, seed):
    """n tracks from the beam line through the four barrel layers (radii times scale)."""
    rng = np.random.default_rng(seed)
    r = np.array([2.9, 6.8, 10.9, 16.0]) * (1 + 1e-3 * rng.uniform(-1, 1, (n, 4)))
    off = rng.choice([0.0, 1e-8, 1e-7, 3e-7, 1e-6, 1e-5, 1e-4, 1e-2], n) * rng.choice([-1, 1], n)
    curv = kmax * (1 + off) * rng.choice([-1, 1], n)
    edge = 2 * np.pi / bins * rng.integers(-2, 3, n) + 1e-6 * rng.integers(-1, 2, n)
    phi0 = np.where(np.arange(n) % 3 == 0, np.pi, rng.uniform(-np.pi, np.pi, n)) + edge
    phi = phi0[:, None] + np.arcsin(np.clip(0.5 * curv[:, None] * r, -1, 1))
    z = rng.normal(0, 3, n)[:, None] + r * rng.uniform(-1.4, 1.4, n)[:, None]
    x, y, z = ((scale * v).astype(np.float32).ravel()
               for v in (r * np.cos(phi), r * np.sin(phi), z))
    order = rng.permutation(4 * n)
    layer = np.tile(np.arange(4, dtype=np.uint8), n)
    return [np.ascontiguousarray(v[order]) for v in (x, y, z, layer)]


@pytest.mark.parametrize("kmax,scale,n", [
    (0.0253, 1.0, 300),    # the library's cuts
    (0.0004, 1.0, 300),    # windows below a bin
    (0.0570, 1.0, 200),    # the low-momentum cuts
    (0.0870, 1.0, 120),    # just below and just above where the curvature bound ends
    (0.0880, 1.0, 120),
    (0.6000, 1.0, 80),     # half planes
    (0.0253, 1e-10, 100),  # radii below and above the quick form's range
    (0.0253, 1e10, 100),
    (0.0, 1.0, 100),
])
@pytest.mark.parametrize("bins", [16, 256, 4096])
@pytest.mark.parametrize("room", [4096, 65536])  # windows found in the search, or before it
def test_cells_and_links(cuts, kmax, scale, n, bins, room):
    c = dict(cuts, kmax=kmax / scale, z0max=cuts["z0max"] * scale, rz0=cuts["rz0"] * scale,
             dca_b0=cuts["dca_b0"] * scale, dca_other=cuts["dca_other"] * scale)
    hits = _event(kmax, scale, n, bins, 97 + bins)
    ref = oracle.reconstruct(*hits, c)
    n_hits = len(hits[0])
    cap = pt.default_capacity(max_events=1, hits_per_event=room, cells_per_event=1 << 20,
                              links_per_event=1 << 20, ntuplets_per_event=1 << 16, phi_bins=bins)
    with pt.Context(cuts=c, capacity=cap) as ctx:
        ctx.pt_load_batch(np.array([0, n_hits], np.int32), *hits)
        ctx.pt_build_doublets()
        ctx.pt_build_doublets()  # the search leaves nothing behind that a second one trips on
        ctx.pt_connect_cells()
        ci, co, _ = ctx.pt_get_cells()
        h0, h1, h2, q, _ = ctx.pt_get_links()
    assert len(ci) == len(ref["cell_inner"])
    assert cell_set(ci, co) == cell_set(ref["cell_inner"], ref["cell_outer"])

    def bits(v):  # 0 / 0 at vanishing radii: the bits of a NaN are not defined
        return np.where(np.isnan(v), np.float32(np.nan), v).view(np.uint32)

    got = dict(zip(zip(h0.tolist(), h1.tolist(), h2.tolist()), bits(q).tolist()))
    ref["link_q"] = bits(ref["link_q"]).view(np.float32)
    assert len(q) == len(got) and got == oracle_link_triples(ref)
