"""The work that users of the library have it do, as timed and compared cases.

A case is a dict of plain values; its "kind" says which public calls one pass makes:

  chain    pt_reconstruct_batch: hits -> ntuplets and fitted tracks, one event or a batch,
           host or device buffers, plain or gated, with the skip-layer table and the
           fishbone step as options
  serve    a burst of requests through the request server (pt_submit, pt_poll)
  raw      pt_load_raw and pt_get_hits: raw digis -> hits
  refit    pt_fit_tracks and pt_refit_broken_line on a reconstructed batch
  vertex   pt_find_vertices on a reconstructed batch
  train    one training step of the gate (pt_gate_loss_grad, pt_gate_adam)
  score    pt_gate_score on feature rows

Events are seeded helices in a 3.8 T solenoid on the library's detector (4 barrel layers,
3 disks per side), smeared by 10 um (r-phi) and 20 um (z, disk r), with uniform noise: the
same recipe and sizes as the tests and the benchmark use, drawn here on the GPU so that
inputs are made quickly.  `exact` reconstructs by brute force: the cuts in float32, operation
by operation in the order the C header gives (a decision is part of the definition), and
every number that comes out of the fits in float64.
"""

import ctypes
import math

import numpy as np
import torch

import paper_2501_05520_gb300 as pt
from paper_2501_05520_gb300 import pixels

DEV = "cuda"
BARREL_R = (2.9, 6.8, 10.9, 16.0)
BARREL_Z = 27.0
DISK_Z = (29.1, 39.6, 51.6)
DISK_R = (4.5, 16.0)
BFIELD = 3.8
CURV = 0.299792458 * BFIELD / 100.0  # curvature (1/cm) of a 1 GeV track
VERTEX_DZ = 0.02                     # cm, the library's default cut
MATERIAL = 0.02                      # radiation lengths per layer, the library's default
SENSORS = (12, 28, 44, 64), 8, 48, 2  # barrel sectors per layer, z segments; disk sectors, rings

# ------------------------------------------------------------------------------- cases


def _case(kind, events, particles, **more):
    """particles: mean per event; spread "same" (every event), "poisson" (pileup of 50-particle
    interactions, Poisson) or "uniform" (pileup uniform between a quarter and the whole)."""
    c = dict(kind=kind, events=events, particles=particles, spread="same", spectrum="inv_pt",
             barrel=False, low_pt=False, gated=False, gap=False, fishbone=False,
             hit_eff=1.0, overlap=0.0, host=False, phi_bins=256, blocks=4, search_blocks=5)
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: one 50-particle barrel event (200 hits) from and to host memory,
        # where a user waits for launches and copies
        _case("chain", 1, 50, name="one_barrel", barrel=True, spectrum="inv_pt", host=True),
        # one pileup-50 event with the low-pT cuts, host memory: the ordinary latency of a call
        _case("chain", 1, 2500, name="one_pu50", spectrum="exp", low_pt=True, host=True),
        # one pileup-200 event with the learned gate, host memory: the largest single event
        _case("chain", 1, 10000, name="one_pu200_gated", gated=True, host=True),
        # the throughput workload: 64 pileup-200 events in one call on device buffers, with the
        # bin count and launch sizes that the autotuner picks for it
        _case("chain", 64, 10000, name="batch_pu200", phi_bins=2048, blocks=8, search_blocks=8),
        # a batch of uneven events (Poisson(140) pileup) with the gate, default launch sizes
        _case("chain", 64, 7000, name="batch_poisson_gated", spread="poisson", gated=True,
              phi_bins=512),
        # recovering tracks that missed a layer: skip-layer pairs and fishbone cleaning on an
        # odd number of events with inefficient, overlapping sensors
        _case("chain", 7, 7000, name="batch_gap_fishbone", gap=True, fishbone=True, hit_eff=0.9,
              overlap=0.2, phi_bins=512),
        # serving: a burst of requests of mixed size from one client, 4 slots, 2 GB
        _case("serve", 32, 10000, name="serve_burst", spread="uniform", host=True),
        # raw data of pileup-200 events to hits
        _case("raw", 6, 10000, name="raw_pu200"),
        # broken-line refit of a batch's tracks through material
        _case("refit", 24, 2500, name="refit_pu50", spectrum="exp", phi_bins=512),
        # primary vertices of pileup-200 events
        _case("vertex", 12, 10000, name="vertex_pu200", phi_bins=512),
        # gate training: the minibatch that the training script takes
        dict(kind="train", name="train_4096", rows=4096),
        # gate inference on rows that a user keeps
        dict(kind="score", name="score_300k", rows=300_001),
    ]


def draw(rng):
    kind = rng.choice(("chain", "chain", "chain", "chain", "serve", "raw", "refit", "vertex",
                       "train", "score"))

    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if kind == "train":
        return dict(kind=kind, rows=log(500, 100_000))
    if kind == "score":
        return dict(kind=kind, rows=log(1000, 1_000_000))
    if kind == "chain":
        events, particles = log(1, 64), log(50, 12500)
        gap = rng.random() < 0.25
        # events x particles^2 measures the pairs: at most the largest listed case's
        budget = 64 * 10000.0**2 / (8 if gap else 1)
        events = max(1, min(events, int(budget / particles**2)))
        low = particles <= 3000 and rng.random() < 0.3
        return _case(kind, events, particles, spread=rng.choice(("same", "poisson", "uniform")),
                     spectrum="exp" if low else "inv_pt", low_pt=low,
                     barrel=particles <= 200 and rng.random() < 0.5, gated=rng.random() < 0.4,
                     gap=gap, fishbone=rng.random() < 0.25, hit_eff=0.9 if gap else 1.0,
                     overlap=rng.choice((0.0, 0.0, 0.2)), host=events == 1 or rng.random() < 0.2,
                     phi_bins=rng.choice((128, 256, 512, 1024, 2048)),
                     blocks=rng.choice((2, 4, 8)), search_blocks=rng.choice((3, 5, 8)))
    if kind == "serve":
        return _case(kind, log(2, 48), log(2500, 10000), spread="uniform", host=True)
    if kind == "raw":
        return _case(kind, log(1, 16), log(500, 10000))
    if kind == "refit":
        return _case(kind, log(1, 32), log(500, 5000), spectrum=rng.choice(("exp", "inv_pt")),
                     phi_bins=512)
    return _case(kind, log(1, 24), log(500, 12500), phi_bins=512)


def _counts(case, seed):
    """Particles of each event."""
    rng = np.random.default_rng(seed)
    n, e = case["particles"], case["events"]
    if case["spread"] == "poisson":
        return np.clip(50 * rng.poisson(n / 50.0, e), 50, 12500)
    if case["spread"] == "uniform":
        return rng.integers(max(1, n // 4), n + 1, e)
    return np.full(e, n)


def work(case):
    """Inputs read once and outputs written once; operations: the cut tests of the doublets that
    exist (about 25 each), the links' (60) and the fits', which no method can leave out."""
    if case["kind"] == "train":
        return dict(bytes=case["rows"] * 52.0 + 5057 * 4 * 7, flops=case["rows"] * 6.0 * 4928)
    if case["kind"] == "score":
        return dict(bytes=case["rows"] * 52.0, flops=case["rows"] * 2.0 * 4928)
    n = case["particles"] * {"same": 1.0, "poisson": 1.0, "uniform": 0.625}[case["spread"]]
    hits = 4.1 * n * case["hit_eff"] * (1 + case["overlap"])
    tracks = 1.06 * n
    e = case["events"]
    if case["kind"] == "raw":
        return dict(bytes=e * hits * (3.6 * 8 + 13), flops=e * hits * 60.0)
    if case["kind"] == "refit":
        return dict(bytes=e * (hits * 13 + tracks * 61), flops=e * tracks * 2500.0)
    if case["kind"] == "vertex":
        return dict(bytes=e * (tracks * 13 + n / 50 * 16),
                    flops=e * tracks * (4 + math.log2(max(2.0, tracks))))
    cells = 1.5e-3 * hits**2 * (1.8 if case["low_pt"] else 1.0) * (2.4 if case["gap"] else 1.0)
    if case["barrel"]:
        cells *= 2.5
    return dict(bytes=e * (hits * 13 + tracks * 61),
                flops=e * (cells * 25 + 2.0 * hits * 60 + tracks * 400))


# ------------------------------------------------------------------------------- inputs


class _Hits:
    """Hits of a batch, events in order: event, x, y, z (float64), layer, particle."""

    def __init__(self, ev, x, y, z, layer, pid, n_events):
        self.ev, self.x, self.y, self.z, self.layer, self.pid = ev, x, y, z, layer, pid
        self.offsets = np.zeros(n_events + 1, np.int64)
        self.offsets[1:] = torch.cumsum(torch.bincount(ev, minlength=n_events), 0).cpu().numpy()

    def floats(self):
        return self.x.float(), self.y.float(), self.z.float(), self.layer.to(torch.uint8)


def _events(case, seed, vertices=False, scatter=False):
    counts = _counts(case, seed)
    g = torch.Generator(DEV).manual_seed(int(seed))
    P = int(counts.sum())

    def uni(n, lo=0.0, hi=1.0):
        return lo + (hi - lo) * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)

    def normal(n):
        return torch.randn(n, generator=g, device=DEV, dtype=torch.float64)

    ev = torch.repeat_interleave(torch.arange(len(counts), device=DEV),
                                 torch.as_tensor(counts, device=DEV))
    if case["spectrum"] == "exp":
        pT = 0.3 - torch.log(1.0 - uni(P))
    else:
        pT = 1.0 / uni(P, 0.1, 2.0)
    eta_max = 1.0 if case["barrel"] else 2.5
    sh = torch.sinh(uni(P, -eta_max, eta_max))
    phi0, q = uni(P, 0.0, 2 * math.pi), torch.where(uni(P) < 0.5, -1.0, 1.0).double()
    z0 = 5.0 * normal(P)
    if vertices:  # groups of 50 particles share a vertex
        z0 = z0[torch.arange(P, device=DEV) // 50 * 50]
    R = pT / CURV
    surfaces = [(L, True, r) for L, r in enumerate(BARREL_R)]
    if not case["barrel"]:
        surfaces += [(4 + k + 3 * s, False, (1 - 2 * s) * z) for s in (0, 1)
                     for k, z in enumerate(DISK_Z)]
    if case["overlap"] > 0:  # a second sensor 0.5 cm behind
        surfaces += [(L, b, v + math.copysign(0.5, v)) for L, b, v in surfaces]
    n_first = 4 if case["barrel"] else 10
    arcs, keep, rr, zz, ph = [], [], [], [], []
    for i, (L, barrel, v) in enumerate(surfaces):
        if barrel:
            ok = v < 2 * R
            s = 2 * R * torch.asin(torch.where(ok, v / (2 * R), 0.0))
            r, z = torch.full_like(s, v), z0 + s * sh
            ok = ok & (z.abs() < BARREL_Z)
        else:
            s = (v - z0) / sh
            ok = torch.isfinite(s) & (s > 0) & (s < math.pi * R)
            s = torch.where(ok, s, 0.0)
            r, z = 2 * R * torch.sin(s / (2 * R)), torch.full_like(s, v)
            ok = ok & (r >= DISK_R[0]) & (r <= DISK_R[1])
        if i >= n_first:
            ok = ok & (uni(P) < case["overlap"])
        if case["hit_eff"] < 1:
            ok = ok & (uni(P) < case["hit_eff"])
        arcs.append(s), keep.append(ok), rr.append(r), zz.append(z)
        ph.append(phi0 - q * s / (2 * R))
    if scatter:  # a kink at every crossing moves the later ones
        cosh = torch.sqrt(1 + sh * sh)
        for j, (_, bj, _) in enumerate(surfaces):
            t = MATERIAL * (cosh if bj else cosh / sh.abs().clamp_min(1e-3))
            th = 0.0136 / (pT * cosh) * torch.sqrt(t) * (1 + 0.038 * torch.log(t)) * keep[j]
            k1, k2 = th * cosh * normal(P), th * cosh * cosh * normal(P)
            for i, (_, bi, _) in enumerate(surfaces):
                d = (arcs[i] - arcs[j]).clamp_min(0.0)
                ph[i] = ph[i] + k1 * d / rr[i].clamp_min(1.0)
                if bi:
                    zz[i] = zz[i] + k2 * d
                else:
                    rr[i] = rr[i] - k2 * d / sh
    idx = [torch.nonzero(k).flatten() for k in keep]
    pid = torch.cat(idx)
    lay = torch.cat([torch.full_like(k, surfaces[i][0]) for i, k in enumerate(idx)])
    r, z, phi = (torch.cat([v[i][k] for i, k in enumerate(idx)]) for v in (rr, zz, ph))
    n = pid.numel()
    phi = phi + 10e-4 * normal(n) / r
    move = 20e-4 * normal(n)
    r, z = torch.where(lay < 4, r, r + move), torch.where(lay < 4, z + move, z)
    hev = ev[pid]
    m = 0 if case["barrel"] else int(round(0.02 * n))
    if m:  # uniform noise by area
        area = torch.tensor([2 * math.pi * v * 2 * BARREL_Z for v in BARREL_R] +
                            [math.pi * (DISK_R[1]**2 - DISK_R[0]**2)] * 6, device=DEV)
        nl = torch.multinomial(area, m, replacement=True, generator=g)
        u = uni(m)
        rl = torch.tensor(BARREL_R + (0.0,) * 6, device=DEV, dtype=torch.float64)[nl]
        zl = torch.tensor((0.0,) * 4 + DISK_Z + tuple(-v for v in DISK_Z), device=DEV,
                          dtype=torch.float64)[nl]
        rd = torch.sqrt(DISK_R[0]**2 + (DISK_R[1]**2 - DISK_R[0]**2) * u)
        hev = torch.cat([hev, hev[(uni(m) * n).long()]])
        r = torch.cat([r, torch.where(nl < 4, rl, rd)])
        z = torch.cat([z, torch.where(nl < 4, BARREL_Z * (2 * u - 1), zl)])
        phi = torch.cat([phi, uni(m, 0.0, 2 * math.pi)])
        lay, pid = torch.cat([lay, nl]), torch.cat([pid, torch.full_like(nl, -1)])
    order = torch.argsort(hev + uni(hev.numel()))  # shuffled within the event
    return _Hits(hev[order], (r * torch.cos(phi))[order], (r * torch.sin(phi))[order], z[order],
                 lay[order], pid[order], len(counts))


def _digis(h):
    """Packed digis of the hits (module << 40 | row << 28 | col << 16 | adc), event by event,
    module by module, in (row, col) order, and their offsets: a hit spreads 200 counts over a
    pixel-sized square, pixels of 4 counts or more are read out."""
    table = pixels.module_table()
    col = {f: torch.as_tensor(table[f].astype(np.float64), device=DEV)
           for f in ("phi0", "dphi_col", "v0", "dv_row", "ncol", "nrow")}
    sectors, segs, dsec, rings = SENSORS
    n_sec = torch.tensor(sectors + (dsec,) * 6, device=DEV)
    n_seg = torch.tensor((segs,) * 4 + (rings,) * 6, device=DEV)
    first = torch.cumsum(n_sec * n_seg, 0) - n_sec * n_seg
    L = h.layer
    phi = torch.atan2(h.y, h.x)
    barrel = L < 4
    v = torch.where(barrel, h.z, torch.sqrt(h.x**2 + h.y**2))
    frac = torch.where(barrel, (v + BARREL_Z) / (2 * BARREL_Z),
                       (v - DISK_R[0]) / (DISK_R[1] - DISK_R[0]))
    s = torch.minimum(((phi + math.pi) / (2 * math.pi) * n_sec[L]).long().clamp_min(0), n_sec[L] - 1)
    k = torch.minimum((frac * n_seg[L]).long().clamp_min(0), n_seg[L] - 1)
    mod = first[L] + s * n_seg[L] + k
    a = (phi - col["phi0"][mod]) / col["dphi_col"][mod]
    b = (v - col["v0"][mod]) / col["dv_row"][mod]
    keys, charge = [], []
    for i in (0, 1):
        for j in (0, 1):
            c, r = torch.floor(a - 0.5) + i, torch.floor(b - 0.5) + j
            share = ((torch.minimum(a + 0.5, c + 1) - torch.maximum(a - 0.5, c)).clamp_min(0) *
                     (torch.minimum(b + 0.5, r + 1) - torch.maximum(b - 0.5, r)).clamp_min(0))
            ok = (c >= 0) & (c < col["ncol"][mod]) & (r >= 0) & (r < col["nrow"][mod])
            key = ((h.ev * 65536 + mod) * 4096 + r.long()) * 4096 + c.long()
            keys.append(key[ok])
            charge.append((share[ok] * 200 * 1024).long())
    key, inv = torch.unique(torch.cat(keys), return_inverse=True)
    adc = torch.zeros_like(key).index_add_(0, inv, torch.cat(charge)) // 1024
    ok = adc >= 4
    key, adc = key[ok], adc[ok].clamp_max(4095)
    words = ((key >> 24) & 65535) << 40 | ((key >> 12) & 4095) << 28 | (key & 4095) << 16 | adc
    off = np.zeros(len(h.offsets), np.int64)
    off[1:] = torch.cumsum(torch.bincount(key >> 40, minlength=len(off) - 1), 0).cpu().numpy()
    return off, words


def _link_rows(rows, seed):
    """Gate features and labels of `rows` links of a pileup event, as the plain cuts make them."""
    h = _events(_case("chain", 1, 4000), seed)
    x, y, z, layer = h.floats()
    c = pt.default_cuts()
    ca = _links(x, y, z, layer, c, pt.DEFAULT_PAIRS)
    h0, h1, h2 = ca["h0"], ca["h1"], ca["h2"]
    g = torch.Generator(DEV).manual_seed(int(seed) + 1)
    pick = torch.randint(h0.numel(), (rows,), generator=g, device=DEV)
    h0, h1, h2 = h0[pick], h1[pick], h2[pick]
    label = ((h.pid[h0] >= 0) & (h.pid[h0] == h.pid[h1]) & (h.pid[h1] == h.pid[h2])).float()
    r = torch.sqrt(x * x + y * y)
    x0, y0, z0, r0, x1, y1, z1, r1, x2, y2, z2, r2 = (v[k] for k in (h0, h1, h2)
                                                      for v in (x, y, z, r))
    lc1 = ((z1 - z0) * (r2 - r0) - (z2 - z0) * (r1 - r0)).abs()
    rc1 = c["rz0"] * (r2 - r0) + c["rz1"] * (z2 - z0).abs()
    num, den, lc2, abc = _circle(x0, y0, x1, y1, x2, y2)
    L = layer.float()
    dca = torch.where(L[h0] == 0, c["dca_b0"], c["dca_other"])
    ta, tb = (z1 - z0) / (r1 - r0), (z2 - z1) / (r2 - r1)
    f = torch.stack([lc1 / rc1, lc2 / abc / c["kmax"], num.abs() / den / dca, ta / c["cotmax"],
                     10 * (tb - ta), r0 / 16, r1 / 16, r2 / 16, (z0 - r0 * ta) / c["z0max"],
                     L[h0] / 9, L[h1] / 9, L[h2] / 9], 1)
    return f.contiguous(), label


def _cuts(case):
    return pt.default_cuts("pt_min_0p25" if case["low_pt"] else "pt_min_0p45")


def _pairs(case):
    return pt.DEFAULT_PAIRS + pt.gap_pairs() if case["gap"] else pt.DEFAULT_PAIRS


def _context(case, offsets):
    """A context with room for the batch, set up as the case says."""
    n = np.diff(offsets).astype(np.float64)
    k = 2.0e-3 * (2.0 if case["low_pt"] else 1.0) * (2.6 if case["gap"] else 1.0)
    cells = int((k * n * n).sum()) + (1 << 22)
    hits = int(n.sum())
    many = 8 if case["gap"] or case["low_pt"] or case["overlap"] > 0 else 3
    cap = dict(max_events=len(n), max_hits=hits + 1024, max_cells=cells,
               max_links=many * hits + (1 << 21), max_ntuplets=many * hits + (1 << 18),
               phi_bins=case["phi_bins"], reserved=0)
    ctx = pt.Context(cuts=_cuts(case), capacity=cap)
    ctx.pt_set_launch(case["blocks"], case["search_blocks"])
    if case["gap"]:
        ctx.pt_set_layer_pairs(_pairs(case))
    if case["fishbone"]:
        ctx.pt_set_fishbone(True)
    if case["gated"]:
        ctx.pt_set_gate(*pt.default_gate())
    return ctx


def _room(case):
    """Tracks that the user's output arrays hold; what a call does not fill stays zero."""
    return case["events"] * (2 * case["particles"] + 256)


def _out(n_events, n_out, host):
    def new(shape, dtype):
        if host:
            return torch.zeros(shape, dtype=dtype, pin_memory=True)
        return torch.zeros(shape, dtype=dtype, device=DEV)

    return dict(hits=new((n_out, 6), torch.int32), nhits=new((n_out,), torch.uint8),
                tracks=new((n_out, 9), torch.float32),
                event_offsets=new((n_events + 1,), torch.int64))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        x, y = _link_rows(case["rows"], seed)
        w, m, v = _optimiser(seed)
        return dict(kind=kind, x=x, y=y, w=w, m=m, v=v, grad=torch.zeros_like(w),
                    loss=torch.zeros(1, device=DEV))
    if kind == "score":
        x, _ = _link_rows(case["rows"], seed)
        ctx = pt.Context(capacity=dict(max_events=1, max_hits=1024, max_cells=1024,
                                       max_links=case["rows"], max_ntuplets=1024, phi_bins=64,
                                       reserved=0))
        ctx.pt_set_gate(*pt.default_gate())
        return dict(kind=kind, ctx=ctx, x=x, out=torch.zeros(case["rows"], device=DEV))
    h = _events(case, seed, vertices=kind == "vertex", scatter=kind == "refit")
    arrays = h.floats()
    if kind == "serve":
        arrays = [a.cpu().numpy() for a in arrays]
        off = h.offsets
        server = pt.Server(cuts=_cuts(case), budget_bytes=2 << 30, slots=4)
        per = _room(case) // case["events"]
        return dict(kind=kind, server=server, per=per, out=_out(1, _room(case), True),
                    n=np.zeros(case["events"], np.int64),
                    events=[tuple(a[off[e]:off[e + 1]] for a in arrays)
                            for e in range(case["events"])])
    if kind == "raw":
        off, words = _digis(h)
        n = case["events"] * (6 * case["particles"] + 1024)
        ctx = pt.Context(capacity=dict(max_events=case["events"], max_hits=n, max_cells=1024,
                                       max_links=1024, max_ntuplets=1024, phi_bins=256,
                                       reserved=0))
        ctx.pt_set_modules()
        out = [torch.zeros(n, dtype=t, pin_memory=True)
               for t in (torch.float32, torch.float32, torch.float32, torch.uint8)]
        out.append(torch.zeros(case["events"] + 1, dtype=torch.int64, pin_memory=True))
        return dict(kind=kind, ctx=ctx, offsets=off, words=words, out=out)
    ctx = _context(case, h.offsets)
    if case["host"]:
        arrays = [a.cpu().pin_memory() for a in arrays]
    n = _room(case)
    out = _out(case["events"], n, case["host"])
    s = dict(kind=kind, ctx=ctx, offsets=h.offsets, hits=arrays, out=out)
    if kind in ("refit", "vertex"):
        ctx.pt_reconstruct_batch(h.offsets, *arrays, out=out)
        s["tracks"] = torch.zeros((n, 9), device=DEV)
        s["vertices"] = torch.zeros((n // 2 + 1, 4), device=DEV)
        s["track_vertex"] = torch.zeros(n, dtype=torch.int32, device=DEV)
        s["vertex_offsets"] = torch.zeros(case["events"] + 1, dtype=torch.int64, device=DEV)
    return s


def _optimiser(seed):
    """Parameters in the middle of a training: weights, first and second moments."""
    g = torch.Generator(DEV).manual_seed(int(seed) + 2)

    def normal(n):
        return torch.randn(n, generator=g, device=DEV)

    w = torch.cat([normal(768) / 12**0.5, 0.1 * normal(64), normal(4096) / 8, 0.1 * normal(64),
                   normal(64) / 8, 0.1 * normal(1)])
    return w, 1e-3 * normal(5057), 1e-6 * (0.5 + normal(5057)**2)


# ------------------------------------------------------------------------------- a pass

TRACK = ("kappa", "phi0", "d0", "cot_theta", "z0", "pt", "chi2_circle", "chi2_line")
ADAM = dict(lr=2e-3, step=1000)


def _track_fields(t):
    """[S, 9] track words -> the float fields, charge and hit count."""
    d = {f: t[:, i] for i, f in enumerate(TRACK)}
    b = t.view(torch.int8)
    return dict(d, charge=b[:, 32], nhits=b[:, 33])


_I64 = ctypes.POINTER(ctypes.c_int64)


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def _ok(status):
    if status != pt.PT_OK:
        raise pt.PtError(status, pt.lib().pt_last_error().decode())


def run(state):
    kind = state["kind"]
    if kind == "chain":
        out = state["out"]
        state["ctx"].pt_reconstruct_batch(state["offsets"], *state["hits"], out=out)
        return dict(_track_fields(out["tracks"]), hits=out["hits"], n=out["nhits"],
                    offsets=out["event_offsets"])
    if kind == "serve":
        out, n, per = state["out"], state["n"], state["per"]
        tickets = [state["server"].pt_submit(*e) for e in state["events"]]
        for i, t in enumerate(tickets):
            rows = slice(i * per, (i + 1) * per)
            _ok(pt.lib().pt_poll(state["server"].handle, t, -1, _ptr(out["hits"][rows]),
                                 _ptr(out["nhits"][rows]), _ptr(out["tracks"][rows]), per,
                                 ctypes.cast(n[i:].ctypes.data, _I64)))
        return dict(_track_fields(out["tracks"]), hits=out["hits"], n=out["nhits"], offsets=n)
    if kind == "raw":
        ctx, out = state["ctx"], state["out"]
        ctx.pt_load_raw(state["offsets"], state["words"], sync=False)
        _ok(pt.lib().pt_get_hits(ctx.handle, *(_ptr(t) for t in out), out[0].numel(),
                                 ctypes.byref(ctypes.c_int64(0))))
        return out
    if kind == "refit":
        ctx, tracks = state["ctx"], state["tracks"]
        ctx.pt_fit_tracks(sync=False)
        ctx.pt_refit_broken_line(MATERIAL, MATERIAL, sync=False)
        _ok(pt.lib().pt_get_tracks(ctx.handle, _ptr(tracks), tracks.shape[0],
                                   ctypes.byref(ctypes.c_int64(0)), 1))
        return _track_fields(tracks)
    if kind == "vertex":
        ctx, v = state["ctx"], state["vertices"]
        ctx.pt_find_vertices(4, VERTEX_DZ, sync=False)
        _ok(pt.lib().pt_get_vertices(ctx.handle, _ptr(v), _ptr(state["vertex_offsets"]),
                                     _ptr(state["track_vertex"]), v.shape[0],
                                     ctypes.byref(ctypes.c_int64(0)), 1))
        return dict(z=v[:, 0], sum_pt2=v[:, 1], counts=v.view(torch.int32)[:, 2:],
                    offsets=state["vertex_offsets"], track_vertex=state["track_vertex"])
    if kind == "train":
        pt.pt_gate_loss_grad(state["w"], state["x"], state["y"], state["grad"], state["loss"])
        pt.pt_gate_adam(state["w"], state["m"], state["v"], state["grad"], **ADAM)
        return {k: state[k] for k in ("w", "m", "v", "grad", "loss")}
    state["ctx"].pt_gate_score(state["x"], state["out"])
    return state["out"]


# ------------------------------------------------------------------------------- exact


def _filled(t, n):
    """`t` at the front of an output array of n entries."""
    return torch.nn.functional.pad(t, (0, n - t.numel()))


def _circle(x0, y0, x1, y1, x2, y2):
    """The circle through three points: distance to the z axis as num / den, and its curvature
    as lc2 / abc, in the operation order of the library's cuts."""
    ax, ay, bx, by = x1 - x0, y1 - y0, x2 - x0, y2 - y0
    cx, cy = x2 - x1, y2 - y1
    a2, b2 = ax * ax + ay * ay, bx * bx + by * by
    cr = ax * by - ay * bx
    abc = torch.sqrt(a2) * torch.sqrt(b2) * torch.sqrt(cx * cx + cy * cy)
    D = cr * 2
    ux, uy = by * a2 - ay * b2, ax * b2 - bx * a2
    num = (x0 * x0 + y0 * y0) * D + (x0 * ux + y0 * uy) * 2
    px, py = x0 * D + ux, y0 * D + uy
    den = torch.sqrt(px * px + py * py) + torch.sqrt(ux * ux + uy * uy)
    return num, den, cr.abs() * 2, abc


def _links(x, y, z, layer, cuts, pairs):
    """Cells (inner, outer) and links of one event by brute force, the cuts in float32."""
    f32 = {k: torch.tensor(v, dtype=torch.float32, device=DEV) for k, v in cuts.items()}
    r = torch.sqrt(x * x + y * y)
    where = [torch.nonzero(layer == L).flatten() for L in range(10)]
    ins, outs = [], []
    for a, b in pairs:
        for i in where[a].split(4096):
            o = where[b]
            xi, yi, zi, ri = (v[i][:, None] for v in (x, y, z, r))
            xo, yo, zo, ro = (v[o][None] for v in (x, y, z, r))
            dr, dz = ro - ri, zo - zi
            ok = (dr > 0) & (xi * xo + yi * yo > 0)
            ok &= (zi * dr - ri * dz).abs() <= f32["z0max"] * dr
            ok &= dz.abs() <= f32["cotmax"] * dr
            dx, dy = xo - xi, yo - yi
            ok &= ((xi * yo - yi * xo).abs() * 2 <=
                   f32["kmax"] * ((ri * ro) * torch.sqrt(dx * dx + dy * dy)))
            k = torch.nonzero(ok)
            ins.append(i[k[:, 0]]), outs.append(o[k[:, 1]])
    ins, outs = torch.cat(ins), torch.cat(outs)
    # cells leaving each hit, then every incoming x outgoing pair in pieces
    by_in = torch.argsort(ins, stable=True)
    n_out = torch.bincount(ins, minlength=x.numel())
    first = torch.cumsum(n_out, 0) - n_out
    src, dst, qual = [], [], []
    for a in torch.arange(ins.numel(), device=DEV).split(200_000):
        reps = n_out[outs[a]]
        s = torch.repeat_interleave(a, reps)
        k = torch.arange(s.numel(), device=DEV) - torch.repeat_interleave(
            torch.cumsum(reps, 0) - reps, reps)
        d = by_in[first[outs[s]] + k]
        h0, h1, h2 = ins[s], outs[s], outs[d]
        dz, dr = z[h2] - z[h0], r[h2] - r[h0]
        ok = (((z[h1] - z[h0]) * dr - dz * (r[h1] - r[h0])).abs() <=
              f32["rz0"] * dr + f32["rz1"] * dz.abs())
        s, d = s[ok], d[ok]
        h0, h1, h2 = ins[s], outs[s], outs[d]
        num, den, lc2, abc = _circle(x[h0], y[h0], x[h1], y[h1], x[h2], y[h2])
        dca = torch.where(layer[h0] == 0, f32["dca_b0"], f32["dca_other"])
        ok = (lc2 <= f32["kmax"] * abc) & (num.abs() <= dca * den)
        src.append(s[ok]), dst.append(d[ok]), qual.append((num.abs() / den)[ok])
    src, dst, qual = torch.cat(src), torch.cat(dst), torch.cat(qual)
    return dict(ins=ins, outs=outs, src=src, dst=dst, q=qual, h0=ins[src], h1=outs[src],
                h2=outs[dst])


def _ntuplets(x, y, z, layer, cuts, pairs):
    """Cleaned ntuplets of one event, [S, 6] padded with -1, in canonical order."""
    ca = _links(x, y, z, layer, cuts, pairs)
    ins, outs, src, dst, q = (ca[k] for k in ("ins", "outs", "src", "dst", "q"))
    C = ins.numel()
    n_out, n_in = torch.bincount(src, minlength=C), torch.bincount(dst, minlength=C)
    order = torch.argsort(src, stable=True)
    first = torch.cumsum(n_out, 0) - n_out
    path = torch.nonzero((n_out > 0) & (n_in == 0))
    qs = torch.zeros(path.shape[0], device=DEV)
    done = []
    while path.shape[0]:
        last = path[:, -1]
        reps = n_out[last]
        p = torch.repeat_interleave(torch.arange(len(path), device=DEV), reps)
        k = torch.arange(p.numel(), device=DEV) - torch.repeat_interleave(
            torch.cumsum(reps, 0) - reps, reps)
        link = order[first[last[p]] + k]
        path = torch.cat([path[p], dst[link][:, None]], 1)
        qs = qs[p] + q[link]
        leaf = n_out[path[:, -1]] == 0
        done.append((path[leaf], qs[leaf]))
        path, qs = path[~leaf], qs[~leaf]
    cells = torch.cat([torch.nn.functional.pad(p, (0, 5 - p.shape[1]), value=-1)
                       for p, _ in done]) if done else torch.zeros((0, 5), dtype=torch.long,
                                                                   device=DEV)
    qs = torch.cat([v for _, v in done]) if done else torch.zeros(0, device=DEV)
    hits = torch.cat([ins[cells[:, :1]], torch.where(cells >= 0, outs[cells], -1)], 1)
    for k in (5, 4, 3, 2, 1, 0):  # canonical order
        o = torch.argsort(hits[:, k], stable=True)
        cells, qs, hits = cells[o], qs[o], hits[o]
    n = (hits >= 0).sum(1)
    o = torch.argsort(qs, stable=True)
    o = o[torch.argsort(-n[o], stable=True)]
    rank = torch.empty_like(o)
    rank[o] = torch.arange(o.numel(), device=DEV)
    best = torch.full((C,), o.numel(), device=DEV)
    has = cells >= 0
    best.scatter_reduce_(0, cells[has], rank[:, None].expand_as(cells)[has], "amin")
    alive = ((best[cells] == rank[:, None]) | ~has).all(1)
    used = torch.zeros(x.numel(), dtype=torch.bool, device=DEV)
    longer = hits[alive & (n >= 4)]
    used[longer[longer >= 0]] = True
    return hits[alive & ~((n == 3) & used[hits[:, :3]].any(1))]


def _fit(x, y, z, hits):
    """Circle (Karimaki, equal weights) and line fit of every ntuplet in float64."""
    ok = hits >= 0
    n = ok.sum(1, keepdim=True).double()
    X, Y, Z = (torch.where(ok, v.double()[hits], 0.0) for v in (x, y, z))

    def mean(v):
        return torch.where(ok, v, 0.0).sum(1, keepdim=True) / n

    W = X * X + Y * Y
    dx, dy, dw = X - mean(X), Y - mean(Y), W - mean(W)
    cxx, cxy, cyy = mean(dx * dx), mean(dx * dy), mean(dy * dy)
    cxw, cyw, cww = mean(dx * dw), mean(dy * dw), mean(dw * dw)
    phi = 0.5 * torch.atan2(2 * (cww * cxy - cxw * cyw),
                            cww * (cxx - cyy) - cxw * cxw + cyw * cyw)
    last = (n.long() - 1)
    along = (torch.cos(phi) * (X.gather(1, last) - X[:, :1]) +
             torch.sin(phi) * (Y.gather(1, last) - Y[:, :1]))
    phi = torch.where(along < 0, torch.where(phi > 0, phi - math.pi, phi + math.pi), phi)
    s, c = torch.sin(phi), torch.cos(phi)
    k = (s * cxw - c * cyw) / cww
    delta = -k * mean(W) + s * mean(X) - c * mean(Y)
    root = torch.sqrt(1 - 4 * delta * k)
    rho, d = 2 * k / root, 2 * delta / (1 + root)
    F = (k * dw - dx * s + dy * c) / root
    eps = 2 * F / (1 + torch.sqrt(1 + 2 * rho * F))
    lx, ly = X - d * s, Y + d * c
    chord = torch.sqrt(lx * lx + ly * ly)
    t = (0.5 * rho.abs() * chord).clamp_max(1.0)
    arc = chord * torch.where(t > 1e-9, torch.asin(t) / t.clamp_min(1e-9), 1.0)
    arc = torch.where(c * lx + s * ly >= 0, arc, -arc)
    ds, dz = arc - mean(arc), Z - mean(Z)
    cot = mean(ds * dz) / mean(ds * ds)
    z0 = mean(Z) - cot * mean(arc)
    chi_c = n * mean((eps / 10e-4)**2)
    chi_l = n * mean(((dz - cot * ds) / 20e-4)**2)
    kap = -rho
    v = dict(kappa=kap, phi0=phi, d0=d, cot_theta=cot, z0=z0, pt=CURV / kap.abs(),
             chi2_circle=chi_c, chi2_line=chi_l)
    return {f: a[:, 0] for f, a in v.items()}


def _normal(blocks, weights, rhs_w, rhs):
    """Solves min sum w (rhs - u_i)^2 + sum over blocks of w_b (coefficients . u)^2."""
    A = torch.diag_embed(rhs_w)
    for (cols, coef), w in zip(blocks, weights):
        for i, ci in zip(cols, coef):
            for j, cj in zip(cols, coef):
                A[:, i, j] += w * ci * cj
    return torch.linalg.solve(A, (rhs_w * rhs)[:, :, None])[:, :, 0]


def _refit(x, y, z, layer, hits, fit):
    """Broken-line refit in float64 (Blobel, NIM A566 (2006) 14, in the library's form)."""
    ok, n = hits >= 0, (hits >= 0).sum(1)
    X, Y, Z = (torch.where(ok, v.double()[hits], 0.0) for v in (x, y, z))
    barrel = torch.where(ok, layer[hits] < 4, True)
    f = {k: v.clone() for k, v in fit.items()}
    todo = torch.ones_like(n, dtype=torch.bool)
    one = torch.ones_like(X[:, 0])
    for _ in range(4):
        k0, p0, d0, cot, z0 = (f[k] for k in ("kappa", "phi0", "d0", "cot_theta", "z0"))
        cx, cy = (d0 - 1 / k0) * torch.sin(p0), -(d0 - 1 / k0) * torch.cos(p0)
        bx, by = X - cx[:, None], Y - cy[:, None]
        ax, ay = (torch.sin(p0) / k0)[:, None], (-torch.cos(p0) / k0)[:, None]
        s = torch.atan2(ax * by - ay * bx, ax * bx + ay * by) / k0[:, None]
        eps = torch.sign(k0)[:, None] * (1 / k0.abs()[:, None] - torch.sqrt(bx * bx + by * by))
        s, eps = torch.where(ok, s, 0.0), torch.where(ok, eps, 0.0)
        seg = ok[:, 1:]
        h = torch.where(seg, s[:, 1:] - s[:, :-1], 1.0)
        go = todo & torch.isfinite(k0 + p0 + d0 + cot + z0) & (k0.abs() >= 1e-7)
        go &= ((h > 1e-6) | ~seg).all(1)
        sth = 1 / torch.sqrt(1 + cot * cot)
        p = CURV / k0.abs() / sth
        psi = p0[:, None] + k0[:, None] * s
        inc = ((sth[:, None] * (torch.cos(psi) * X + torch.sin(psi) * Y)).abs() /
               torch.sqrt(X * X + Y * Y).clamp_min(1e-9))
        inc = torch.where(barrel, inc, (cot * sth).abs()[:, None]).clamp_min(1e-3)
        t = MATERIAL / inc
        th = 0.0136 / p[:, None] * torch.sqrt(t) * (1 + 0.038 * torch.log(t))
        kink = ok.clone()
        kink[:, 0] = False
        kink[:, :-1] &= ok[:, 1:]
        kink[:, -1] = False
        wt = torch.where(kink, (sth[:, None] / th)**2, 0.0)
        wl = wt * (sth * sth)[:, None]
        a = k0[:, None] / torch.sin(k0[:, None] * h)
        c = torch.cos(k0[:, None] * h)
        g = 2 * torch.sin(0.5 * k0[:, None] * h)**2 / (k0 * k0)[:, None]
        blocks = [((i - 1, i, i + 1, 6),
                   (a[:, i - 1], -(a[:, i] * c[:, i] + a[:, i - 1] * c[:, i - 1]), a[:, i],
                    -(a[:, i] * g[:, i] + a[:, i - 1] * g[:, i - 1]))) for i in range(1, 5)]
        wm = torch.where(ok, 1e6, 1.0).double()
        wm = torch.cat([wm, torch.zeros_like(wm[:, :1])], 1)
        full = torch.cat([eps, torch.zeros_like(eps[:, :1])], 1)
        bad = ~go  # keeps its fit: an empty system in its place
        blocks = [(i, tuple(torch.where(bad, 0.0, v) for v in co)) for i, co in blocks]
        u = _normal(blocks + [((6,), (torch.where(bad, 1.0, 0.0),))],
                    [torch.where(bad, 0.0, wt[:, i]) for i in range(1, 5)] + [one],
                    torch.where(bad[:, None], 1.0, wm), torch.where(bad[:, None], 0.0, full))
        dk = u[:, 6]
        c2t = (torch.where(ok, (eps - u[:, :6])**2 * 1e6, 0.0)).sum(1)
        for (cols, co), w in zip(blocks, wt[:, 1:5].T):
            c2t = c2t + w * sum(q * u[:, i] for i, q in zip(cols, co))**2
        du1 = a[:, 0] * (u[:, 1] - c[:, 0] * u[:, 0]) - a[:, 0] * g[:, 0] * dk
        s0 = s[:, 0]
        cs, sn = torch.cos(k0 * s0), torch.sin(k0 * s0) / k0
        gs = 2 * torch.sin(0.5 * k0 * s0)**2 / (k0 * k0)
        u0 = u[:, 0] * cs + gs * dk - du1 * sn
        du0 = du1 * cs + k0 * k0 * u[:, 0] * sn - dk * sn
        acc = s0 * (u0 + u[:, 0]) * 0.5 - dk * s0**3 / 12
        sp = [s0 - k0 * acc]
        for i in range(1, 6):
            hh = h[:, i - 1]
            acc = acc + torch.where(seg[:, i - 1], hh * (u[:, i - 1] + u[:, i]) * 0.5 -
                                    dk * hh**3 / 12, 0.0)
            sp.append(torch.where(ok[:, i], s[:, i] - k0 * acc, 0.0))
        sp = torch.stack(sp, 1)
        ih = 1 / torch.where(seg, sp[:, 1:] - sp[:, :-1], 1.0)
        wz = torch.where(barrel, 1 / 20e-4**2, (1 / (cot.abs() * 20e-4).clamp_min(1e-12)**2)[:, None])
        wz = torch.where(ok, wz, 0.0)
        dl = torch.where(ok, Z - (z0[:, None] + cot[:, None] * sp), 0.0)
        blocks = [((i - 1, i, i + 1), (ih[:, i - 1], -(ih[:, i - 1] + ih[:, i]), ih[:, i]))
                  for i in range(1, 5)]
        blocks = [(i, tuple(torch.where(bad, 0.0, v) for v in co)) for i, co in blocks]
        wv = _normal(blocks, [torch.where(bad, 0.0, wl[:, i]) for i in range(1, 5)],
                     torch.where(bad[:, None] | ~ok, 1.0, wz),
                     torch.where(bad[:, None], 0.0, dl))
        c2l = (torch.where(ok, (dl - wv)**2 * wz, 0.0)).sum(1)
        for (cols, co), w in zip(blocks, wl[:, 1:5].T):
            c2l = c2l + w * sum(q * wv[:, i] for i, q in zip(cols, co))**2
        dw1 = (wv[:, 1] - wv[:, 0]) * ih[:, 0]
        kap = k0 + dk
        new = dict(kappa=kap, phi0=torch.remainder(p0 + du0 + math.pi, 2 * math.pi) - math.pi,
                   d0=d0 - u0, cot_theta=cot + dw1, z0=z0 + wv[:, 0] - sp[:, 0] * dw1,
                   pt=CURV / kap.abs(), chi2_circle=c2t, chi2_line=c2l)
        f = {k: torch.where(go, new[k], f[k]) for k in f}
        todo = go & (dk.abs() / k0.abs() > 1e-3)
        if not todo.any():
            break
    return f


def _reconstructed(case, seed, **more):
    """Cleaned ntuplets of the case's batch event by event, with the event's float32 hits."""
    h = _events(case, seed, **more)
    arrays = h.floats()
    for e in range(case["events"]):
        a = [v[h.offsets[e]:h.offsets[e + 1]] for v in arrays]
        yield a, _ntuplets(*a, _cuts(case), _pairs(case))


def _mlp(w):
    W1, b1, W2, b2, w3, b3 = torch.split(w, (768, 64, 4096, 64, 64, 1))
    return W1.view(64, 12), b1, W2.view(64, 64), b2, w3, b3


def _exact_train(case, seed):
    x, y = (v.double() for v in _link_rows(case["rows"], seed))
    w, m, v = (t.double() for t in _optimiser(seed))
    w.requires_grad_(True)
    W1, b1, W2, b2, w3, b3 = _mlp(w)
    s = torch.relu(torch.relu(x @ W1.T + b1) @ W2.T + b2) @ w3 + b3
    loss = torch.nn.functional.binary_cross_entropy_with_logits(s, y)
    loss.backward()
    g = w.grad
    m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
    step = ADAM["lr"] * (m / (1 - 0.9**ADAM["step"])) / (
        torch.sqrt(v / (1 - 0.999**ADAM["step"])) + 1e-8)
    return dict(w=w.detach() - step, m=m, v=v, grad=g, loss=loss.detach().reshape(1))


def _exact_score(case, seed):
    def bf16(t):
        return t.to(torch.bfloat16).double()

    x, _ = _link_rows(case["rows"], seed)
    W1, b1, W2, b2, w3, b3 = _mlp(torch.as_tensor(pt.default_gate()[0], device=DEV))
    h = torch.relu(bf16(x) @ bf16(W1).T + b1.double())
    return torch.relu(bf16(h) @ bf16(W2).T + b2.double()) @ w3.double() + b3.double()


def _exact_raw(case, seed):
    off, words = _digis(_events(case, seed))
    ev = torch.repeat_interleave(torch.arange(case["events"], device=DEV),
                                 torch.as_tensor(np.diff(off), device=DEV))
    mod, row, col, adc = words >> 40, (words >> 28) & 4095, (words >> 16) & 4095, words & 65535
    key = ((ev * 65536 + mod) * 4098 + row + 1) * 4098 + col + 1  # a margin on every side
    n = key.numel()
    me, near = [], []
    for d in (1, 4097, 4098, 4099):
        k = torch.searchsorted(key, key + d).clamp_max(n - 1)
        hit = torch.nonzero(key[k] == key + d).flatten()
        me.append(hit), near.append(k[hit])
    a, b = torch.cat(me + near), torch.cat(near + me)
    lab = torch.arange(n, device=DEV)
    while True:
        new = lab.clone().scatter_reduce_(0, a, lab[b], "amin")
        new = new[new]
        if torch.equal(new, lab):
            break
        lab = new
    root = torch.nonzero(lab == torch.arange(n, device=DEV)).flatten()

    def total(v):
        return torch.zeros(n, dtype=torch.long, device=DEV).index_add_(0, lab, v)[root].double()

    w = 2 * total(adc)
    t = {f: torch.as_tensor(pixels.module_table()[f].astype(np.float64), device=DEV)[mod[root]]
         for f in ("kind", "rz", "phi0", "dphi_col", "v0", "dv_row")}
    phi = t["phi0"] + total(adc * (2 * col + 1)) / w * t["dphi_col"]
    v = t["v0"] + total(adc * (2 * row + 1)) / w * t["dv_row"]
    flat = t["kind"] == 0
    rad = torch.where(flat, t["rz"], v)
    room = case["events"] * (6 * case["particles"] + 1024)
    return [_filled(a, room) for a in (rad * torch.cos(phi), rad * torch.sin(phi),
                                       torch.where(flat, v, t["rz"]))] + [None, None]


def _exact_vertex(case, seed):
    zs, ps = [], []
    for (x, y, z, layer), hits in _reconstructed(case, seed, vertices=True):
        f = _fit(x, y, z, hits)
        take = ((hits >= 0).sum(1) >= 4) & torch.isfinite(f["z0"])
        z0, order = torch.sort(f["z0"][take])
        p2 = f["pt"][take][order]**2
        if (z0[1:] - z0[:-1] - VERTEX_DZ).abs().min() < 1e-5:
            return None  # a step so close to the cut falls on either side in float32
        start = torch.ones_like(z0, dtype=torch.bool)
        start[1:] = z0[1:] - z0[:-1] > VERTEX_DZ
        group = torch.cumsum(start, 0) - 1
        n = torch.bincount(group)
        zs.append((torch.zeros(n.numel(), dtype=torch.float64, device=DEV).index_add_(
            0, group, z0) / n)[n >= 2])
        ps.append(torch.zeros(n.numel(), dtype=torch.float64, device=DEV).index_add_(
            0, group, p2)[n >= 2])
    n = _room(case) // 2 + 1
    return dict(z=_filled(torch.cat(zs), n), sum_pt2=_filled(torch.cat(ps), n), counts=None,
                offsets=None, track_vertex=None)


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "score":
        return _exact_score(case, seed)
    if kind == "raw":
        return _exact_raw(case, seed)
    if kind == "vertex":
        return _exact_vertex(case, seed) if case["events"] <= 12 else None
    if case["gated"] or case["fishbone"]:
        return None  # which links are kept is decided by a network, or by a rule of its own
    if case["events"] * case["particles"]**2 > 12e8 or kind == "serve" and case["events"] > 16:
        return None  # brute force over every pair of hits takes too long
    fits = []
    for (x, y, z, layer), hits in _reconstructed(case, seed, scatter=kind == "refit"):
        f = _fit(x, y, z, hits)
        fits.append(_refit(x, y, z, layer, hits, f) if kind == "refit" else f)
    if kind == "serve":  # every request has its own part of the output arrays
        per = _room(case) // case["events"]
        fits = [{f: _filled(v[f], per) for f in TRACK} for v in fits]
    out = {f: _filled(torch.cat([v[f] for v in fits]), _room(case)) for f in TRACK}
    out.update(charge=None, nhits=None)
    if kind != "refit":
        out.update(hits=None, n=None, offsets=None)
    return out
