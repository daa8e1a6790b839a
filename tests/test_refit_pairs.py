"""The broken-line refit solves its two planes in pairs of float32 (48 bits) while no kink outweighs
the hits by more than a limit, and in float64 beyond.  This file restates the pair arithmetic and
the elimination of solve_plane over numpy float32, takes the limit from the kernel's source, and
solves both planes at the limit: the offsets must agree with the exact solution (rationals) to half
a unit in the last place of a float32 offset of 0.1 cm, 3.7e-9 cm, so that what the pairs lose
against float64 does not reach the float32 results.
"""

import os
import re
from fractions import Fraction

import numpy as np
import pytest

f32, f64 = np.float32, np.float64
SRC = os.path.join(os.path.dirname(__file__), "..", "paper_2501_05520_gb300", "csrc",
                   "brokenline.cu")
STIFF = float(re.search(r"kStiffMax = ([0-9.e+]+)f;", open(SRC).read()).group(1))
SIGMA_T, SIGMA_L = 10e-4, 20e-4  # cm
TOL = 2.0 ** -28                 # cm


def fma(a, b, c):  # float32; the product is exact in float64
    return (a.astype(f64) * b.astype(f64) + c.astype(f64)).astype(f32)


class F2:
    """h + l, as the kernel's F2."""

    def __init__(self, h, l):
        self.h, self.l = h, l

    @staticmethod
    def of(v):
        h = np.asarray(v, f64).astype(f32)
        return F2(h, (v - h.astype(f64)).astype(f32))

    @staticmethod
    def quick(a, b):
        s = a + b
        return F2(s, b - (s - a))

    def __neg__(self):
        return F2(-self.h, -self.l)

    def __add__(self, o):
        s = self.h + o.h
        t = s - self.h
        e = (self.h - (s - t)) + (o.h - t)
        return F2.quick(s, e + (self.l + o.l))

    def __mul__(self, o):
        p = self.h * o.h
        return F2.quick(p, fma(self.l, o.h, fma(self.h, o.l, fma(self.h, o.h, -p))))

    def mad(self, b, c):
        p = self.h * b.h
        e = fma(self.l, b.h, fma(self.h, b.l, fma(self.h, b.h, -p)))
        s = p + c.h
        t = s - p
        r = (p - (s - t)) + (c.h - t)
        return F2.quick(s, r + (e + c.l))

    def recip(self):
        r = f32(1) / self.h
        e = fma(-self.l, r, fma(-self.h, r, np.ones_like(r)))
        return F2.quick(r, r * e)

    def value(self):
        return self.h.astype(f64) + self.l.astype(f64)


def solve_pairs(n, wm, w, a, b, g, e, bend):
    """solve_plane in pairs: the offsets u_0..u_n-1."""
    zero = F2.of(np.zeros_like(e[0].value()))
    d0, d1, d2 = wm[0], wm[1], wm[2]
    e1 = f1 = e2 = b0 = b1 = b2 = bb = rb = zero
    r0, r1, r2 = e[0] * d0, e[1] * d1, e[2] * d2
    L1, L2, LB, U = [], [], [], []
    for j in range(n):
        if j + 2 < n:
            q0, q1, q2 = a[j], -(b[j] + b[j + 1]), a[j + 1]
            q3 = -(g[j] + g[j + 1])
            w0, w1, w2, w3 = (w[j + 1] * q for q in (q0, q1, q2, q3))
            d0, e1, e2, b0 = w0.mad(q0, d0), w0.mad(q1, e1), w0 * q2, w0.mad(q3, b0)
            d1, f1, b1 = w1.mad(q1, d1), w1 * q2, w1.mad(q3, b1)
            d2, b2, bb = w2.mad(q2, d2), w2 * q3, w3.mad(q3, bb)
        inv = d0.recip()
        l1, l2, lb = e1 * inv, e2 * inv, b0 * inv
        L1.append(l1), L2.append(l2), LB.append(lb), U.append(r0 * inv)
        bb, rb = (-lb).mad(b0, bb), (-lb).mad(r0, rb)
        r0 = (-l1).mad(r0, r1)
        r1 = (-l2).mad(U[j] * d0, r2)
        b0, b1 = (-lb).mad(e1, b1), (-lb).mad(e2, b2)
        d0, d1 = (-l1).mad(e1, d1), (-l2).mad(e2, d2)
        e1 = (-l2).mad(e1, f1)
        e2 = f1 = b2 = zero
        d2 = wm[j + 3] if j + 3 < n else F2.of(np.ones_like(d0.value()))
        r2 = e[j + 3] * d2 if j + 3 < n else zero
    dk = rb * bb.recip() if bend else zero
    x1 = x2 = zero
    for j in reversed(range(n)):
        x = (-L1[j]).mad(x1, (-L2[j]).mad(x2, (-LB[j]).mad(dk, U[j])))
        U[j], x2, x1 = x, x1, x
    return [u.value() for u in U]


def solve_exact(n, wm, w, h, e, bend):
    m = n + bend
    A = [[Fraction(0)] * m for _ in range(m)]
    r = [Fraction(0)] * m
    for i in range(n):
        A[i][i] += Fraction(wm[i])
        r[i] += Fraction(wm[i]) * Fraction(e[i])
    for i in range(1, n - 1):
        hp, hn = Fraction(h[i - 1]), Fraction(h[i])
        q = {i - 1: 1 / hp, i: -(1 / hp + 1 / hn), i + 1: 1 / hn}
        if bend:
            q[n] = -(hp + hn) / 2
        for x in q:
            for y in q:
                A[x][y] += Fraction(w[i]) * q[x] * q[y]
    for j in range(m):
        for i in range(j + 1, m):
            f = A[i][j] / A[j][j]
            r[i] -= f * r[j]
            for k in range(j, m):
                A[i][k] -= f * A[j][k]
    for j in reversed(range(m)):
        r[j] = (r[j] - sum(A[j][k] * r[k] for k in range(j + 1, m))) / A[j][j]
    return [float(v) for v in r[:n]]


@pytest.mark.parametrize("n", [4, 6])
@pytest.mark.parametrize("plane,cot", [("transverse", 0.0), ("barrel z", 0.5), ("disk r", 6.0),
                                       ("disk r", 12.0), ("barrel and disk", 2.0)])
def test_offsets_at_the_limit(plane, cot, n):
    rng = np.random.default_rng(11)
    trials = 12
    h = rng.uniform(2.0, 9.0, (n - 1, trials)).astype(f32).astype(f64)
    sth2 = f64(f32(1.0 / (1.0 + cot * cot)))
    sigma = {"transverse": [SIGMA_T] * n, "barrel z": [SIGMA_L] * n,
             "disk r": [cot * SIGMA_L] * n,
             "barrel and disk": [SIGMA_L] * 2 + [cot * SIGMA_L] * (n - 2)}[plane]
    kf = 1.0 if plane == "transverse" else sth2
    # the kernel's measure, at its limit: kink weight times the larger inverse step squared,
    # times |cot| / 2 where that is above 1
    w = np.zeros((n, trials))
    for i in range(1, n - 1):
        w[i] = (STIFF / max(1.0, cot / 2) * np.minimum(h[i - 1], h[i])**2).astype(f32)
    wm = [1.0 / (s * s) for s in sigma]
    e = rng.normal(size=(n, trials)) * np.array(sigma)[:, None]
    hp = [F2.of(v) for v in h]
    a = [v.recip() for v in hp]
    half = F2.of(np.full(trials, 0.5))
    bend = plane == "transverse"
    g = [x * (v * v * half) if bend else F2.of(np.zeros(trials)) for x, v in zip(a, hp)]
    pairs = solve_pairs(n, [F2.of(np.full(trials, v)) for v in wm],
                        [F2.of(np.full(trials, kf)) * F2.of(v) for v in w], a, a, g,
                        [F2.of(v) for v in e], bend)
    for t in range(trials):
        exact = solve_exact(n, wm, kf * w[:, t], h[:, t], e[:, t], bend)
        worst = max(abs(p[t] - x) for p, x in zip(pairs, exact))
        assert worst <= TOL, (plane, t, worst)
