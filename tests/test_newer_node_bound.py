"""The mixed pair kernel's newer-node bound, restated in FP32 (CPU only): whenever it accepts, the newer node's test is
true in exact arithmetic, near that node's light sphere, for bent trajectories and over gamma; it accepts pairs well
inside the bracket; and without its margin it would accept wrong ones.
"""
from fractions import Fraction

import numpy as np
import pytest

F = np.float32
C = 299792458.0
U = 2.0 ** -24
MARGIN = F(33.0 * U)


def fma(a, b, c):
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(F)


def dot3(a, b):
    return fma(a[:, 2], b[:, 2], fma(a[:, 1], b[:, 1], a[:, 0] * b[:, 0]))


def cases(rng, m, near):
    """m pairs: older node A, newer node B off A's line, target near B's light sphere (relative distance `near`)."""
    gamma = np.exp(rng.uniform(np.log(1.02), np.log(128.0), m))
    beta = np.sqrt(1.0 - 1.0 / gamma ** 2)
    vd = rng.normal(size=(m, 3))
    vd /= np.linalg.norm(vd, axis=1)[:, None]
    v = beta[:, None] * C * vd
    dt = 1e-15 * np.exp(rng.uniform(0, 3, m))
    nA = np.exp(rng.uniform(np.log(2.0), np.log(1000.0), m))  # slots from A to the present
    tA, tB = -nA * dt, -(nA - 1.0) * dt
    wA = rng.normal(size=(m, 3)) * 50e-6
    dev = rng.normal(size=(m, 3)) * (C * dt * 10.0 ** rng.uniform(-9, -2, m))[:, None]
    wB = wA + v * (tB - tA)[:, None] + dev
    fwd = rng.random(m) < 0.5  # half of the targets ahead of the source, where the solve is badly conditioned
    nh = rng.normal(size=(m, 3))
    nh = np.where(fwd[:, None], vd + 0.3 / gamma[:, None] * nh, nh)
    nh /= np.linalg.norm(nh, axis=1)[:, None]
    eps = near * rng.choice([-1.0, 1.0], m) * rng.random(m)
    r = wB + nh * (-C * tB * (1.0 + eps))[:, None]
    return r, wA, wB, v, tA, tB, gamma


def accepts(rng, r, wA, wB, v, tA, tB, gamma, margin):
    """The kernel's FP32 sequence, with up to 2 units in the last place of error in its approximate operations."""
    ulp = lambda x: (x * (1.0 + rng.uniform(-2, 2, x.shape) * U)).astype(F)  # noqa: E731
    hi = lambda x: x.astype(F)  # noqa: E731
    lo = lambda x: (x - x.astype(F)).astype(F)  # noqa: E731
    d = (hi(r) - hi(wA)) + (lo(r) - lo(wA))
    beta = v / C
    ref = (beta * (1.0 + rng.normal(size=beta.shape) * 1e-4)).astype(np.float64)
    db = (beta - ref).astype(F)
    bref = ref.astype(F)
    b1 = bref + db
    ct = C * (0.0 - tA)
    L1 = ct.astype(F)
    L1lo = (ct - L1).astype(F)
    icdt = (1.0 / (C * (tB - tA))).astype(F)
    ig2, g2 = (1.0 / gamma ** 2).astype(F), (gamma ** 2).astype(F)
    one = np.ones_like(L1)[:, None]
    p = fma(-b1, L1lo[:, None] * one, fma(-db, L1[:, None] * one, fma(-bref, L1[:, None] * one, d)))
    pv, pp = dot3(p, b1), dot3(p, p)
    Dh = fma(pp, ig2, pv * pv)
    sq = Dh * ulp(1.0 / np.sqrt(Dh))
    s = sq + np.abs(pv)
    tau = np.where(pv >= 0, s * g2, pp * ulp(1.0 / s)).astype(F)
    f = (L1 - tau) * icdt
    dv = wB - wA - v * (tB - tA)[:, None]
    dev = (np.sqrt((dv * dv).sum(1)) * 1.0301 * (1 + 4 * U)).astype(F)
    return fma(-f, sq, sq) > (tau * icdt) * fma(margin * np.ones_like(L1), L1, dev)


def p_true(r, w, t):
    """P of a node at w, time t (present 0): (c t)^2 <= |r - w|^2 in exact arithmetic, and its relative margin."""
    out = np.empty(len(t))
    for k in range(len(t)):
        d2 = sum((Fraction(float(a)) - Fraction(float(b))) ** 2 for a, b in zip(r[k], w[k]))
        L2 = (Fraction(C) * Fraction(float(t[k]))) ** 2
        out[k] = float((d2 - L2) / L2)
    return out


@pytest.mark.parametrize("near", [1e-8, 1e-6, 1e-5, 1e-3])
def test_accepted_pairs_have_a_true_newer_node(near):
    rng = np.random.default_rng(int(-np.log10(near)))
    x = cases(rng, 4000, near)
    ok = accepts(rng, *x, MARGIN)
    r, wA, wB, v, tA, tB, gamma = x
    ok &= ((r - wA) ** 2).sum(1) < (C * tA) ** 2  # the kernel asks only with P(A) false
    m = p_true(r[ok], wB[ok], tB[ok])
    assert np.all(m > 4 * U * 2), m.min()  # true, by more than the FP64 node test's rounding


def test_pairs_inside_the_bracket_are_accepted():
    rng = np.random.default_rng(11)
    r, wA, wB, v, tA, tB, gamma = cases(rng, 4000, 0.0)
    # the retarded time in the middle of the bracket: on A's line halfway between the nodes
    mid, tm = 0.5 * (wA + wB), 0.5 * (tA + tB)
    nh = rng.normal(size=mid.shape)
    nh /= np.linalg.norm(nh, axis=1)[:, None]
    r = mid + nh * (-C * tm)[:, None]
    wB = wA + v * (tB - tA)[:, None]
    sel = gamma < 5.0
    ok = accepts(rng, r, wA, wB, v, tA, tB, gamma, MARGIN)
    assert ok[sel].mean() > 0.98


def test_without_margin_wrong_pairs_would_pass():
    rng = np.random.default_rng(12)
    x = cases(rng, 4000, 1e-7)
    ok = accepts(rng, *x, F(0.0))
    r, wA, wB, v, tA, tB, gamma = x
    ok &= ((r - wA) ** 2).sum(1) < (C * tA) ** 2
    assert np.any(p_true(r[ok], wB[ok], tB[ok]) < 0)
