"""The FP32 decision bands of the 2-opt and 3-opt hold with the approximate square root.

The searches decide most moves from FP32 estimates of the FP64 gain: distances
from sqrt.approx (at most 2^-23 off, relatively) or FP64 distances rounded once,
four terms in the 2-opt, six in the 3-opt, and a band of 4e-6 times the terms'
sum (plus 1e-18) inside which FP64 decides.  This restates the rule with numpy
float32 operations, taking any value that the root's bound allows, and checks on
millions of candidate moves that

  * each distance is within 5 units of 2^-24 of the FP64 one,
  * "certainly not improving" never meets an FP64 gain above 1e-10 and
    "certainly improving" none at or below it, and likewise for the partial
    gains g1 and g2,
  * the moves the 3-opt's scan leaves out as null (they add the edges they remove)
    have FP64 gains below 1e-10,

on point sets that stress it: lattices (gains exactly zero), tiny and large
scales, near-duplicates and duplicates.
"""
import numpy as np
import pytest

from test_two_opt_fp32_rule import F, G1_LO, LS_GAIN, d64, gain_class, point_sets

BAND = F(4e-6)
U = 2.0 ** -24


def d32_approx(rng, p, q):
    """FP32 distances, each root anywhere within 2^-23 of the exact root of its FP32 argument."""
    dx = q[:, 0] - p[:, 0]
    dy = q[:, 1] - p[:, 1]
    root = np.sqrt((dx * dx + dy * dy).astype(np.float64))
    e = rng.choice([-1.0, 1.0, 0.0], len(root)) * rng.choice([1.0, 0.5], len(root))
    v = (root * (1.0 + e * 2 * U)).astype(F)
    over = np.abs(v.astype(np.float64) - root) > root * 2 * U      # rounded past the bound: one step back
    return np.where(over, np.nextafter(v, root.astype(F)), v)


def gain_class6(g2, mag2, d56, d61):
    est = (g2 + d56) - d61
    tol = BAND * (mag2 + (d56 + d61)) + F(1e-18)
    return np.where(~(est > F(LS_GAIN) - tol), 0, np.where(est > F(LS_GAIN) + tol, 2, 1))


@pytest.mark.parametrize("name,pts", list(point_sets()), ids=[n for n, _ in point_sets()])
def test_two_opt_classes(name, pts):
    rng = np.random.default_rng(17)
    m = 1_000_000
    a, an, b, bn = (pts[rng.integers(0, len(pts), m)] for _ in range(4))
    Da, Dab, Dbb, Dn = d64(a, an), d64(a, b), d64(b, bn), d64(an, bn)
    da, dbb, dn = d32_approx(rng, a, an), d32_approx(rng, b, bn), d32_approx(rng, an, bn)
    for x32, x64 in ((da, Da), (dbb, Dbb), (dn, Dn)):
        ok = x64 > 1e-17
        assert np.abs(x32[ok].astype(np.float64) / x64[ok] - 1.0).max() <= 5 * U, name
    dab = Dab.astype(F)
    gain = ((Da - Dab) + Dbb) - Dn
    c = gain_class(da, dab, dbb, dn)
    assert not np.any((c == 0) & (gain > LS_GAIN)), name
    assert not np.any((c == 2) & ~(gain > LS_GAIN)), name
    assert not np.any((da * G1_LO > dab) & ~(Da > Dab)), name
    assert not np.any(~(da > dab * G1_LO) & (Da > Dab)), name


@pytest.mark.parametrize("name,pts", list(point_sets()), ids=[n for n, _ in point_sets()])
def test_three_opt_classes(name, pts):
    rng = np.random.default_rng(19)
    m = 1_000_000
    t1, t2, t3, t4, t5, t6 = (pts[rng.integers(0, len(pts), m)] for _ in range(6))
    # a third of the moves with t4 = t2 or t5 = t1: the terms cancel
    k = m // 6
    t4[:k], t5[k:2 * k] = t2[:k], t1[k:2 * k]
    D12, D23, D34, D45, D56, D61 = (d64(*e) for e in ((t1, t2), (t2, t3), (t3, t4), (t4, t5), (t5, t6), (t6, t1)))
    d12, d34, d56, d61 = (d32_approx(rng, *e) for e in ((t1, t2), (t3, t4), (t5, t6), (t6, t1)))
    d23, d45 = D23.astype(F), D45.astype(F)
    G2 = ((D12 - D23) + D34) - D45
    gain = (G2 + D56) - D61
    g2 = ((d12 - d23) + d34) - d45
    mag2 = ((d12 + d23) + d34) + d45
    c = gain_class6(g2, mag2, d56, d61)
    assert not np.any((c == 0) & (gain > LS_GAIN)), name
    assert not np.any((c == 2) & ~(gain > LS_GAIN)), name
    tol2 = BAND * mag2 + F(1e-18)
    assert not np.any(~(g2 > -tol2) & (G2 > 0.0)), name
    assert not np.any((g2 > tol2) & ~(G2 > 0.0)), name
    # closing to t1 after t4: four terms, in the 2-opt's class
    D41, d41 = d64(t4, t1), d32_approx(rng, t4, t1)
    c = gain_class(d12, d23, d34, d41)
    gain4 = ((D12 - D23) + D34) - D41
    assert not np.any((c == 0) & (gain4 > LS_GAIN)), name
    assert not np.any((c == 2) & ~(gain4 > LS_GAIN)), name


def test_null_moves_gain_nothing():
    rng = np.random.default_rng(23)
    x, y, z = 10.0 ** rng.uniform(-12, 3.5, (3, 2_000_000))      # lengths whose sums stay below 1e4
    keep = x + y + y + x + z < 9e3
    x, y, z = x[keep], y[keep], z[keep]
    assert np.abs(((x - y) + y) - x).max() < LS_GAIN                         # t4 = t2
    assert np.abs((((((x - y) + y) - x) + z) - z)).max() < LS_GAIN           # t4 = t2, t5 = t1
