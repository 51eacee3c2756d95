"""The walk's short form of its geometric tests against the interval form.

For a group whose box sides are in [1, 2^29) grid units and a prune distance
below 2^29, the walk takes gaps as signed differences (csrc/og_walk.cu,
classify_short).  The CPU test repeats both forms in integers and compares every
decision, with record centres placed at the edges of the box, of the cell and of
the far side of the circle.  The GPU test compares interaction counts and
accelerations with the oracle where a launch mixes both forms: groups of one
particle or flat on an axis (interval form) beside ordinary ones, and cutoffs on
either side of an eighth of the box.
"""
from __future__ import annotations

import numpy as np
import pytest

import og_inputs as gi
import oracle
from paper_2609_17658_gb300 import build as B
from paper_2609_17658_gb300 import og

from parity import check_accel

M = 2 ** 32


def _s32(x):
    return (x + 2 ** 31) % M - 2 ** 31


def _point_gap(c, lo, length):
    d = (c - lo) % M
    return np.where(d <= length, 0, np.minimum((d - length) % M, (-d) % M))


def _box_gap(alo, la, blo, lb):
    meet = ((blo - alo) % M <= la) | ((alo - blo) % M <= lb)
    return np.where(meet, 0, np.minimum((blo - (alo + la)) % M, (alo - (blo + lb)) % M))


@pytest.mark.parametrize("seed", range(8))
def test_short_form_takes_the_interval_form_decisions(seed):
    rng = np.random.default_rng(seed)
    n = 100_000
    lev = rng.integers(1, 22, n)
    particle = rng.random(n) < 0.3
    s2 = np.where(particle, 0, 0x80000000 >> lev)
    mask = np.where(particle, 0, 0xffffffff >> lev)
    blim = np.where(particle, 0, 0x99999999 >> lev)
    assert np.array_equal(blim, 6 * s2 // 5)
    length = np.clip((rng.random((3, n)) * 2.0 ** rng.integers(0, 30, (3, n))).astype(np.int64), 1, 2 ** 29 - 1)
    lo = rng.integers(0, M, (3, n))
    hi = (lo + length) % M
    edge = rng.integers(-3, 4, (3, n))
    off = np.choose(rng.integers(0, 4, (3, n)),
                    [rng.integers(0, M, (3, n)), length + edge, 2 ** 31 + edge + length * rng.integers(0, 2, (3, n)),
                     rng.integers(-4, 5, (3, n)) * (0x80000000 >> lev) + edge])
    c = (lo + off) % M
    # squared distances as exact integers (numpy objects would be slow: two float64 halves are not needed,
    # the sums stay below 2^63 for every value that can decide)
    rprune = ((2.0 ** rng.uniform(10, 28.99, n)) ** 2).astype(np.int64)
    isn = (~particle).astype(np.int64)
    cap = 2 ** 30                       # gaps above this are beyond any prune distance here
    g2, e2 = np.zeros(n, np.int64), np.zeros(n, np.int64)
    far_side = np.full(n, -2 ** 40)
    near = np.ones(n, bool)
    com_equal = np.ones(n, bool)
    for k in range(3):
        cc = (c[k] & ~mask) | s2
        a, d = _s32(lo[k] - cc), _s32(cc - hi[k])
        far_side = np.maximum(far_side, np.maximum(a, d))
        gap = np.maximum(np.maximum(_s32(d - isn), a) + isn - s2, 0)
        exact = np.where(particle, _point_gap(cc, lo[k], length[k]),
                         _box_gap(lo[k], length[k], (cc - s2) % M, np.maximum(2 * s2 - 1, 0)))
        g2 += np.minimum(gap, cap) ** 2
        e2 += np.minimum(exact, cap) ** 2
        near &= _point_gap(cc, lo[k], length[k]) <= blim
        com = np.maximum(np.maximum(_s32(lo[k] - c[k]), _s32(c[k] - hi[k])), 0)
        com_equal &= com == _point_gap(c[k], lo[k], length[k])
    keep = e2 <= rprune
    assert np.array_equal(g2 <= rprune, keep)
    node = keep & ~particle
    assert np.array_equal((far_side <= blim)[node], near[node])
    # the opening test reads the gap of the centre of mass where the boundary check
    # leaves it open; level 1 takes the exact branch
    assert com_equal[node & ~near & (lev > 1)].all()
    assert com_equal[keep & particle].all()


@pytest.mark.parametrize("seed", range(4))
def test_short_form_of_refitted_extents(seed):
    rng = np.random.default_rng(100 + seed)
    n = 200_000
    length = np.clip((rng.random((3, n)) * 2.0 ** rng.integers(0, 30, (3, n))).astype(np.int64), 1, 2 ** 29 - 1)
    ext = np.minimum((rng.random((3, n)) * 2.0 ** rng.integers(0, 31, (3, n))).astype(np.int64), 2 ** 30 - 1)
    lo = rng.integers(0, M, (3, n))
    hi = (lo + length) % M
    edge = rng.integers(-3, 4, (3, n))
    off = np.choose(rng.integers(0, 4, (3, n)),
                    [rng.integers(0, M, (3, n)), length + edge, edge - ext, 2 ** 31 + edge + length * rng.integers(0, 2, (3, n))])
    s = (lo + off) % M
    side = ext.max(axis=0) + 1
    blim = 3 * side // 5
    high = ((3 * side).astype(np.uint64) * np.uint64(0xCCCCCCCD)) >> np.uint64(32)
    assert np.array_equal((high >> np.uint64(2)).astype(np.int64), blim)
    rprune = ((2.0 ** rng.uniform(10, 28.99, n)) ** 2).astype(np.int64)
    cap = 2 ** 30
    g2, e2 = np.zeros(n, np.int64), np.zeros(n, np.int64)
    dc, near = np.full(n, -2 ** 40), np.ones(n, bool)
    for k in range(3):
        gap = np.maximum(np.maximum(_s32(lo[k] - (s[k] + ext[k])), _s32(s[k] - hi[k])), 0)
        g2 += np.minimum(gap, cap) ** 2
        e2 += np.minimum(_box_gap(lo[k], length[k], s[k], ext[k]), cap) ** 2
        cc = (s[k] + (ext[k] + 1 >> 1)) % M
        dc = np.maximum(dc, np.maximum(_s32(lo[k] - cc), _s32(cc - hi[k])))
        near &= _point_gap(cc, lo[k], length[k]) <= blim
    keep = e2 <= rprune
    assert np.array_equal(g2 <= rprune, keep)
    assert np.array_equal((dc <= blim)[keep], near[keep])


@pytest.fixture(scope="module")
def ctx():
    B.build()
    oracle.build()
    c = og.Context(0)
    yield c
    c.close()


@pytest.mark.gpu
@pytest.mark.parametrize("rcut", [0.03, 0.1249, 0.1251, 0.4])
@pytest.mark.parametrize("n,kind", [(1, "uniform"), (2, "uniform"), (3, "uniform"), (33, "uniform"), (65, "uniform"),
                                    (1000, "halo"), (3001, "plane"), (4096, "lattice")])
def test_walk_with_both_forms_against_the_oracle(ctx, n, kind, rcut):
    if kind == "lattice":
        pos, mass = gi.lattice(16, offset=0.25)
        mass = mass * np.random.default_rng(5).uniform(0.5, 2.0, n)
    else:
        pos, mass = (gi.halo_mix if kind == "halo" else gi.uniform)(n, 11)
        if kind == "plane":
            pos[: n // 2, 2] = 0.25          # groups flat on one axis
    for opening in (gi.OPEN_BH, gi.OPEN_REL):
        prm = gi.default_params(eps=0.002, r_s=rcut / 4.5, opening=opening, alpha=0.002, theta=0.7)
        a_old = np.random.default_rng(3).normal(size=(n, 3)).astype(np.float32)
        gt, ot = og.Tree(ctx, pos, mass, prm), oracle.Tree(pos, mass, prm)
        acc, npp, npn = gt.force(a_old=a_old)
        ref, rpp, rpn = ot.force(a_old=a_old)
        assert np.array_equal(npp, rpp) and np.array_equal(npn, rpn)
        check_accel(acc, ref)
        gt.free()
