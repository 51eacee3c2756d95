"""FP32 accumulation of the walk, seen where it is all there is: no split (no erfc), no
softening, every node opened, so a target's potential is the sum of m / r over all
particles, terms of one sign.  Each carries the reciprocal square root's error, which
averages out over thousands of them up to a common factor (taken out with the median).
What is left are the roundings of the sums, with u = 2^-24 and 0.42 u the rms of one
rounding relative to its result:
* the result's own, 0.42 u;
* of plain sums over q terms, L / q of them in L terms: 0.42 u q / sqrt(3 L).
Sums of chunks, of replicas and of parts carry compensations and add less.
"""
from __future__ import annotations

import numpy as np
import pytest

import og_inputs as gi
import oracle
from paper_2609_17658_gb300 import build as B
from paper_2609_17658_gb300 import og
from tests import parity

pytestmark = pytest.mark.gpu
ONE = 0.42 * 2.0 ** -24


@pytest.fixture(scope="module")
def ctx():
    B.build()
    oracle.build()
    c = og.Context(0)
    yield c
    c.close()


def _exact(pos, mass):
    q = np.floor(pos * 2.0 ** 32).astype(np.int64)
    pot = np.zeros(len(q))
    for i in range(0, len(q), 250):
        d = (q[None, :] - q[i:i + 250, None] + 2 ** 31) % 2 ** 32 - 2 ** 31
        r = np.sqrt(((d * 2.0 ** -32) ** 2).sum(2))
        pot[i:i + 250] = -(mass[None, :] / np.where(r > 0, r, np.inf)).sum(1)
    return pot


def _error(pot, ref):
    e = pot.astype(np.float64) / ref - 1.0
    return e - np.median(e)


def _rms(e):
    return float(np.sqrt((e ** 2).mean()))


def _params(**kw):
    return gi.default_params(eps=0.0, r_s=0.0, group_max=32, **kw)


def test_parts_add_no_rounding(ctx):
    """The relative criterion's walk in eight parts (every group leaves, with a slot or
    without) against the Barnes-Hut walk of the same particles in one: plain sums of
    the parts' rounded totals would add 1.8 x 0.42 u to its 1.1 x 0.42 u."""
    e = {}
    for seed in range(3):
        n = 4001
        pos, mass = gi.uniform(n, seed)
        ref = _exact(pos, mass)
        for opening in (gi.OPEN_BH, gi.OPEN_REL):
            t = og.Tree(ctx, pos, mass, _params(opening=opening, theta=0.0, alpha=0.0))
            _, npp, npn, pot = t.force_pot(a_old=np.ones((n, 3), np.float32))
            assert (npp == n - 1).all() and (npn == 0).all()
            e.setdefault(opening, []).append(_error(pot, ref))
            t.free()
    whole, parts = (_rms(np.concatenate(e[o])) for o in (gi.OPEN_BH, gi.OPEN_REL))
    assert parts <= 1.1 * whole, (parts / ONE, whole / ONE)


def test_plain_sums_stay_within_half_a_chunk(ctx):
    """Groups of 31 and 32 targets (two replicas) at the default chunk of 256 entries: the
    error of plain sums over at most 128 terms."""
    n, e = 2000, []
    for seed in range(6):
        pos, mass = gi.uniform(n, 40 + seed)
        t = og.Tree(ctx, pos, mass, _params(opening=gi.OPEN_BH, theta=0.0, walk_chunk=256))
        _, npp, _, pot = t.force_pot()
        assert (npp == n - 1).all()
        beg, end, perm = t.export(og.OG_F_GBEG), t.export(og.OG_F_GEND), t.export(og.OG_F_PERM)
        full = np.concatenate([perm[b:f] for b, f in zip(beg, end) if f - b >= 31])
        assert len(full) > n // 4
        e.append(_error(pot, _exact(pos, mass))[full])
        t.free()
    limit = ONE * np.sqrt(1.0 + 128 ** 2 / (3.0 * n))
    assert _rms(np.concatenate(e)) <= limit, (_rms(np.concatenate(e)) / ONE, limit / ONE)


@pytest.mark.parametrize("walk_chunk", [64, 65, 191, 192, 321, 1024])
@pytest.mark.parametrize("group_max", [1, 2, 3])
def test_small_groups_at_the_edges_of_a_chunk(ctx, group_max, walk_chunk):
    """One pair of targets takes 32 replicas, whose padding ends at the chunk's last
    entries; a softening wide enough that near entries fill their chunk too."""
    n = 3000
    pos, mass = gi.halo_mix(n, 9, n_halo=4)
    prm = gi.default_params(eps=0.02, r_s=0.08, opening=gi.OPEN_BH, theta=0.2, group_max=group_max,
                            walk_chunk=walk_chunk)
    t, ot = og.Tree(ctx, pos, mass, prm), oracle.Tree(pos, mass, prm)
    acc, npp, npn = t.force()
    ref, rpp, rpn = ot.force()
    assert np.array_equal(npp, rpp) and np.array_equal(npn, rpn)
    parity.check_accel(acc, ref)
    t.free()
