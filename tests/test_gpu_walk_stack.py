"""Walks that open so much of a tree that the stack of child ranges fills up
(csrc/og_walk.cu, kStackSafe): rounds are undone and taken again with fewer ranges.
Lists, counts and forces of a few groups against the oracle."""
from __future__ import annotations

import numpy as np
import pytest

import og_inputs as gi
import oracle
from paper_2609_17658_gb300 import build as B
from paper_2609_17658_gb300 import og
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    B.build()
    oracle.build()
    c = og.Context(0)
    yield c
    c.close()


def _check(t, ot, active, a_old=None):
    """The groups of the active particles, all of their members against the oracle."""
    n = len(active)
    acc, npp, npn = np.zeros((n, 3), np.float32), np.zeros(n, np.uint32), np.zeros(n, np.uint32)
    beg, end, perm = t.export(og.OG_F_GBEG), t.export(og.OG_F_GEND), t.export(og.OG_F_PERM)
    groups = [g for g, (b, e) in enumerate(zip(beg, end)) if active[perm[b:e]].any()]
    for g in groups:
        active[perm[beg[g]:end[g]]] = 1
    og.og_tree_force_active(t.h, active, acc, a_old, npp, npn)
    ref, rpp, rpn = ot.force(a_old=a_old, groups=np.array(groups))
    on = active > 0
    assert np.array_equal(npp[on], rpp[on]) and np.array_equal(npn[on], rpn[on])
    parity.check_accel(acc[on], ref[on])


@pytest.mark.parametrize("opening", [gi.OPEN_BH, gi.OPEN_REL])
@pytest.mark.parametrize("r_s", [0.0, 0.1])
def test_every_node_opened(ctx, opening, r_s):
    n = 150_001                                      # within the sizes of walks in parts
    pos, mass = gi.halo_mix(n, 23, n_halo=100)
    prm = gi.default_params(eps=1e-3, r_s=r_s, opening=opening, theta=0.0, alpha=0.0)
    a_old = np.ones((n, 3), np.float32) if opening == gi.OPEN_REL else None
    active = np.zeros(n, np.uint8)
    active[np.random.default_rng(1).choice(n, 6, replace=False)] = 1
    t, ot = og.Tree(ctx, pos, mass, prm), oracle.Tree(pos, mass, prm)
    _check(t, ot, active, a_old)
    t.free()


@pytest.mark.parametrize("fraction", [0.001, 0.1])
def test_after_drifts_across_the_box(ctx, fraction):
    n = 100_003
    pos, mass = gi.halo_mix(n, 29, n_halo=50)
    prm = gi.default_params(eps=1e-3, r_s=0.02)
    rng = np.random.default_rng(2)
    new = np.where((rng.random(n) < fraction)[:, None], rng.random((n, 3)), pos)
    t, ot = og.Tree(ctx, pos, mass, prm), oracle.Tree(pos, mass, prm)
    t.refit(new)
    ot.refit(new)
    active = np.zeros(n, np.uint8)
    active[rng.choice(n, 12, replace=False)] = 1
    _check(t, ot, active)
    t.free()
