"""Calls of every kind on one context, in orders that hand the walk's counters from one
call to the next: the build's and the force call's last kernels leave them at zero, the
other calls do not, and a walk clears them where they may not be.  Every result and
interaction count is bitwise that of the same call on a fresh context.
"""
from __future__ import annotations

import numpy as np
import pytest

import og_inputs as gi
from paper_2609_17658_gb300 import build as B
from paper_2609_17658_gb300 import og

pytestmark = pytest.mark.gpu


def _tree(ctx, rel, flags=0):
    pos, mass, prm = gi.config("clustered-2m", n=4000)
    prm = dict(prm, r_s=0.015, opening=gi.OPEN_REL if rel else gi.OPEN_BH, flags=flags)
    return og.Tree(ctx, pos, mass, prm)


def _call(kind, t, rel, seed):
    """(results, interactions) of one call"""
    n = t.n
    r = np.random.default_rng(seed)
    if kind == "force":
        out = t.force()
    elif kind == "aold":
        out = t.force(a_old=r.normal(size=(n, 3)).astype(np.float32)) if rel else t.force()
    elif kind == "pot":
        out = t.force_pot()
    elif kind == "f64":
        out = (np.zeros((n, 3)), np.zeros(n, np.uint32), np.zeros(n, np.uint32))
        og.og_tree_force_f64(t.h, out[0], None, out[1], out[2])
    elif kind == "active":
        out = (np.zeros((n, 3), np.float32), np.zeros(n, np.uint32), np.zeros(n, np.uint32))
        og.og_tree_force_active(t.h, (r.random(n) < 0.3).astype(np.uint8), out[0], None, out[1], out[2])
    else:
        raise AssertionError(kind)
    return [np.asarray(x) for x in out if x is not None], t.info()["interactions"]


ORDERS = [("force", "force", "active", "force"), ("active", "force", "pot", "aold"),
          ("f64", "force", "f64", "pot", "force"), ("aold", "active", "active", "pot", "f64", "force")]


@pytest.mark.parametrize("rel", [False, True])
@pytest.mark.parametrize("flags", [0, og.OG_DEBUG_DUMP_LISTS])
@pytest.mark.parametrize("order", ORDERS)
def test_orders(rel, flags, order):
    B.build()
    ctx = og.Context(0)
    t = _tree(ctx, rel, flags)
    for k, kind in enumerate(order):
        got, inter = _call(kind, t, rel, k)
        fresh = og.Context(0)
        ft = _tree(fresh, rel, flags)
        want, winter = _call(kind, ft, rel, k)
        assert inter == winter and inter > 0
        for a, b in zip(got, want):
            assert np.array_equal(a, b)
        fresh.close()
    ctx.close()
