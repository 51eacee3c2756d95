"""Groups whose walk is split into parts (csrc/og_walk.cu, kQuota): the relative
criterion with small previous accelerations gives lists of thousands of entries,
far above the 48 rounds of 64 records after which a walk is split.  Lists,
counts and forces equal the oracle's, and a group's sums do not depend on what
else the launch holds: an active subset, a batch and the potential call give the
same bits.  The sizes are the ends of the range in which walks are split."""
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


def _case(n, dist="halo"):
    pos, mass = gi.halo_mix(n, 31, n_halo=max(1, n // 1000)) if dist == "halo" else gi.uniform(n, 31)
    side = n ** (1.0 / 3.0)
    prm = gi.default_params(eps=1 / (50 * side), r_s=min(1.25 / side, 0.08), opening=gi.OPEN_REL, alpha=0.002)
    a_old = (np.random.default_rng(7).normal(size=(n, 3)) * 0.05).astype(np.float32)
    return pos, mass, prm, a_old


@pytest.mark.parametrize("n", [2048, 2049, 30011, 196608, 196609])
def test_split_walks_against_the_oracle(ctx, n):
    pos, mass, prm, a_old = _case(n)
    gt, ot = og.Tree(ctx, pos, mass, prm), oracle.Tree(pos, mass, prm)
    acc, npp, npn = gt.force(a_old=a_old)
    assert n < 30000 or int((npp + npn).max()) > 64 * 48          # some walks are split
    sel = None if n < 40000 else np.sort(np.argsort(-(npp + npn)[ot.get(oracle.F_PERM)][ot.get(oracle.F_GBEG)])[:200])
    ref, rpp, rpn = ot.force(a_old=a_old) if sel is None else ot.force(a_old=a_old, groups=sel)
    on = np.isfinite(ref[:, 0])
    assert np.array_equal(npp[on], rpp[on]) and np.array_equal(npn[on], rpn[on])
    parity.check_accel(acc[on], ref[on])
    gt.free()


def test_split_walks_do_not_depend_on_the_launch(ctx):
    pos, mass, prm, a_old = _case(30011)
    n = len(mass)
    t = og.Tree(ctx, pos, mass, prm)
    acc, npp, npn = t.force(a_old=a_old)
    again, _, _ = t.force(a_old=a_old)
    assert np.array_equal(again, acc)
    acc_p, npp_p, _, _ = t.force_pot(a_old=a_old)
    assert np.array_equal(acc_p, acc) and np.array_equal(npp_p, npp)
    on = np.random.default_rng(3).random(n) < 0.01
    out, cnt = np.zeros((n, 3), np.float32), np.zeros(n, np.uint32)
    og.og_tree_force_active(t.h, on.astype(np.uint8), out, a_old, cnt)
    assert np.array_equal(out[on], acc[on]) and np.array_equal(cnt[on], npp[on])
    other = _case(5003, "uniform")
    boxes = [dict(pos=q[0], mass=q[1], params=q[2], a_old=q[3], acc=np.zeros((len(q[1]), 3), np.float32),
                  n_pp=np.zeros(len(q[1]), np.uint32), n_pn=np.zeros(len(q[1]), np.uint32))
             for q in (other, (pos, mass, prm, a_old))]
    og.og_batch_force(ctx.h, boxes)
    assert np.array_equal(boxes[1]["acc"], acc) and np.array_equal(boxes[1]["n_pn"], npn)
    t.free()
