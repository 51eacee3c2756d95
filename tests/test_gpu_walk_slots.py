"""Slots of groups walked in parts (csrc/og_walk.cu, Parts): a group that finds no slot
walks its parts in its own warp.  Which groups those are depends on the timing, so
repeated calls have the same bits only if both ways give them; a subset of a few groups
finds slots for all.  And the scratch of a pass does not grow with the number of groups."""
from __future__ import annotations

import ctypes as C

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


@pytest.mark.parametrize("n,group_max", [(9001, 32), (9001, 5), (8192, 1), (8193, 1), (16001, 1)])
def test_with_and_without_a_slot(ctx, n, group_max):
    """Every group's list spans a third of the box, so nearly all leave parts: up to 8192
    groups find slots, a half of 16,001 groups do not."""
    pos, mass = gi.uniform(n, 17)
    prm = gi.default_params(eps=0.002, r_s=0.1, opening=gi.OPEN_REL, alpha=1e-9, group_max=group_max)
    a_old = np.random.default_rng(2).normal(size=(n, 3)).astype(np.float32)
    t = og.Tree(ctx, pos, mass, prm)
    acc, npp, npn = t.force(a_old=a_old)
    assert t.info()["groups"] > 128
    accp, _, _, pot = t.force_pot(a_old=a_old)
    _, _, _, pot2 = t.force_pot(a_old=a_old)
    assert np.array_equal(pot, pot2)
    for _ in range(3):
        again, pp, pn = t.force(a_old=a_old)
        assert np.array_equal(again, acc) and np.array_equal(pp, npp) and np.array_equal(pn, npn)
    assert np.array_equal(accp, acc)
    r = np.random.default_rng(3)
    for _ in range(4):
        on = np.zeros(n, np.uint8)
        on[r.choice(n, 10, replace=False)] = 1
        out, cnt = np.zeros((n, 3), np.float32), np.zeros(n, np.uint32)
        og.og_tree_force_active(t.h, on, out, a_old, cnt)
        assert np.array_equal(out[on > 0], acc[on > 0]) and np.array_equal(cnt[on > 0], npp[on > 0])
    ot = oracle.Tree(pos, mass, prm)
    ref, rpp, rpn = ot.force(a_old=a_old, groups=np.arange(0, t.info()["groups"], 32))
    on = np.isfinite(ref[:, 0])
    assert np.array_equal(npp[on], rpp[on]) and np.array_equal(npn[on], rpn[on])
    parity.check_accel(acc[on], ref[on])
    t.free()


def test_scratch_of_a_pass_is_bounded(ctx):
    """Groups of one particle: 60,000 groups.  A place of 3 KB for each would take 190 MB;
    8192 slots, the warps' own places, the staged arrays and the order of the groups
    take 15, 5, 2 and some 2 MB."""
    n = 60000
    pos, mass = gi.halo_mix(n, 5, n_halo=60)
    side = n ** (1.0 / 3.0)
    prm = gi.default_params(eps=1 / (50 * side), r_s=1.25 / (2 * side), opening=gi.OPEN_REL, alpha=0.002, group_max=1)
    a_old = np.random.default_rng(2).normal(size=(n, 3)).astype(np.float32)
    cudart = None
    for name in ("libcudart.so.13", "libcudart.so"):
        try:
            cudart = C.CDLL(name)
            break
        except OSError:
            continue
    if cudart is None:
        pytest.skip("no shared CUDA runtime to ask for the memory pool's high-water mark")
    used_current, used_high = 7, 8                    # cudaMemPoolAttrUsedMemCurrent, UsedMemHigh
    pool, v = C.c_void_p(), C.c_uint64(0)
    assert cudart.cudaDeviceGetDefaultMemPool(C.byref(pool), 0) == 0
    t = og.Tree(ctx, pos, mass, prm)
    assert t.info()["groups"] == n
    for _ in range(2):                                # the second call orders the groups
        assert cudart.cudaMemPoolGetAttribute(pool, used_current, C.byref(v)) == 0
        before = v.value
        v.value = 0
        assert cudart.cudaMemPoolSetAttribute(pool, used_high, C.byref(v)) == 0
        t.force(a_old=a_old)
        assert cudart.cudaMemPoolGetAttribute(pool, used_high, C.byref(v)) == 0
        assert v.value - before < 48 << 20, (v.value, before)
    t.free()
