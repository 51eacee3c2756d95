"""The one-launch sort of up to 65536 keys (csrc/og_sort.cu): sorted keys and permutation of
a build against a stable numpy argsort of the same Morton keys, at the edges of its
slices and rounds and one past them, with digits that all keys share (passes that
move nothing: the lowest, the highest, a middle one, all of them).
"""
from __future__ import annotations

import numpy as np
import pytest

import og_inputs as gi
from paper_2609_17658_gb300 import build as B
from paper_2609_17658_gb300 import og

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    B.build()
    c = og.Context(0)
    yield c
    c.close()


def _morton(pos):
    q = np.floor(pos * 2.0 ** 32).astype(np.uint64) >> np.uint64(11)      # 21 bits per axis
    key = np.zeros(len(pos), np.uint64)
    for b in range(21):
        for a in range(3):
            key |= ((q[:, a] >> np.uint64(b)) & np.uint64(1)) << np.uint64(3 * b + 2 - a)
    return key


def _positions(layout, n):
    pos = np.random.default_rng(n).random((n, 3))
    if layout == "lattice":            # the low digits are 0 for every key, many keys equal
        pos = np.floor(pos * 32) / 32
    elif layout == "corner":           # the top digits are shared
        pos = 0.626 + pos * 2.0 ** -8
    elif layout == "middle":           # digits in the middle are 0
        pos = np.floor(pos * 64) / 64 + np.floor(pos * 64) * 2.0 ** -21
    elif layout == "same":
        pos = np.tile([[0.3, 0.6, 0.9]], (n, 1))
    return pos


@pytest.mark.parametrize("n", [2, 33, 511, 1025, 16383, 16384, 16385, 32769, 49153, 65535, 65536, 65537])
@pytest.mark.parametrize("layout", ["spread", "lattice", "corner", "middle", "same"])
def test_sorted_like_a_stable_argsort(ctx, layout, n):
    if layout == "same" and n > 2000:
        n = 2000 + n % 7
    pos = _positions(layout, n)
    t = og.Tree(ctx, pos, np.full(n, 1.0 / n), gi.default_params(eps=1e-3, r_s=0.01))
    key = _morton(pos)
    order = np.argsort(key, kind="stable")
    assert np.array_equal(t.export(og.OG_F_PERM), order)
    assert np.array_equal(t.export(og.OG_F_SKEY), key[order])
    t.free()
