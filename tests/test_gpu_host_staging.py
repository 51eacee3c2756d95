"""Host arrays of small calls go through page-locked memory, larger ones are copied
directly (512 KB: 16384 particles in, 26214 out): results on both sides of both lines
are bitwise those of device arrays, with and without the counts, also when calls on
two contexts and trees follow each other on the same host arrays.
"""
from __future__ import annotations

import numpy as np
import pytest

import og_inputs as gi
from paper_2609_17658_gb300 import build as B
from paper_2609_17658_gb300 import og

pytestmark = pytest.mark.gpu


def _device_result(ctx, pos, mass, prm, a_old):
    import torch
    n = len(pos)
    acc = torch.zeros((n, 3), dtype=torch.float32, device="cuda")
    npp, npn = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    h = og.og_tree_build(ctx.h, torch.from_numpy(pos).cuda(), torch.from_numpy(mass).cuda(), prm)
    og.og_tree_force(h, acc, None if a_old is None else torch.from_numpy(a_old).cuda(), npp, npn)
    og.og_tree_free(h)
    return acc.cpu().numpy(), npp.cpu().numpy().view(np.uint32), npn.cpu().numpy().view(np.uint32)


@pytest.mark.parametrize("n", [1, 3, 4096, 16383, 16384, 16385, 26214, 26215])
@pytest.mark.parametrize("rel", [False, True])
def test_host_arrays_equal_device_arrays(n, rel):
    B.build()
    pos, mass = gi.uniform(n, 7)
    prm = gi.default_params(eps=1e-3, r_s=0.02)
    prm = dict(prm, opening=gi.OPEN_REL if rel else gi.OPEN_BH)
    a_old = np.random.default_rng(n).normal(size=(n, 3)).astype(np.float32) if rel else None
    one, two = og.Context(0), og.Context(0)
    want = _device_result(one, pos, mass, prm, a_old)
    other = np.ascontiguousarray(pos[::-1]), np.ascontiguousarray(mass[::-1])
    t1, t2 = og.Tree(one, pos, mass, prm), og.Tree(two, *other, prm)
    got = t1.force(a_old=a_old)
    t2.force(a_old=None if a_old is None else np.ascontiguousarray(a_old[::-1]))
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
    again, none_pp, none_pn = t1.force(a_old=a_old, counts=False)
    assert none_pp is None and none_pn is None and np.array_equal(again, want[0])
    t1.free()
    t2.free()
    one.close()
    two.close()
