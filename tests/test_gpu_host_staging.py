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


def _status_of_device_arrays(ctx, n, outputs):
    """Status of a build (or of a force call's outputs) that is given device memory in a
    host-pointer call, and the forces if it took it."""
    import ctypes as C

    import torch
    pos, mass = gi.uniform(n, 7)
    prm = og.params_from_dict(gi.default_params(eps=1e-3, r_s=0.02, opening=gi.OPEN_BH))
    dpos, dmass = torch.from_numpy(pos).cuda(), torch.from_numpy(mass).cuda()
    dacc = torch.zeros((n, 3), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    h, acc = C.c_void_p(), np.zeros((n, 3), np.float32)
    src = (pos.ctypes.data, mass.ctypes.data) if outputs else (dpos.data_ptr(), dmass.data_ptr())
    st = og.lib().og_tree_build(ctx.h, C.c_void_p(src[0]), C.c_void_p(src[1]), n, C.byref(prm), C.byref(h))
    if st != og.OG_OK:
        return st, None
    dst = dacc.data_ptr() if outputs else acc.ctypes.data
    st = og.lib().og_tree_force(h, None, C.c_void_p(dst), None, None)
    og.og_tree_free(h)
    torch.cuda.synchronize()
    return st, dacc.cpu().numpy() if outputs else acc


@pytest.mark.parametrize("outputs", [False, True])
def test_device_arrays_in_a_host_call(outputs):
    """The host's own copies of small arrays must not touch device memory: a call that
    is given it answers as it does for large arrays, which are copied by CUDA."""
    B.build()
    with og.Context(0) as ctx:
        large, _ = _status_of_device_arrays(ctx, 40000, outputs)
        small, got = _status_of_device_arrays(ctx, 4096, outputs)
        assert small == large
        pos, mass = gi.uniform(4096, 7)
        want, _, _ = og.Tree(ctx, pos, mass, gi.default_params(eps=1e-3, r_s=0.02, opening=gi.OPEN_BH)).force()
        if small == og.OG_OK:
            assert np.array_equal(got, want)
