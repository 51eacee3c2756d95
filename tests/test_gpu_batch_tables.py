"""og_batch_force on device arrays reads and writes each box's own arrays through
a table: the results equal the host call's bit for bit, for one box and several,
boxes of one particle, with and without previous accelerations and counts, and
when the accelerations overwrite the previous ones in place."""
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


@pytest.mark.parametrize("sizes", [(257,), (1, 300, 1), (5000, 4097, 33)])
@pytest.mark.parametrize("opening,given", [(gi.OPEN_BH, False), (gi.OPEN_REL, False), (gi.OPEN_REL, True)])
def test_device_boxes_equal_host_boxes(ctx, sizes, opening, given):
    torch = pytest.importorskip("torch")
    host, dev = [], []
    for k, n in enumerate(sizes):
        pos, mass = gi.uniform(n, 50 + k, box=1.0 + k)
        prm = gi.default_params(eps=0.002, r_s=0.02 * (1 + k), box=1.0 + k, opening=opening)
        b = dict(pos=pos, mass=mass * (1 + k), params=prm, acc=np.zeros((n, 3), np.float32))
        if given:
            b["a_old"] = np.random.default_rng(k).normal(size=(n, 3)).astype(np.float32)
        if k != 1:                      # the second box leaves out its counts
            b.update(n_pp=np.zeros(n, np.uint32), n_pn=np.zeros(n, np.uint32))
        host.append(b)
        d = {q: torch.from_numpy(v.view(np.int32) if v.dtype == np.uint32 else v.copy()).cuda()
             for q, v in b.items() if isinstance(v, np.ndarray)}
        if given:
            d["acc"] = d["a_old"]       # in place
        dev.append(dict(d, params=prm))
    torch.cuda.synchronize()
    og.og_batch_force(ctx.h, host)
    og.og_batch_force(ctx.h, dev)
    torch.cuda.synchronize()
    for h, d in zip(host, dev):
        assert np.array_equal(d["acc"].cpu().numpy(), h["acc"])
        for q in ("n_pp", "n_pn"):
            if q in h:
                assert np.array_equal(d[q].cpu().numpy().view(np.uint32), h[q])


@pytest.mark.parametrize("shift", [1, 2, 4])
@pytest.mark.parametrize("nbox", [1, 3])
def test_device_arrays_off_their_elements_boundary(ctx, shift, nbox):
    """Device arrays `shift` bytes past an aligned address, in one box of several: the
    copies take any address, a kernel's loads and stores do not, so such a batch goes
    through the concatenated buffer.  Bit for bit the aligned call."""
    torch = pytest.importorskip("torch")
    sizes = (300, 4097, 33)[:nbox]
    prm = gi.default_params(eps=0.002, r_s=0.02, opening=gi.OPEN_REL)
    want, boxes, keep = [], (og.og_box * nbox)(), []
    for k, n in enumerate(sizes):
        pos, mass = gi.uniform(n, 70 + k)
        a = np.random.default_rng(k).normal(size=(n, 3)).astype(np.float32)
        want.append(dict(pos=pos, mass=mass, params=prm, a_old=a, acc=np.zeros((n, 3), np.float32),
                         n_pp=np.zeros(n, np.uint32), n_pn=np.zeros(n, np.uint32)))
        x = boxes[k]
        x.n, x.params = n, og.params_from_dict(prm, og.OG_DEVICE_PTRS)
        off = shift if k == 0 else 0
        for field in ("pos", "mass", "a_old", "acc", "n_pp", "n_pn"):
            raw = want[k][field].view(np.uint8).reshape(-1)
            t = torch.zeros(raw.size + 16, dtype=torch.uint8, device="cuda")
            t[off:off + raw.size] = torch.from_numpy(raw.copy()).cuda()
            setattr(x, field, t.data_ptr() + off)
            keep.append((k, field, t, off, raw.size))
    torch.cuda.synchronize()
    og.og_batch_force(ctx.h, want)
    assert og.lib().og_batch_force(ctx.h, nbox, boxes, None) == og.OG_OK
    torch.cuda.synchronize()
    for k, field, t, off, size in keep:
        got = t[off:off + size].cpu().numpy()
        assert np.array_equal(got, want[k][field].view(np.uint8).reshape(-1)), (k, field)
        assert not t[:off].any() and not t[off + size:].any()
