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
