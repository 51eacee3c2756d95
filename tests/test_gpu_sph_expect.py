"""Who searches a group with many candidates (csrc/og_sph.cu, k_sph_expect): from 16384
groups on, a warp each where more than an eighth of the groups are expected to be long,
a block each otherwise.  Mean smoothing lengths for all particles of a clustered set, for
a few of them and for none: counts equal and densities within float32 sums of the
oracle's on sampled targets, and the same bits again.
"""
from __future__ import annotations

import numpy as np
import pytest

import og_inputs as gi
from oracle import pm, sph
from paper_2609_17658_gb300 import build as B
from paper_2609_17658_gb300 import og

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    B.build()
    c = og.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("share", [0.0, 0.002, 0.05, 1.0])
def test_sampled_targets_against_the_oracle(ctx, share):
    n = 420_000
    pos, mass = gi.halo_mix(n, 31, n_halo=400)
    rng = np.random.default_rng(7)
    mean = (3.0 * 32.0 / (4.0 * np.pi * n)) ** (1.0 / 3.0)
    h = np.full(n, 0.1 * mean, np.float32)
    far = rng.random(n) < share
    h[far] = mean
    t = og.Tree(ctx, pos, mass, gi.default_params(r_s=0.005, eps=1e-4))
    assert t.info()["groups"] >= 16384
    rho, cnt = t.sph_density(h)
    pick = np.concatenate([rng.choice(n, 200, replace=False),
                           rng.choice(np.flatnonzero(far), 100) if far.any() else np.arange(100)])
    ref, rcnt = sph.density(pm.quantize(pos, 1.0), mass, h, 1.0, targets=pick)
    assert np.array_equal(cnt[pick].astype(np.int64), rcnt)
    assert np.all(np.abs(rho[pick] - ref) <= 1e-4 * ref)
    again, _ = t.sph_density(h)
    assert np.array_equal(again, rho)
    t.free()
