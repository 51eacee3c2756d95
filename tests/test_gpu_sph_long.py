"""Groups with more candidates than one warp searches by itself (csrc/og_sph.cu,
k_sph_long): sparse particles whose smoothing lengths reach into a dense clump,
counts equal and densities within float32 sums of the oracle's.  The candidate
numbers lie around the limits (1024 and 2048), around the chunk of the block
search (512 and 1024 entries) and far above, and the clump holds a bucket of
coincident particles larger than a round of the block (512 records)."""
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


@pytest.mark.parametrize("clump,same", [(500, 0), (1000, 3), (1025, 0), (2049, 600), (3000, 513), (20000, 1400)])
def test_long_searches_against_the_oracle(ctx, clump, same):
    rng = np.random.default_rng(clump)
    pos = np.concatenate([rng.random((2000, 3)), 0.5 + 1e-3 * rng.normal(size=(clump, 3)),
                          np.full((same, 3), 0.5 + 2e-3)])
    n = len(pos)
    mass = rng.uniform(0.5, 1.5, n) / n
    h = np.full(n, 0.08, np.float32)
    near = np.linalg.norm(pos - 0.5, axis=1) < 0.02
    h[near] = (2e-4 * rng.uniform(0.5, 2.0, int(near.sum()))).astype(np.float32)
    h[2000] = 0.05                                   # one member of the clump that sees all of it
    prm = gi.default_params(r_s=0.01, eps=1e-4)
    t = og.Tree(ctx, pos, mass, prm)
    rho, cnt = t.sph_density(h)
    ref, rcnt = sph.density(pm.quantize(pos, 1.0), mass, h, 1.0)
    assert int(rcnt.max()) > clump
    assert np.array_equal(cnt.astype(np.int64), rcnt)
    assert np.all(np.abs(rho - ref) <= 1e-4 * ref)
    again, _ = t.sph_density(h)
    assert np.array_equal(again, rho)
    t.free()
