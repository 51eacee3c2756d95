"""A refit's node extents from ranges of the sorted particles (tiles of 32 and 1024,
csrc/og_build.cu) against the oracle's joined extents, bit for bit: sizes around
the tiles, drifts across the box's faces, just below and at a quarter of the box
(where the level-by-level form takes over), and particles placed anywhere."""
from __future__ import annotations

import numpy as np
import pytest

import og_inputs as gi
import oracle
from paper_2609_17658_gb300 import build as B
from paper_2609_17658_gb300 import og
from tests.test_gpu_refit import _compare_refit

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    B.build()
    oracle.build()
    c = og.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n", [1, 31, 33, 49, 1023, 1025, 3000, 70001])
@pytest.mark.parametrize("drift", ["small", "faces", "below", "quarter", "anywhere"])
def test_extents_equal_the_oracle(ctx, n, drift):
    rng = np.random.default_rng(n)
    pos, mass = gi.halo_mix(n, 17, n_halo=max(1, n // 500)) if n > 2000 else gi.uniform(n, 17)
    prm = gi.default_params(eps=1e-3, r_s=0.01)
    gt, ot = og.Tree(ctx, pos, mass, prm), oracle.Tree(pos, mass, prm)
    step = {"small": 1e-4 * rng.normal(size=(n, 3)), "faces": np.full((n, 3), -0.013),
            "below": np.sign(rng.normal(size=(n, 3))) * (0.25 - 2.0 ** -20),
            "quarter": np.where(rng.random((n, 3)) < 0.01, 0.25, 0.001),
            "anywhere": rng.random((n, 3))}[drift]
    new = np.mod(pos + step, 1.0)
    new[new >= 1.0] = 0.0
    gt.refit(new)
    ot.refit(new)
    _compare_refit(gt, ot)
    gt.free()
