"""Builds and refits whose stages share launches (up to 2^18 particles) and the same
with a launch per stage, against the oracle bit for bit: sizes at that line, at the tiles
of the splits (1024), the moments (512 particles) and the scans (4096), and
masses whose set bits span more than the sums hold.
"""
from __future__ import annotations

import numpy as np
import pytest

import og_inputs as gi
import oracle
from paper_2609_17658_gb300 import build as B
from paper_2609_17658_gb300 import og
from tests import parity
from tests.test_gpu_refit import _compare_refit

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    B.build()
    oracle.build()
    c = og.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n", [1, 2, 257, 512, 513, 1025, 4096, 4097, 131073, 262144, 262145])
def test_build_and_refit(ctx, n):
    pos, mass = gi.halo_mix(n, 23, n_halo=max(1, n // 2000)) if n > 5000 else gi.uniform(n, 23)
    prm = gi.default_params(eps=1e-3, r_s=0.01)
    gt, ot = og.Tree(ctx, pos, mass, prm), oracle.Tree(pos, mass, prm)
    parity.compare_build(gt, ot)
    new = np.mod(pos + 1e-4 * np.random.default_rng(n).normal(size=(n, 3)), 1.0)
    new[new >= 1.0] = 0.0
    gt.refit(new)
    ot.refit(new)
    _compare_refit(gt, ot)
    gt.free()


@pytest.mark.parametrize("n", [600, 262145])
def test_wide_mass_span_is_refused(ctx, n):
    pos, mass = gi.uniform(n, 29)
    mass[n // 2] = np.ldexp(1.0, -200)
    with pytest.raises(og.OGError, match="mass"):
        og.Tree(ctx, pos, mass, gi.default_params(eps=1e-3, r_s=0.01))
    mass[n // 2] = mass[0]
    og.Tree(ctx, pos, mass, gi.default_params(eps=1e-3, r_s=0.01)).free()
