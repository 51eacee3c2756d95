"""The mesh kernels at their edges: runs of particles of one mesh cell that end inside
a warp, on its border and beyond it (the deposit sums each run within its warps), mesh
rows shorter and longer than a warp (the Green's factors take a warp per row), and
stencils that wrap around a mesh of two or four points.

Bars: those of the mesh force on any input, 1e-4 of the rms acceleration for every
particle and 1e-5 for the rms error (FP32 mesh and transform).
"""
from __future__ import annotations

import numpy as np
import pytest

import og_inputs as gi
from oracle import pm
from paper_2609_17658_gb300 import build as B
from paper_2609_17658_gb300 import og

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    B.build()
    c = og.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("mesh", [2, 4, 8, 32, 64, 128])
@pytest.mark.parametrize("runs", [(1,), (2, 31, 33), (32, 64, 5, 96)])
def test_runs_and_rows(ctx, mesh, runs):
    r = np.random.default_rng(mesh + len(runs))
    _, _, prm = gi.config("uniform-32k", n=1)
    prm = dict(prm, r_s=min(1.0 / mesh, 0.1))
    parts = [r.random((200, 3))]
    for k in runs:                                        # k particles inside one cell
        cell = r.integers(0, mesh, 3)
        parts.append((cell + 0.05 + 0.9 * r.random((k, 3))) / mesh)
    pos = np.concatenate(parts)
    mass = r.random(len(pos)) / len(pos)
    acc = og.Tree(ctx, pos, mass, prm).pm_force(mesh).astype(np.float64)
    ref = pm.pm_accel(pm.quantize(pos, prm["box"]), mass, mesh, prm["box"], prm["G"], prm["r_s"])
    assert np.isfinite(acc).all()
    if mesh == 2:                                         # the stencil's points coincide in pairs
        assert not acc.any() and not ref.any()
        return
    rms = np.sqrt((ref ** 2).sum(axis=1).mean())
    err = np.linalg.norm(acc - ref, axis=1)
    assert err.max() <= 1e-4 * rms and np.sqrt((err ** 2).mean()) <= 1e-5 * rms
