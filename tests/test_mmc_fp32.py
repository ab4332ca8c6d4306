"""FP32 MMC (paired fluxes; in 2D the fluxes kept per cell) against the oracle at every block
shape, limiter and resistivity, and at the persistent grid's remainders.

Bound: an FP32 update rounds each of the ~40 operations between u and the new u to 2^-24
relative to fluxes and states of order one, scaled by dt/dx <= 0.2 per face difference, so a
cell's error stays below some 16 units of 2^-24 ~ 1e-6 per step; the mean over the mesh is
held to 2e-6 of the variable's mean (floored at 1e-3 of the largest) after two steps."""

from __future__ import annotations

import numpy as np
import pytest

import workloads as w
from oracle import Oracle

pytestmark = pytest.mark.gpu

_GEOM = {
    "2d16": lambda: w.uniform_mesh(2, 16, (3, 2)),
    "2d8": lambda: w.uniform_mesh(2, 8, (5, 3)),
    "2d8_many": lambda: w.uniform_mesh(2, 8, (31, 37)),
    "2d16_outflow_one": lambda: w.uniform_mesh(2, 16, (1, 1), bc=w.mesh.OUTFLOW),
    "3d16": lambda: w.uniform_mesh(3, 16, (2, 1, 1)),
    "3d8": lambda: w.uniform_mesh(3, 8, (2, 3, 1)),
}


def _state(X, Y, Z, **_):
    t = 2 * np.pi
    rho = 1 + 0.2 * np.sin(t * (X + 2 * Y + Z))
    return w.conserved_from_primitive(rho, 0.1 * np.cos(t * Y), 0.05 * np.sin(t * X), -0.1 * np.sin(t * (X - Y)),
                                      0.5 + 0.05 * np.sin(t * Y), 0.2 + 0.1 * np.cos(t * X), 0.1 * np.cos(t * (X + Y)),
                                      1.0 + 0.1 * np.cos(t * (X - Y)), 5 / 3, 0.01 * np.sin(t * (Y + Z)))


@pytest.mark.parametrize("geom", sorted(_GEOM))
@pytest.mark.parametrize("limiter", ["minmod", "vanleer"])
@pytest.mark.parametrize("eta", [0.0, 2e-3])
def test_fp32_mmc_against_the_oracle(gpulib, geom, limiter, eta):
    from paper_1204_5849_gb300 import MAP_FP32_FIX64, Pool
    mesh = _GEOM[geom]()
    U0 = w.evaluate_on_mesh(mesh, _state)
    p = dict(gamma=5 / 3, c_cfl=0.4, scheme="mmc", limiter=limiter, eta=eta)
    pool = Pool(mesh, MAP_FP32_FIX64)
    pool.write_leaves(U0)
    pool.advance(p, 2)
    orc = Oracle(mesh, U0)
    orc.advance(p, 2)
    G, R = pool.read_leaves(), orc.get_state()
    assert pool.check() == 0
    big = max(float(np.abs(R[:, v]).mean()) for v in range(9))
    for v in range(9):
        scale = max(float(np.abs(R[:, v]).mean()), 1e-3 * big)
        assert float(np.abs(G[:, v] - R[:, v]).mean()) <= 2e-6 * scale, v
    sums = pool.last_sums()[0]
    fresh = pool.conservation()[0]
    assert np.abs(sums - fresh).max() <= 1e-6 * np.abs(fresh).max()
