"""The HLLC contact speed in FP32 near the top of the range: its denominator, the sum of both
sides' mass fluxes, exceeds 2^126 for a dense slow gas whose densities, pressures and speeds are
all well inside the range.  A gas at rest with a pressure jump then still starts to move, as in
the oracle.

Bound: one step from piecewise constant states, some 40 rounded operations of 2^-24 relative on
values no larger than the state's largest M: 40 * 2^-24 ~ 2.4e-6, held to 1e-5 of each variable's
largest value.  A contact speed of 0 changes the new momentum by over a tenth of it."""

from __future__ import annotations

import numpy as np
import pytest

import workloads as w
from oracle import Oracle

pytestmark = pytest.mark.gpu

G = 5 / 3
_GEOM = {
    "2d16": lambda: w.uniform_mesh(2, 16, (2, 1), bc=w.mesh.OUTFLOW),
    "3d8": lambda: w.uniform_mesh(3, 8, (2, 1, 1), bc=w.mesh.OUTFLOW),
    "3d16": lambda: w.uniform_mesh(3, 16, (2, 1, 1), bc=w.mesh.OUTFLOW),
}


@pytest.mark.parametrize("geom", sorted(_GEOM))
@pytest.mark.parametrize("limiter", ["minmod", "vanleer"])
def test_contact_speed_of_a_dense_gas(gpulib, geom, limiter):
    from paper_1204_5849_gb300 import MAP_FP32_FIX64, Pool
    mesh = _GEOM[geom]()
    rho, big = 1.5 * 2.0 ** 125, 2.0 ** 124

    def state(X, Y, Z, **_):
        p = np.where(X < 0.5, big, 0.5 * big)
        return w.conserved_from_primitive(rho + 0 * X, 0 * X, 0 * X, 0 * X, 0 * X, 0 * X, 0 * X, p, G, 0 * X)

    U = w.evaluate_on_mesh(mesh, state)
    p = dict(gamma=G, c_cfl=0.4, scheme="lf", limiter=limiter, riemann="hllc")
    pool = Pool(mesh, MAP_FP32_FIX64)
    pool.write_leaves(U)
    pool.fill_ghosts()
    pool.cfl_dt(p)
    pool.step(p)
    orc = Oracle(mesh, U)
    orc.fill_ghosts()
    orc.cfl(p)
    orc.step(p)
    got, want = pool.read_leaves(), orc.get_state()
    assert np.isfinite(want).all()
    for v in (0, 1, 7):
        top = np.abs(want[:, v]).max()
        assert top > 0
        assert np.abs(got[:, v] - want[:, v]).max() <= 1e-5 * top, v
