"""Where a limited gradient has no value, FP32 answers 0 as the oracle does.

FP32 MMC where the predictor overdraws the density (Sec. 3.1): with c_cfl above one, heavy cells
in a light, fast gas lose more than they hold in the first-order predictor, so u~ has rho~ < 0
there and its signal speed is NaN while u itself is fine.  The limiter answers 0 for such a
gradient, and the faces beside it fall back to the first-order flux, as the oracle's do.

Bound: one FP32 update of a cell adds some 40 terms, each rounded to 2^-24 of split fluxes that,
times dt/dx, are at most c_cfl = 2 times the largest value M of the state; a term of 1/rho~ with
|rho~| >= 0.25 grows its rounding fourfold.  40 * 2^-24 * 2 * 4 ~ 1.9e-5: each cell is held to 4e-5 M.
A gradient taken from the overdrawn predictor instead of 0 changes a cell by over 1e-2 M.

And LF and MMC beside a NaN cell: its neighbours' slopes are 0, which the cells next to them see
through the faces they share; the same bound (c_cfl 0.4, no small density)."""

from __future__ import annotations

import numpy as np
import pytest

import workloads as w
from oracle import Oracle

G = 5 / 3
TOL = 4e-5

_GEOM = {
    "2d16": (lambda: w.uniform_mesh(2, 16, (2, 2)), 2.0),
    "2d8": (lambda: w.uniform_mesh(2, 8, (3, 2)), 2.0),
    "3d16": (lambda: w.uniform_mesh(3, 16, (2, 1, 1)), 2.0),
    "3d8": (lambda: w.uniform_mesh(3, 8, (2, 2, 1)), 2.0),
}


def state(mesh):
    """p = 1, a weak field, rho = 0.01 but for single cells of density 1 (in a block's middle, next
    to its faces and in its corners)."""
    nb = mesh.nb
    shape = (mesh.nleaves,) + mesh.block_shape()
    rho = np.full(shape, 0.01)
    for at in (nb // 2, 0, nb - 1, 3):
        for leaf in range(mesh.nleaves):
            z = (at if mesh.ndim == 3 else 0)
            rho[leaf, z, at, (at + 3 * leaf) % nb] = 1.0
    one = np.ones(shape)
    U = w.conserved_from_primitive(rho, 0.02 * one, -0.01 * one, 0.0 * one, 0.05 * one, 0.02 * one, 0.01 * one, one, G)
    return np.moveaxis(U, 0, 1).copy()


def params(geom, limiter):
    return dict(gamma=G, c_cfl=_GEOM[geom][1], scheme="mmc", limiter=limiter)


def one_step(mesh, p):
    orc = Oracle(mesh, state(mesh))
    orc.fill_ghosts()
    orc.cfl(p)
    orc.step(p)
    return orc.get_state()


@pytest.mark.parametrize("geom", sorted(_GEOM))
def test_the_predictor_is_overdrawn(geom):
    # without its limited terms the scheme returns u~'s density
    R = one_step(_GEOM[geom][0](), params(geom, "zero"))
    low = R[:, 0] < 0
    assert low.sum() >= 8 and R[:, 0][low].max() < -0.25 and np.abs(R[:, 0]).min() > 0.005


@pytest.mark.gpu
@pytest.mark.parametrize("geom", sorted(_GEOM))
@pytest.mark.parametrize("limiter", ["minmod", "vanleer"])
def test_fp32_falls_back_as_the_oracle(gpulib, geom, limiter):
    from paper_1204_5849_gb300 import MAP_FP32_FIX64, Pool
    mesh = _GEOM[geom][0]()
    p = params(geom, limiter)
    pool = Pool(mesh, MAP_FP32_FIX64)
    pool.write_leaves(state(mesh))
    pool.fill_ghosts()
    pool.cfl_dt(p)
    pool.step(p)
    got, want = pool.read_leaves(), one_step(mesh, p)
    assert np.isfinite(want).all() and np.isfinite(got).all()
    assert np.abs(got - want).max() <= TOL * np.abs(want).max()


def nan_state(mesh, seed=12):
    rng = np.random.default_rng(seed)
    shape = (mesh.nleaves,) + mesh.block_shape()
    r = lambda a, b: a + (b - a) * rng.random(shape)     # noqa: E731
    U = w.conserved_from_primitive(r(1, 2), r(-.2, .2), r(-.2, .2), r(-.2, .2), r(.3, .6), r(.1, .2), r(-.1, .1),
                                   r(1, 2), G, r(-.01, .01))
    U = np.moveaxis(U, 0, 1).copy()
    nb = mesh.nb
    U[0, 5, nb // 2 if mesh.ndim == 3 else 0, nb // 2, nb // 2] = np.nan      # B_y in mid-block
    U[1, 0, 0, 0, 1] = np.nan                                                # rho at a block edge
    return U


@pytest.mark.gpu
@pytest.mark.parametrize("geom", sorted(_GEOM))
@pytest.mark.parametrize("scheme", ["lf", "mmc"])
@pytest.mark.parametrize("limiter", ["minmod", "vanleer"])
@pytest.mark.parametrize("prec", [0, 1])
def test_slopes_beside_a_nan(gpulib, geom, scheme, limiter, prec):
    from paper_1204_5849_gb300 import Pool
    mesh = _GEOM[geom][0]()
    U = nan_state(mesh)
    p = dict(gamma=G, c_cfl=0.4, scheme=scheme, limiter=limiter, dt_override=0.02 * float(mesh.leaf_dx(0)[0]), ch_mode="fixed",
             ch=2.0)
    pool = Pool(mesh, prec)
    pool.write_leaves(U)
    pool.fill_ghosts()
    pool.step(p)
    want = Oracle(mesh, U)
    want.fill_ghosts()
    want.cfl(p)
    want.step(p)
    got, want = pool.read_leaves(), want.get_state()
    np.testing.assert_array_equal(np.isnan(got), np.isnan(want))
    ok = np.isfinite(want)
    assert 0 < (~ok).sum() < want.size // 2
    assert np.abs(got[ok] - want[ok]).max() <= (TOL if prec else 1e-13) * np.abs(want[ok]).max()
