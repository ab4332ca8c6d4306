"""map_advance replays captured steps (four to a graph, or one) after its first ones: the states are
bitwise those of plain launches, over every kind of step with three launches and more, through host
writes, a regrid, other parameters and calls of every length; several pools share the device."""

from __future__ import annotations

import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu

P = w.mesh.PERIODIC
_CASES = {
    "outflow_lf": (lambda: w.uniform_mesh(2, 16, (3, 3), bc=w.mesh.OUTFLOW), dict(scheme="lf", limiter="vanleer")),
    "uniform_weno": (lambda: w.uniform_mesh(2, 8, (5, 4)), dict(scheme="weno")),
    "quadtree_mmc": (lambda: w.radial_amr_mesh(2, 8, (4, 4), 1, radii=(0.2,), bc=P), dict(scheme="mmc", limiter="minmod")),
    "quadtree_weno": (lambda: w.radial_amr_mesh(2, 16, (4, 4), 2, radii=(0.16, 0.44), bc=P),
                      dict(scheme="weno", eta=1e-3)),
    "quadtree_hllc": (lambda: w.radial_amr_mesh(2, 16, (4, 4), 2, radii=(0.16, 0.44), bc=w.mesh.OUTFLOW),
                      dict(scheme="lf", limiter="minmod", riemann="hllc")),
    "octree_lf": (lambda: w.radial_amr_mesh(3, 8, (4, 4, 4), 1, radii=(0.2,), bc=P), dict(scheme="lf", limiter="minmod")),
}


def _wave(X, Y, Z, **_):
    t = 2 * np.pi
    return w.conserved_from_primitive(1 + 0.2 * np.sin(t * X), 0.1 * np.cos(t * Y), 0.05 * np.sin(t * X), 0 * X,
                                      0.5 + 0.1 * np.sin(t * Y), 0.2 + 0 * X, 0.1 + 0 * X, 1 + 0.1 * np.cos(t * X), 5 / 3,
                                      0.01 * np.sin(t * X))


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("name", sorted(_CASES))
def test_replayed_steps_are_the_plain_ones(gpulib, name, prec):
    from paper_1204_5849_gb300 import Pool
    mesh, method = _CASES[name][0](), _CASES[name][1]
    p = dict(gamma=5 / 3, c_cfl=0.3, **method)
    U = w.evaluate_on_mesh(mesh, _wave)
    replayed, plain = Pool(mesh, prec), Pool(mesh, prec)

    def both(n, q=p):
        replayed.advance(q, n)
        for _ in range(n):
            plain.set_launch()                               # drops what is captured: plain launches
            plain.advance(q, 1)
        np.testing.assert_array_equal(replayed.read_leaves(), plain.read_leaves())
        a, b = replayed.last_sums(), plain.last_sums()       # (atomics: the order of the sums varies)
        assert np.abs(a - b).max() <= 1e-13 * mesh.ncells * np.abs(b).max()
        np.testing.assert_array_equal(replayed.speeds(), plain.speeds())
        assert replayed.check() == 0 and plain.check() == 0
        assert replayed.kernel_launches() == plain.kernel_launches()

    for pool in (replayed, plain):
        pool.write_leaves(U)
    for n in (1, 16, 5, 12, 3, 7):
        both(n)
    for pool in (replayed, plain):
        pool.write_leaves(U)
    both(9)
    for pool in (replayed, plain):
        pool.fill_ghosts()
        pool.cfl_dt(p)
        pool.step(p)                                         # the other entry point in between
    both(6)
    both(21, dict(p, c_cfl=0.2))
    if mesh.leaves[:, 1].max() > 0:
        other = w.uniform_mesh(mesh.ndim, mesh.nb, mesh.problems[0].nbase[:mesh.ndim], lo=mesh.problems[0].lo,
                               hi=mesh.problems[0].hi, bc=mesh.problems[0].bc)
        for pool in (replayed, plain):
            pool.set_tree(other)
            pool.write_leaves(w.evaluate_on_mesh(other, _wave))
            pool.advance(p, 2)
            pool.set_tree(mesh)
            pool.write_leaves(U)
        both(30)


def test_replayed_steps_of_several_pools(gpulib):
    from paper_1204_5849_gb300 import MAP_FP32_FIX64, Pool
    mesh, method = _CASES["quadtree_weno"][0](), _CASES["quadtree_weno"][1]
    p = dict(gamma=5 / 3, c_cfl=0.3, **method)
    U = w.evaluate_on_mesh(mesh, _wave)
    pools = [Pool(mesh, MAP_FP32_FIX64) for _ in range(4)]
    for k, q in enumerate(pools):
        q.write_leaves(U * (1 + 0.001 * k))
    for _ in range(12):
        for q in pools:
            q.advance(p, 5)
    for k, q in enumerate(pools):
        assert q.check() == 0
        ref = Pool(mesh, MAP_FP32_FIX64)
        ref.write_leaves(U * (1 + 0.001 * k))
        for _ in range(60):
            ref.set_launch()
            ref.advance(p, 1)
        np.testing.assert_array_equal(q.read_leaves(), ref.read_leaves())
