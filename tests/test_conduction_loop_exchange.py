"""The conduction loop's exchange between leaves (tagged words, no grid barrier): problems with
different substep counts in one launch, more leaves than SMs, and tags over many launches."""

from __future__ import annotations

import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu

_MESHES = {
    "problems": lambda: w.ensemble_mesh(16, [32, 64, 48]),
    "leaves_420": lambda: w.uniform_mesh(2, 16, (21, 20)),
    "one_leaf": lambda: w.uniform_mesh(2, 8, (1, 1)),
    "strip_3d": lambda: w.uniform_mesh(3, 8, (1, 1, 7), bc=((0, 0), (1, 1), (0, 0))),
}


def _state(mesh, seed=1204):
    rng = np.random.default_rng(seed)
    n = (mesh.nleaves,) + mesh.block_shape()
    rho = 1.0 + 0.5 * rng.random(n)
    p = 0.5 + rng.random(n)
    b = [0.5 + 0.2 * rng.random(n) for _ in range(3)]
    U = w.conserved_from_primitive(rho, 0.0, 0.0, 0.0, b[0], b[1], b[2], p, 5 / 3)
    return np.moveaxis(U, 0, 1).copy()


@pytest.mark.parametrize("geom", sorted(_MESHES))
@pytest.mark.parametrize("mode", ["isotropic", "aligned"])
@pytest.mark.parametrize("prec", [0, 1])
def test_loop_equals_per_substep_path(gpulib, geom, mode, prec):
    from paper_1204_5849_gb300 import Pool
    mesh = _MESHES[geom]()
    U0 = _state(mesh)
    # dt / dt_c ~ kappa0 / dx: several substeps per step at every resolution
    kappa0 = 3.0 * max(float(min(mesh.leaf_dx(i)[:mesh.ndim])) for i in range(mesh.nleaves))
    p = dict(gamma=5 / 3, c_cfl=0.4, scheme="lf", limiter="minmod", conduction=mode, kappa0=kappa0, subcycle=1)
    out, counts = [], []
    for loop in (True, False):
        pool = Pool(mesh, prec)
        pool.write_leaves(U0)
        pool.set_conduction_loop(loop)
        pool.advance(p, 4)
        counts.append(pool.last_conduction()[1])
        assert pool.check() == 0
        out.append(pool.read_leaves())
        pool.close()
    np.testing.assert_array_equal(counts[0], counts[1])
    if geom == "problems":
        assert len(set(int(q) for q in counts[0])) > 1, counts[0]      # the problems differ in substeps
    assert int(counts[0].max()) > 1
    np.testing.assert_array_equal(out[0], out[1])


def test_loops_of_several_pools_at_once(gpulib):
    """Three pools on streams of their own, each with more leaves than SMs: their substep loops
    are enqueued without waiting for one another and give what one pool alone gives."""
    from paper_1204_5849_gb300 import MAP_FP32_FIX64, Pool
    mesh = w.uniform_mesh(2, 16, (16, 16))
    U0 = _state(mesh)
    p = dict(gamma=5 / 3, c_cfl=0.4, scheme="lf", limiter="minmod", conduction="aligned", kappa0=3.0 / 256, subcycle=1)
    pools = [Pool(mesh, MAP_FP32_FIX64) for _ in range(3)]
    for q in pools:
        q.write_leaves(U0)
    for _ in range(6):
        for q in pools:
            q.advance(p, 1)
    assert [q.check() for q in pools] == [0, 0, 0]
    ref = Pool(mesh, MAP_FP32_FIX64)
    ref.write_leaves(U0)
    ref.set_conduction_loop(False)
    ref.advance(p, 6)
    want = ref.read_leaves()
    for q in pools:
        np.testing.assert_array_equal(q.read_leaves(), want)
