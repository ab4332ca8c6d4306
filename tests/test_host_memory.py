"""The device memory a pool holds, without a GPU: the C ABI (capi.cpp, tree.cpp) built against
tests/host/host_runtime.cpp, whose allocations are host memory that can be made to run out and
whose launchers check that every table they are given reaches to its last entry."""

from __future__ import annotations

import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import workloads as w

HERE = os.path.dirname(os.path.abspath(__file__))
PARAMS = dict(gamma=5 / 3, c_cfl=0.4, scheme="lf", limiter="minmod")


@pytest.fixture(scope="module")
def hostlib(tmp_path_factory):
    from paper_1204_5849_gb300 import _build, binding
    try:
        cuda = _build._cuda_home(_build._nvcc())
    except RuntimeError as e:
        pytest.skip(str(e))
    out = str(tmp_path_factory.mktemp("hostlib") / "libhost.so")
    # (-Bsymbolic: the library keeps its own runtime where the process has loaded another)
    cmd = ["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-pthread", "-Wl,-Bsymbolic", "-I", _build.INCLUDE,
           "-I", os.path.join(cuda, "include"), os.path.join(_build.CSRC, "capi.cpp"),
           os.path.join(_build.CSRC, "tree.cpp"), os.path.join(HERE, "host", "host_runtime.cpp"), "-o", out]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = C.CDLL(out)
    for name, (res, args) in binding._SIGS.items():
        fn = getattr(lib, name)
        fn.restype, fn.argtypes = res, args
    lib.host_fail_from.argtypes = [C.c_longlong]
    return lib


@pytest.fixture
def host(hostlib, monkeypatch):
    from paper_1204_5849_gb300 import binding
    monkeypatch.setattr(binding, "_lib", hostlib)
    hostlib.host_fail_from(0)
    yield hostlib
    hostlib.host_fail_from(0)


def counts(lib):
    v = (C.c_longlong * 6)()
    lib.host_counts(v)
    return dict(zip(("bytes", "launches", "bad", "syncs", "d2h", "graphs"), (int(x) for x in v)))


def _small():
    return w.uniform_mesh(2, 8, (4, 4), lo=(-0.5, -0.5, 0), hi=(0.5, 0.5, 1))


def _amr(levels=2):
    return w.radial_amr_mesh(2, 8, (4, 4), levels, radii=(0.12, 0.45)[2 - levels:], bc=w.mesh.PERIODIC)


def _use(pool, mesh):
    """Every call that walks the tree's tables."""
    pool.write_leaves(np.ones((mesh.nleaves,) + pool.interior_shape()))
    pool.advance(PARAMS, 3)
    pool.fill_ghosts()
    pool.cfl_dt(PARAMS)
    pool.step(PARAMS)
    pool.flag_refine(PARAMS, dict(thr=0.2))
    pool.conservation()
    pool.read_leaves()
    pool.read_block(0)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("how", ["set_tree", "regrid"])
def test_a_tree_that_does_not_fit_leaves_no_tree(host, prec, how):
    """Memory that runs out anywhere while a larger tree is installed: the call fails, no later
    call launches a kernel on tables of two trees, and a tree that fits is taken again."""
    from paper_1204_5849_gb300 import MapError, Pool
    small, big = _small(), _amr(1)
    failed = 0
    for k in range(1, 40):
        pool = Pool(small, prec, max_blocks=400)
        host.host_set_blocks(400)
        _use(pool, small)
        host.host_fail_from(k)
        try:
            getattr(pool, how)(big)
        except MapError:
            failed += 1
            host.host_fail_from(0)
            before = counts(host)
            taken = []
            for call in (lambda: pool.fill_ghosts(), lambda: pool.cfl_dt(PARAMS), lambda: pool.advance(PARAMS, 2),
                         lambda: pool.conservation(), lambda: pool.read_block(0)):
                try:
                    call()
                    taken.append(True)
                except MapError as e:
                    taken.append(e.code != -8)               # MAP_ESTATE
            after = counts(host)
            assert after["bad"] == before["bad"], (k, taken)
            # either the old tree still stands whole, or there is none
            assert len(set(taken)) == 1, (k, taken)
            if not taken[0]:
                assert after["launches"] == before["launches"], k
            for mesh in (small, big):
                pool.set_tree(mesh)
                _use(pool, mesh)
            assert counts(host)["bad"] == before["bad"], k
            pool.close()
            assert counts(host)["bad"] == before["bad"], k
        else:
            host.host_fail_from(0)
            _use(pool, big)
            pool.close()
            assert counts(host)["bad"] == 0
            break
    assert failed >= 5
    assert counts(host)["bytes"] == 0


@pytest.mark.parametrize("how", ["write_leaves_async_ptr", "read_leaves_async_ptr", "read_leaves_async_f32_ptr"])
def test_staging_that_does_not_fit_is_not_used(host, how):
    """Memory that runs out while the staging buffers of the asynchronous copies grow: a later
    copy of a smaller tree takes new buffers, not the ones given back."""
    from paper_1204_5849_gb300 import MapError, Pool
    small, big = _small(), _amr(1)
    U = np.ones((big.nleaves, 9) + big.block_shape())
    for k in (1, 2):
        pool = Pool(small, 1, max_blocks=400)
        host.host_set_blocks(400)
        getattr(pool, how)(U.ctypes.data)
        pool.set_tree(big)
        host.host_fail_from(k)
        with pytest.raises(MapError):
            getattr(pool, how)(U.ctypes.data)
        host.host_fail_from(0)
        pool.set_tree(small)
        before = counts(host)["bad"]
        getattr(pool, how)(U.ctypes.data)
        getattr(pool, how)(U.ctypes.data)
        pool.close()
        assert counts(host)["bad"] == before


@pytest.mark.parametrize("prec", [0, 1])
def test_a_pool_that_has_coarsened_gives_its_memory_back(host, prec):
    """One pool through trees that grow, shrink and grow again: every table fits its tree (the
    launches check it), and a small tree after a large one holds at most four times what the same
    tree holds in a pool of its own, and 256 KB for each of the twelve tables, besides the copies'
    staging and flags, which stay at the largest."""
    from paper_1204_5849_gb300 import Pool
    cap = 16000

    def held(mesh, fine):
        """Bytes of one pool with `mesh`, after `fine` where given."""
        base = counts(host)["bytes"]
        pool = Pool(fine or mesh, prec, max_blocks=cap)
        if fine:
            pool.set_tree(mesh)
        n = counts(host)["bytes"] - base
        pool.close()
        return n

    host.host_set_blocks(cap)
    small = _small()
    fine = w.radial_amr_mesh(2, 8, (4, 4), 5, radii=(0.25, 0.33, 0.4, 0.55, 0.9), bc=w.mesh.PERIODIC)
    assert fine.nleaves > 3000
    state = 3 * cap * 9 * 12 * 12 * (8 if prec == 0 else 4)           # the block pool itself
    kept = (fine.nleaves - small.nleaves) * (9 * 64 * 8 + 9)           # staging and flags
    assert held(small, fine) - state - kept <= 4 * (held(small, None) - state) + 12 * (256 << 10)
    pool = Pool(small, prec, max_blocks=cap)
    for mesh in (small, _amr(1), fine, small, _amr(2), small, fine, _amr(1)):
        pool.set_tree(mesh)
        _use(pool, mesh)
    pool.close()
    assert counts(host)["bad"] == 0 and counts(host)["bytes"] == 0


@pytest.mark.parametrize("radii", [((0.2,), (0.1,)), ((0.12, 0.45), (0.05, 0.3)), ((0.3, 0.44, 0.9), (0.2, 0.34, 0.7))])
def test_a_pool_between_two_trees_allocates_nothing(host, radii):
    """A tree that is refined and coarsened again by turns, to half its leaves, keeps its tables."""
    from paper_1204_5849_gb300 import Pool
    b, a = (w.radial_amr_mesh(2, 8, (8, 8), len(r), radii=r, bc=w.mesh.PERIODIC) for r in radii)
    assert 0.4 * b.nleaves < a.nleaves < 0.8 * b.nleaves
    pool = Pool(b, 1, max_blocks=4 * b.nleaves)
    host.host_set_blocks(4 * b.nleaves)
    for mesh in (a, b, a, b):
        pool.set_tree(mesh)
    host.host_fail_from(1)                                              # no allocation succeeds
    for mesh in (a, b, a, b):
        pool.set_tree(mesh)
    host.host_fail_from(0)
    _use(pool, b)
    pool.close()
    assert counts(host)["bad"] == 0 and counts(host)["bytes"] == 0


def test_schemes_that_alternate_keep_their_block_lists(host):
    """A 2D FP32 pool whose steps alternate between schemes (persistent grids of two sizes): the
    reordered block lists are built once per tree and grid, without waiting for the stream, and
    again after the active leaves or the tree change."""
    from paper_1204_5849_gb300 import Pool
    mesh = w.uniform_mesh(2, 8, (12, 12))                   # 144 blocks, grids of 24 and 32 CTAs
    pool = Pool(mesh, 1, max_blocks=400)
    host.host_set_blocks(400)
    schemes = ("mmc", "lf", "weno")

    def waits(n):
        c0 = counts(host)
        for _ in range(n):
            for s in schemes:
                pool.advance(dict(PARAMS, scheme=s), 1)
        c1 = counts(host)
        assert c1["bad"] == 0
        assert c1["d2h"] == c0["d2h"]                       # no ids are read back
        return c1["syncs"] - c0["syncs"]

    assert waits(1) <= 2                                    # one wait per list
    assert waits(5) == 0
    pool.set_active(np.arange(100, dtype=np.int32))
    for s in ("mmc", "lf"):
        pool.cfl_dt(dict(PARAMS, scheme=s))
        pool.step(dict(PARAMS, scheme=s))
    pool.set_active(None)
    assert waits(1) <= 2
    assert waits(5) == 0
    pool.set_tree(mesh)
    assert waits(1) <= 2
    assert waits(5) == 0
    pool.close()
    assert counts(host)["bad"] == 0 and counts(host)["bytes"] == 0


def test_long_advances_do_not_wait_for_their_launches(host):
    """map_advance on a refined mesh: after its first steps the host enqueues four steps at a time,
    so several hundred of them fit CUDA's queue; the count of kernels is that of plain steps.
    A change of parameters, tree or launch settings starts anew, and a caller's capture holds plain
    launches only."""
    from paper_1204_5849_gb300 import Pool
    mesh = _amr(2)
    U = np.ones((mesh.nleaves, 9) + mesh.block_shape())
    host.host_set_blocks(800)
    p = dict(PARAMS, scheme="weno")
    pool, plain = Pool(mesh, 1, max_blocks=800), Pool(mesh, 1, max_blocks=800)

    def calls(n, **kw):
        c0 = counts(host)
        k0 = pool.kernel_launches()
        pool.advance(dict(p, **kw), n)
        c1 = counts(host)
        assert c1["bad"] == 0
        return c1["launches"] - c0["launches"], c1["graphs"] - c0["graphs"], pool.kernel_launches() - k0

    def plain_kernels(n, **kw):
        k0 = plain.kernel_launches()
        for _ in range(n):
            plain.set_launch()                                           # drops what is captured
            plain.advance(dict(p, **kw), 1)
        return plain.kernel_launches() - k0

    for q in (pool, plain):
        q.write_leaves(U)
    assert calls(16)[1] == 0                                             # plain at first
    per = plain_kernels(16) // 16
    assert per >= 8
    k = plain_kernels(300)
    assert calls(300) == (0, 75, k)
    assert calls(3) == (0, 3, plain_kernels(3))                          # one at a time
    for q in (pool, plain):
        q.write_leaves(U)                                                # every region is filled again
    k = plain_kernels(9)                                                 # (with the first speeds' reduction)
    got = calls(9)
    assert got[1:] == (3, k) and got[0] == 2
    assert calls(10, eta=1e-3)[1] == 0                                   # other parameters
    plain_kernels(10, eta=1e-3)
    pool.advance(p, 16)
    pool.set_launch(3)
    assert calls(8)[1] == 0
    pool.set_launch()
    pool.set_tree(mesh)
    pool.write_leaves(U)
    assert calls(16)[1] == 0
    host.host_set_capturing(1)
    assert calls(8)[1:] == (0, 8 * per)
    host.host_set_capturing(0)
    pool.close()
    plain.close()
    assert counts(host)["bad"] == 0 and counts(host)["bytes"] == 0


def test_a_step_of_two_launches_stays_plain(host):
    """... also where the first step of a call fills every ghost region, as after a host write."""
    from paper_1204_5849_gb300 import Pool
    mesh = w.uniform_mesh(2, 8, (4, 4))
    host.host_set_blocks(400)
    pool = Pool(mesh, 1, max_blocks=400)
    c = counts(host)["graphs"]
    for _ in range(5):
        pool.write_leaves(np.ones((16, 9) + mesh.block_shape()))
        pool.advance(PARAMS, 20)
    assert counts(host)["graphs"] == c
    pool.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_autotune_leaves_the_weights_of_2d_mmc(host, prec):
    """The schedule of 2D MMC holds units of one kind, which every weight shares out alike: the
    tuner tries its grids only and keeps the default weights."""
    from paper_1204_5849_gb300 import Pool
    mesh = w.uniform_mesh(2, 8, (6, 6))
    host.host_set_blocks(400)
    tried = {}
    for scheme in ("mmc", "lf"):
        pool = Pool(mesh, prec, max_blocks=400)
        pool.write_leaves(np.ones((36, 9) + mesh.block_shape()))
        r = pool.autotune(dict(PARAMS, scheme=scheme), reps=1)
        assert (r["w_pred"], r["w_face"]) == (7, 4)
        tried[scheme] = r["trials"]
        pool.close()
    assert tried["lf"] - tried["mmc"] == 8                              # the weight ratios
    assert counts(host)["bad"] == 0 and counts(host)["bytes"] == 0
