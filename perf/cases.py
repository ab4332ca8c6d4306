"""The work a user has this library do, as cases that can be timed and checked.

A case is a dict of plain values: what the pool looks like (dimension, block edge, base
tiling, refinement, problems, precision), the method (scheme, limiter, interface flux,
resistivity, conduction) and which calls a pass makes:

  advance   the batched form: state in, `steps` steps of Pool.advance, state out
  step      the step-by-step form: fill_ghosts, cfl_dt, step (`steps` times)
  flags     the refinement decision: fill_ghosts, flag_refine, plan_regrid
  regrid    the tree moves to another leaf set and back, the state with it
  snapshot  write_leaves and read_leaves of FP64 host arrays

States enter and leave the pool on the GPU through unpack_leaves / pack_leaves (a program
whose state lives in torch tensors), except in `snapshot`, whose arrays are the host's.
Every pass starts from the same input state, so passes repeat.

exact() restates the method in 64 bits on whole-domain arrays, one per refinement level: no
blocks, no ghost tables.
"""

from __future__ import annotations

import functools
import math

import numpy as np
import torch

import workloads as w
from paper_1204_5849_gb300 import MAP_FP32_FIX64, MAP_FP64, Pool

RHO, MX, BX, EN, PSI = 0, 1, 4, 7, 8
C_CFL, C_D = 0.4, 0.18
REFINE = {"harris": dict(vars=("j",), thr=0.2, coarsen=0.1), "rotor": dict(vars=("rho", "p"), thr=0.2, coarsen=0.1)}


def _case(name=None, do="advance", ic="modes", ndim=2, nb=16, bx=8, by=8, bz=1, amr="", levels=0, problems=1,
          scheme="mmc", limiter="minmod", riemann="lf", eta=0.0, conduction="off", prec="f32", steps=10):
    c = dict(do=do, ic=ic, ndim=ndim, nb=nb, bx=bx, by=by, bz=bz, amr=amr, levels=levels, problems=problems,
             scheme=scheme, limiter=limiter, riemann=riemann, eta=eta, conduction=conduction, prec=prec, steps=steps)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the small interactive 2D run (128^2 Orszag-Tang, the paper's MMC): latency and launches
        _case("ot2d_128_mmc", ic="ot"),
        # a parameter study: 96 independent periodic 2D problems of 64^2 .. 512^2 in one pool
        _case("ensemble2d_96_mmc", problems=96, bx=0, by=0, steps=4),
        # the benchmark: a linear Alfven wave on 256^3, TVD-LF with van Leer slopes (largest call)
        _case("alfven3d_256_lf", ic="alfven", ndim=3, bx=16, by=16, bz=16, scheme="lf", limiter="vanleer", steps=4),
        # 3D MMC on a box that is no power of two, 210 blocks of 16^3
        _case("modes3d_7x5x6_mmc", ndim=3, bx=7, by=5, bz=6, steps=4),
        # resistive current sheet on a three-level octree of 8^3 blocks, with reflux (9472 leaves)
        _case("harris3d_amr_lf", ic="harris", ndim=3, nb=8, bx=8, by=8, bz=8, amr="slab", levels=2, scheme="lf",
              eta=1e-3, steps=4),
        # magnetic rotor on a four-level quadtree, WENO-RK2, outflow, with reflux (about 3000 leaves)
        _case("rotor2d_amr_weno", ic="rotor", amr="radial", levels=3, scheme="weno", steps=4),
        # a 2D shock problem on a ragged uniform mesh with the HLLC flux (720 x 528 cells)
        _case("blast2d_45x33_hllc", ic="blast", bx=45, by=33, scheme="lf", limiter="vanleer", riemann="hllc", steps=4),
        # field-aligned thermal conduction, subcycled (about thirty substeps a step), WENO, 256^2
        _case("conduction2d_256_weno", ic="hot", bx=16, by=16, scheme="weno", conduction="aligned", steps=2),
        # the plain FP64 form, step by step with dt on the host (64^3, LF, van Leer): reference runs
        _case("alfven3d_64_lf_f64", do="step", ic="alfven", ndim=3, bx=4, by=4, bz=4, scheme="lf", limiter="vanleer",
              prec="f64", steps=2),
        # the refinement decision of the octree run, taken every few steps
        _case("harris3d_flags", do="flags", ic="harris", ndim=3, nb=8, bx=8, by=8, bz=8, amr="slab", levels=2,
              scheme="lf", eta=1e-3, steps=1),
        # the quadtree follows the flow: regrid to another leaf set and back
        _case("rotor2d_regrid", do="regrid", ic="rotor", amr="radial", levels=3, scheme="weno", steps=1),
        # a checkpoint of a 128^3 run written from and read back to FP64 host arrays
        _case("snapshot3d_128", do="snapshot", ndim=3, bx=8, by=8, bz=8, scheme="lf", steps=1),
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, even over the logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def _method(rng, ndim, nb, prec):
    scheme = rng.choice(["mmc", "lf", "weno"])
    m = dict(scheme=scheme, limiter=rng.choice(["minmod", "vanleer"]), prec=prec)
    if scheme != "mmc":
        m["riemann"] = rng.choice(["lf", "lf", "hllc", "hlld"])
    # a 3D 16^3 FP64 block has no shared memory left for the current density
    if rng.random() < 0.25 and not (prec == "f64" and ndim == 3 and nb == 16):
        m["eta"] = 1e-3
    return m


def draw(rng):
    kind = rng.choice(["2d", "2d", "3d", "3d", "amr2d", "amr3d", "ensemble", "conduction", "f64", "flags", "regrid",
                       "snapshot"])
    nb = rng.choice([8, 16])
    if kind == "2d":
        return _case(ic=rng.choice(["modes", "ot", "blast"]), nb=nb, bx=_log(rng, 2, 90), by=_log(rng, 2, 90),
                     steps=rng.randint(1, 10), **_method(rng, 2, nb, "f32"))
    if kind == "3d":
        top = 12 if nb == 16 else 20
        return _case(ic=rng.choice(["modes", "alfven"]), ndim=3, nb=nb, bx=_log(rng, 1, top), by=_log(rng, 1, top),
                     bz=_log(rng, 1, top), steps=rng.randint(1, 4), **_method(rng, 3, nb, "f32"))
    if kind in ("amr2d", "regrid"):
        b = rng.choice([4, 5, 6, 7, 8, 9, 10])
        c = _case(ic="rotor", nb=nb, bx=b, by=b, amr="radial", levels=rng.randint(1, 3), steps=rng.randint(1, 6),
                  **_method(rng, 2, nb, "f32"))
        return dict(c, do="regrid", steps=1, scheme="weno", eta=0.0) if kind == "regrid" else c
    if kind in ("amr3d", "flags"):
        c = _case(ic="harris", ndim=3, nb=8, bx=_log(rng, 3, 9), by=8, bz=_log(rng, 3, 9), amr="slab",
                  levels=rng.randint(1, 2), steps=rng.randint(1, 4), **_method(rng, 3, 8, "f32"))
        return dict(c, do="flags", steps=1) if kind == "flags" else c
    if kind == "ensemble":
        return _case(problems=_log(rng, 2, 96), bx=0, by=0, steps=rng.randint(1, 4), **_method(rng, 2, 16, "f32"))
    if kind == "conduction":
        return _case(ic="hot", nb=nb, bx=_log(rng, 4, 20), by=_log(rng, 4, 20), steps=rng.randint(1, 3),
                     scheme=rng.choice(["lf", "weno"]), conduction=rng.choice(["isotropic", "aligned"]))
    if kind == "f64":
        ndim = rng.choice([2, 3])
        top = (24 if ndim == 2 else 4) * (16 // nb)
        return _case(do=rng.choice(["step", "advance"]), ndim=ndim, nb=nb, bx=_log(rng, 1, top), by=_log(rng, 1, top),
                     bz=_log(rng, 1, top) if ndim == 3 else 1, steps=rng.randint(1, 2), **_method(rng, ndim, nb, "f64"))
    ndim = rng.choice([2, 3])
    return _case(do="snapshot", ndim=ndim, nb=nb, bx=_log(rng, 2, 10), by=_log(rng, 2, 10),
                 bz=_log(rng, 2, 10) if ndim == 3 else 1, scheme="lf", steps=1)


# ---- meshes and inputs -------------------------------------------------------------------

def _sizes(n):
    return [(64, 128, 256, 512)[p * 4 // n] for p in range(n)]


@functools.lru_cache(maxsize=64)
def _mesh(ndim, nb, bx, by, bz, amr, levels, problems, ic, moved=False):
    if problems > 1:
        return w.ensemble_mesh(nb, _sizes(problems))
    if amr == "radial":     # nested discs; the radii leave room for the 2:1 rule at this tiling
        step = 2.2 / (bx * 2 ** max(levels - 1, 0))
        radii = [0.44 - step if moved else 0.44]       # moved: each leaf changes by one level at most
        for _ in range(levels - 1):
            radii.append(radii[-1] + step)
            step *= 2
        return w.radial_amr_mesh(ndim, nb, (bx, by, bz), levels, radii=radii, bc=w.mesh.OUTFLOW)
    if amr == "slab":
        return w.slab_amr_mesh(ndim, nb, (bx, by, bz), levels, half_widths=(0.07, 0.2)[2 - levels:])
    centred = ic in ("blast", "hot")
    box = dict(lo=(-0.5, -0.5, 0.0), hi=(0.5, 0.5, 1.0)) if centred else {}
    return w.uniform_mesh(ndim, nb, (bx, by, bz), bc=w.mesh.OUTFLOW if ic == "blast" else w.mesh.PERIODIC, **box)


def _the_mesh(c, moved=False):
    return _mesh(c["ndim"], c["nb"], c["bx"], c["by"], c["bz"], c["amr"], c["levels"], c["problems"], c["ic"], moved)


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gamma(c):
    return 1.4 if c["ic"] == "rotor" else 5.0 / 3.0


def _params(c):
    p = dict(gamma=_gamma(c), c_cfl=C_CFL, c_d=C_D, scheme=c["scheme"], limiter=c["limiter"], riemann=c["riemann"],
             eta=c["eta"])
    if c["conduction"] != "off":
        p.update(conduction=c["conduction"], kappa0=1e-3, subcycle=1)
    return p


def _initial(c, seed, mesh):
    """(leaves, 9, nz, nb, nb) in 64 bits on the GPU: the problem named by the case, with
    phases, noise or amplitudes of this seed."""
    dev, nb, ndim = _device(), mesh.nb, mesh.ndim
    g = torch.Generator().manual_seed(int(seed))
    lv = torch.from_numpy(np.ascontiguousarray(mesh.leaves, dtype=np.int64))
    lo = torch.tensor([p.lo for p in mesh.problems], dtype=torch.float64)[lv[:, 0]]
    hi = torch.tensor([p.hi for p in mesh.problems], dtype=torch.float64)[lv[:, 0]]
    nc = torch.tensor([p.nbase for p in mesh.problems], dtype=torch.float64)[lv[:, 0]] * nb * 2.0 ** lv[:, 1:2]
    dx = (hi - lo) / nc
    at = lo + lv[:, 2:5] * nb * dx
    nz = nb if ndim == 3 else 1
    ax = []
    for d in range(3):
        n = nb if d < ndim else 1
        k = (torch.arange(n, dtype=torch.float64) + 0.5) if d < ndim else torch.zeros(1, dtype=torch.float64)
        shape = [len(lv), 1, 1, 1]
        shape[3 - d] = n
        ax.append((at[:, d:d + 1] + k * dx[:, d:d + 1]).reshape(shape).to(dev))
    x, y, z = (a.expand(len(lv), nz, nb, nb) for a in ax)
    one, tau = torch.ones_like(x), 2.0 * math.pi

    def noise(amp):
        gg = torch.Generator(device=dev).manual_seed(int(torch.randint(0, 2 ** 40, (1,), generator=g)))
        return amp * (2.0 * torch.rand(x.shape, dtype=torch.float64, device=dev, generator=gg) - 1.0)

    def phase():
        return tau * float(torch.rand(1, generator=g))

    vx = vy = vz = by = bz = 0.0 * one
    bx, p, rho = 0.0 * one, one, one
    if c["ic"] == "ot":
        s4 = math.sqrt(4.0 * math.pi)
        a, b = phase(), phase()
        rho, p = 25.0 / (36.0 * math.pi) * one, 5.0 / (12.0 * math.pi) * one
        vx, vy = -torch.sin(tau * y + a), torch.sin(tau * x + b)
        bx, by = -torch.sin(tau * y + a) / s4, torch.sin(2 * tau * x + b) / s4
    elif c["ic"] == "alfven":
        s = 1e-6 * torch.sin(tau * (x + y + z) + phase())
        by, bz, vy, vz = s / math.sqrt(2.0), -s / math.sqrt(2.0), -s / math.sqrt(2.0), s / math.sqrt(2.0)
        bx, p = one, 0.1 * one
    elif c["ic"] == "rotor":
        r = torch.sqrt(x * x + y * y)
        f = torch.clamp((0.115 - r) / 0.015, 0.0, 1.0)
        rs = torch.where(r < 0.1, 0.1 * one, torch.clamp(r, min=1e-30))
        rho, bx = 1.0 + 9.0 * f, 5.0 / math.sqrt(4.0 * math.pi) * one
        vx, vy = -2.0 * f * y / rs + noise(1e-3), 2.0 * f * x / rs + noise(1e-3)
    elif c["ic"] == "harris":
        rho = 1.0 + 1.0 / torch.cosh(y / 0.05) ** 2
        bx, p = torch.tanh(y / 0.05), 0.5 * rho
        vx, vy, vz = noise(1e-3), noise(1e-3), noise(1e-3)
        by = 1e-2 * torch.sin(tau * x + phase())
    elif c["ic"] == "blast":
        p = torch.where(x * x + y * y <= 0.01, 10.0 * one, one)
        bx = by = one / math.sqrt(2.0)
        vx, vy = noise(1e-2), noise(1e-2)
    elif c["ic"] == "hot":
        hot = (x.abs() < 0.1) & (y.abs() < 0.1)
        rho = torch.where(hot, 0.025 * one, 0.1 * one) * (1.0 + noise(1e-2))
        bx, by, p = one, one, 0.1 * one
    else:                   # smooth random modes, B divergence-free
        def series(use):
            s = torch.zeros_like(x)
            for _ in range(4):
                k = [int(q) for q in torch.randint(-3, 4, (3,), generator=g)]
                k = [q if u else 0 for q, u in zip(k, use)]
                s = s + torch.sin(tau * (k[0] * x + k[1] * y + k[2] * z) + phase())
            return 0.1 * s / 4.0
        three = ndim == 3
        every = (True, True, three)
        rho = 1.0 + series(every)
        vx, vy, vz = series(every), series(every), series(every)
        bx, by = 0.5 + series((False, True, three)), series((True, False, three))
        bz = series((True, True, False))
    e = p / (_gamma(c) - 1.0) + 0.5 * rho * (vx * vx + vy * vy + vz * vz) + 0.5 * (bx * bx + by * by + bz * bz)
    return torch.stack([rho, rho * vx, rho * vy, rho * vz, bx, by, bz, e, 0.0 * one], dim=1)


def _inputs(c, seed, mesh):
    return _initial(c, seed, mesh).to(torch.float64 if c["prec"] == "f64" else torch.float32).contiguous()


def prepare(case, seed):
    c, mesh = case, _the_mesh(case)
    u0 = _inputs(c, seed, mesh)
    stream = torch.cuda.Stream()
    pool = Pool(mesh, MAP_FP64 if c["prec"] == "f64" else MAP_FP32_FIX64, stream=stream.cuda_stream)
    s = dict(case=c, pool=pool, stream=stream, params=_params(c), mesh=mesh, ids=np.arange(mesh.nleaves, dtype=np.int32))
    if c["do"] == "snapshot":
        s["host"] = u0.double().cpu().numpy()
        s["out"] = np.empty_like(s["host"])
        return s
    s["u0"], s["out"] = u0, torch.empty_like(u0)
    if c["do"] == "flags":
        s["refine"] = dict(REFINE["harris"], max_level=c["levels"])
    if c["do"] == "regrid":
        s["moved"] = _the_mesh(c, moved=True)
        s["moved_ids"] = np.arange(s["moved"].nleaves, dtype=np.int32)
        s["out2"] = torch.empty((s["moved"].nleaves,) + tuple(u0.shape[1:]), dtype=u0.dtype, device=u0.device)
    torch.cuda.synchronize()        # the inputs were made on another stream than the pool's
    return s


def run(state):
    s = state
    c, pool, par = s["case"], s["pool"], s["params"]
    if c["do"] == "snapshot":
        pool.write_leaves(s["host"])
        return pool.read_leaves(s["out"])
    pool.unpack_leaves(s["ids"], s["u0"].data_ptr())
    if c["do"] == "advance":
        pool.advance(par, c["steps"])
        pool.pack_leaves(s["ids"], s["out"].data_ptr())
        return s["out"]
    if c["do"] == "step":
        dts = []
        for _ in range(c["steps"]):
            pool.fill_ghosts()
            dts.append(pool.cfl_dt(par))
            pool.step(par)
        pool.pack_leaves(s["ids"], s["out"].data_ptr())
        return {"u": s["out"], "dt": np.concatenate(dts)}
    if c["do"] == "flags":
        pool.fill_ghosts()
        flags, est = pool.flag_refine(par, s["refine"])
        # the estimate of an FP32 pool is computed in FP32 and widened for the host
        return {"flags": flags, "est": est.astype(np.float32), "plan": pool.plan_regrid(flags, s["refine"]["max_level"])}
    pool.fill_ghosts()
    pool.regrid(s["moved"])
    pool.pack_leaves(s["moved_ids"], s["out2"].data_ptr())
    pool.fill_ghosts()
    pool.regrid(s["mesh"])
    pool.pack_leaves(s["ids"], s["out"].data_ptr())
    return {"moved": s["out2"], "back": s["out"]}


def work(case):
    """Bytes: the state in and out of the pool, and read and written once a step.  Flops: the
    operations the method counts per cell-update (a face once, no ring overhead)."""
    c, mesh = case, _the_mesh(case)
    cells, elem = mesh.ncells, 8 if c["prec"] == "f64" else 4
    state = 9.0 * elem * cells
    if c["do"] == "snapshot":
        return {"bytes": 2.0 * (9.0 * 8.0 * cells + state), "flops": 0.0}
    if c["do"] == "flags":
        return {"bytes": 3.0 * state, "flops": 60.0 * cells}
    if c["do"] == "regrid":
        other = 9.0 * elem * _the_mesh(c, moved=True).ncells
        return {"bytes": 4.0 * (state + other), "flops": 20.0 * 9.0 * cells}
    two = c["ndim"] == 2
    per = {"lf": 1064.0 if two else 1566.0, "weno": 3850.0 if two else 5781.0, "mmc": 1500.0 if two else 2250.0}[c["scheme"]]
    if c["eta"]:
        per += 88.0
    if c["conduction"] != "off":
        per += 30 * 120.0            # about thirty substeps
    return {"bytes": state * 2.0 * (c["steps"] + 1), "flops": per * cells * c["steps"]}


# ---- the method in 64 bits on whole-domain arrays -----------------------------------------

class _Domain:
    """One problem's levels: arrays (9, nz, ny, nx) over the whole domain per level, and which
    cells are leaves, covered by finer leaves, or covered by a coarser leaf."""

    def __init__(self, mesh, p):
        self.nb, self.ndim, self.prob, self.p = mesh.nb, mesh.ndim, mesh.problems[p], p
        self.dims = range(mesh.ndim)
        self.leaves = [[int(v) for v in row] for row in np.asarray(mesh.leaves)]
        self.mine = [i for i, r in enumerate(self.leaves) if r[0] == p]
        self.top = max(self.leaves[i][1] for i in self.mine)
        self.n = [[self.prob.nbase[d] * self.nb * 2 ** L if d in self.dims else 1 for d in range(3)] for L in range(self.top + 1)]
        self.dx = [[(self.prob.hi[d] - self.prob.lo[d]) / self.n[L][d] for d in range(3)] for L in range(self.top + 1)]
        self.leaf = [torch.zeros(self.n[L][::-1], dtype=torch.bool, device=_device()) for L in range(self.top + 1)]
        for i in self.mine:
            self.leaf[self.leaves[i][1]][self.where(i)] = True
        self.finer = [torch.zeros_like(m) for m in self.leaf]
        for L in range(self.top - 1, -1, -1):
            self.finer[L] = self.coarsened((self.leaf[L + 1] | self.finer[L + 1]).double()[None])[0] > 0.5

    def where(self, i, nb=None):
        _, _, bi, bj, bk = self.leaves[i]
        nb = nb or self.nb
        sl = [slice(b * nb, (b + 1) * nb) for b in (bi, bj, bk)]
        return (sl[2] if self.ndim == 3 else slice(0, 1), sl[1], sl[0])

    def pairs(self, a, d):
        """Neighbouring pairs of cells along dimension d, as (low, high)."""
        ax = a.dim() - 1 - d
        n = a.shape[ax]
        lo = a.index_select(ax, torch.arange(0, n, 2, device=a.device))
        return lo, a.index_select(ax, torch.arange(1, n, 2, device=a.device))

    def coarsened(self, a, skip=None):
        for d in self.dims:
            if d != skip:
                lo, hi = self.pairs(a, d)
                a = 0.5 * (lo + hi)
        return a

    def load(self, u):
        U = [torch.zeros([u.shape[1]] + self.n[L][::-1], dtype=torch.float64, device=u.device) for L in range(self.top + 1)]
        for i in self.mine:
            U[self.leaves[i][1]][(slice(None),) + self.where(i)] = u[i].double()
        return U

    def store(self, U, out):
        for i in self.mine:
            out[i] = U[self.leaves[i][1]][(slice(None),) + self.where(i)]

    def pad(self, a, k=2):
        for d in self.dims:
            ax = a.dim() - 1 - d
            n = a.shape[ax]
            i = torch.arange(-k, n + k, device=a.device)
            low, high = self.prob.bc[d]
            i = torch.where(i < 0, i % n if low == 0 else 0 * i, torch.where(i >= n, i % n if high == 0 else 0 * i + n - 1, i))
            a = a.index_select(ax, i)
        return a

    def crop(self, a, k=2):
        for d in self.dims:
            ax = a.dim() - 1 - d
            a = a.narrow(ax, k, a.shape[ax] - 2 * k)
        return a

    def fill(self, U):
        """Restriction bottom-up, then minmod prolongation top-down where only a coarser leaf is."""
        for L in range(self.top - 1, -1, -1):
            U[L] = torch.where(self.finer[L], self.coarsened(U[L + 1]), U[L])
        for L in range(1, self.top + 1):
            v = self.pad(U[L - 1], 1)
            fine = self.crop(v, 1)
            for d in self.dims:
                ax = fine.dim() - 1 - d
                fine = fine.repeat_interleave(2, dim=ax)
            for d in self.dims:
                s = self.crop(_minmod(_at(v, d, 1) - v, v - _at(v, d, -1)), 1)
                for q in self.dims:
                    s = s.repeat_interleave(2, dim=s.dim() - 1 - q)
                sign = torch.arange(fine.shape[fine.dim() - 1 - d], device=v.device) % 2 * 0.5 - 0.25
                shape = [1] * fine.dim()
                shape[fine.dim() - 1 - d] = -1
                fine = fine + s * sign.reshape(shape).double()
            U[L] = torch.where(self.leaf[L] | self.finer[L], U[L], fine)
        return U


def _at(a, d, k):
    """a at the cell k further along dimension d."""
    return torch.roll(a, -k, dims=a.dim() - 1 - d)


def _minmod(a, b):
    return torch.where((a > 0) & (b > 0), torch.minimum(a, b), torch.where((a < 0) & (b < 0), torch.maximum(a, b), torch.zeros_like(a)))


def _limited(a, b, which):
    if which == "minmod":
        return _minmod(a, b)
    return torch.where(a * b > 0, 2.0 * a * b / torch.where(a * b > 0, a + b, torch.ones_like(a)), torch.zeros_like(a))


def _pressure(u, gamma):
    return (gamma - 1.0) * (u[EN] - 0.5 * (u[MX:BX] ** 2).sum(0) / u[RHO] - 0.5 * (u[BX:EN] ** 2).sum(0))


def _flux(u, d, p, ch):
    v = u[MX:BX] / u[RHO]
    B = u[BX:EN]
    pt = p + 0.5 * (B ** 2).sum(0)
    f = torch.empty_like(u)
    f[RHO] = u[MX + d]
    for k in range(3):
        f[MX + k] = u[MX + d] * v[k] - B[d] * B[k]
        f[BX + k] = v[d] * B[k] - B[d] * v[k]
    f[MX + d] += pt
    f[BX + d] = u[PSI]
    f[EN] = v[d] * (u[EN] + pt) - B[d] * (v * B).sum(0)
    f[PSI] = ch * ch * B[d]
    return f


def _fast(u, d, p, gamma):
    a2 = gamma * p.clamp(min=0.0) / u[RHO]
    s = a2 + (u[BX:EN] ** 2).sum(0) / u[RHO]
    disc = (s * s - 4.0 * a2 * u[BX + d] ** 2 / u[RHO]).clamp(min=0.0)
    return torch.sqrt(0.5 * (s + torch.sqrt(disc)))


def _speed(u, d, p, gamma):
    return (u[MX + d] / u[RHO]).abs() + _fast(u, d, p, gamma)


def _speeds9(alpha, d, ch):
    """The dissipation speed of each component: c_h for the (B_d, psi) pair."""
    s = alpha.expand((9,) + tuple(alpha.shape)).clone()
    s[BX + d] = ch
    s[PSI] = ch
    return s


def _rusanov(a, b, d, gamma, ch):
    pa, pb = _pressure(a, gamma), _pressure(b, gamma)
    s = _speeds9(torch.maximum(_speed(a, d, pa, gamma), _speed(b, d, pb, gamma)), d, ch)
    return 0.5 * (_flux(a, d, pa, ch) + _flux(b, d, pb, ch) - s * (b - a))


def _hllc(a, b, d, gamma, ch):
    bm = 0.5 * (a[BX + d] + b[BX + d]) - (b[PSI] - a[PSI]) / (2.0 * ch)
    U, F, un, cf, pt = [], [], [], [], []
    for q in (a, b):
        q2 = q.clone()
        q2[BX + d] = bm
        q2[EN] = q[EN] + 0.5 * (bm * bm - q[BX + d] ** 2)
        p = _pressure(q2, gamma)
        U.append(q2)
        F.append(_flux(q2, d, p, ch))
        un.append(q2[MX + d] / q2[RHO])
        cf.append(_fast(q2, d, p, gamma))
        pt.append(_pressure(q, gamma) + 0.5 * (q2[BX:EN] ** 2).sum(0))
    sl, sr = torch.minimum(un[0] - cf[0], un[1] - cf[1]), torch.maximum(un[0] + cf[0], un[1] + cf[1])
    ra, rb = U[0][RHO], U[1][RHO]
    sm = (rb * un[1] * (sr - un[1]) - ra * un[0] * (sl - un[0]) - pt[1] + pt[0]) / (rb * (sr - un[1]) - ra * (sl - un[0]))
    tang = [k for k in range(3) if k != d]
    bt = {k: (sr * U[1][BX + k] - sl * U[0][BX + k] - (F[1][BX + k] - F[0][BX + k])) / (sr - sl) for k in tang}
    star = []
    for q, f, u, t, s in zip(U, F, un, pt, (sl, sr)):
        v, B = q[MX:BX] / q[RHO], q[BX:EN]
        dk, ds = s - u, s - sm
        r = q[RHO] * dk / ds
        pts = t + q[RHO] * dk * (sm - u)
        o = q.clone()
        o[RHO], o[MX + d], vbs = r, r * sm, sm * bm
        for k in tang:
            o[MX + k] = r * v[k] - bm * (bt[k] - B[k]) / ds
            o[BX + k] = bt[k]
            vbs = vbs + o[MX + k] / r * bt[k]
        o[EN] = (q[EN] * dk - t * u + pts * sm + bm * ((v * B).sum(0) - vbs)) / ds
        star.append(f + s * (o - q))
    out = torch.where(sl >= 0, F[0], torch.where(sr <= 0, F[1], torch.where(sm >= 0, star[0], star[1])))
    out[BX + d] = 0.5 * (a[PSI] + b[PSI] - ch * (b[BX + d] - a[BX + d]))
    out[PSI] = 0.5 * (ch * ch * (a[BX + d] + b[BX + d]) - ch * (b[PSI] - a[PSI]))
    return out


def _cd(a, d, dx):
    return (_at(a, d, 1) - _at(a, d, -1)) / (2.0 * dx[d])


def _eglm(u, dims, dx):
    s = torch.zeros_like(u)
    div = sum(_cd(u[BX + d], d, dx) for d in dims)
    s[MX:BX] = -div * u[BX:EN]
    s[EN] = -sum(u[BX + d] * _cd(u[PSI], d, dx) for d in dims)
    return s


def _curl(a, dims, dx):
    D = lambda k, d: _cd(a[k], d, dx) if d in dims else torch.zeros_like(a[k])  # noqa: E731
    return torch.stack([D(2, 1) - D(1, 2), D(0, 2) - D(2, 0), D(1, 0) - D(0, 1)])


def _resistive(u, dims, dx, eta):
    s = torch.zeros_like(u)
    J = eta * _curl(u[BX:EN], dims, dx)
    s[BX:EN] = -_curl(J, dims, dx)
    s[EN] = -sum(_cd(torch.linalg.cross(J, u[BX:EN], dim=0)[d], d, dx) for d in dims)
    return s


def _rates(c, u, dims, dx, dt, ch):
    """Face fluxes per dimension (face of cells i, i+1) and the sources, of one update."""
    gamma, lim = _gamma(c), c["limiter"]
    face = _hllc if c["riemann"] == "hllc" else _rusanov
    S = _resistive(u, dims, dx, c["eta"]) if c["eta"] else torch.zeros_like(u)
    F = {}
    if c["scheme"] == "weno":
        for d in dims:
            dp, dm = _at(u, d, 1) - u, u - _at(u, d, -1)
            ap, am = 1.0 / (1e-12 + dp * dp) ** 2, 1.0 / (1e-12 + dm * dm) ** 2
            right = (2.0 * ap * (u + 0.5 * dp) + am * (u + 0.5 * dm)) / (2.0 * ap + am)
            left = (ap * (u - 0.5 * dp) + 2.0 * am * (u - 0.5 * dm)) / (ap + 2.0 * am)
            F[d] = face(right, _at(left, d, 1), d, gamma, ch)
        return F, S + _eglm(u, dims, dx)
    if c["scheme"] == "lf":
        phi = {d: _limited(u - _at(u, d, -1), _at(u, d, 1) - u, lim) for d in dims}
        t = u + 0.5 * dt * _eglm(u, dims, dx)
        for d in dims:
            a, b = u + 0.5 * phi[d], u - 0.5 * phi[d]
            t = t - dt / (2.0 * dx[d]) * (_flux(a, d, _pressure(a, gamma), ch) - _flux(b, d, _pressure(b, gamma), ch))
        for d in dims:
            F[d] = face(t + 0.5 * phi[d], _at(t - 0.5 * phi[d], d, 1), d, gamma, ch)
        return F, S + _eglm(t, dims, dx)
    p = _pressure(u, gamma)
    f = {d: _flux(u, d, p, ch) for d in dims}
    al = {d: _speed(u, d, p, gamma) for d in dims}
    t, h = u, {}
    for d in dims:
        s = _speeds9(torch.maximum(al[d], _at(al[d], d, 1)), d, ch)
        h[d] = 0.5 * (f[d] + s * u) + 0.5 * (_at(f[d], d, 1) - s * _at(u, d, 1))
        t = t - dt / dx[d] * (h[d] - _at(h[d], d, -1))
    q = _pressure(t, gamma)
    for d in dims:
        g, sq = _flux(t, d, q, ch), _speed(t, d, q, gamma)
        s = _speeds9(torch.maximum(al[d], _at(al[d], d, 1)), d, ch)
        st = _speeds9(torch.maximum(sq, _at(sq, d, 1)), d, ch)
        up = lambda a, k: _at(a, d, k)  # noqa: E731
        plus = lambda k: 0.5 * (up(f[d], k) + s * up(u, k))  # noqa: E731
        minus = lambda k: 0.5 * (up(f[d], k) - s * up(u, k))  # noqa: E731
        tplus = lambda k: 0.5 * (up(g, k) + st * up(t, k))  # noqa: E731
        tminus = lambda k: 0.5 * (up(g, k) - st * up(t, k))  # noqa: E731
        F[d] = h[d] + 0.5 * (_limited(tplus(0) - plus(-1), tplus(1) - plus(0), lim)
                             - _limited(minus(2) - tminus(1), minus(1) - tminus(0), lim))
    return F, S + _eglm(u, dims, dx)


def _update(u, F, S, dims, dx, dt):
    return u + dt * S - dt * sum((F[d] - _at(F[d], d, -1)) / dx[d] for d in dims)


def _reflux(D, U, F, dt):
    """On the coarse side of each coarse/fine face the mean of the fine fluxes takes the place
    of the coarse flux (psi carries the step's damping)."""
    damp = torch.ones(9, dtype=torch.float64, device=U[0].device)
    damp[PSI] = C_D
    for L in range(D.top):
        for d in D.dims:
            fine = D.coarsened(D.pairs(D.crop(F[L + 1][d]), d)[1], skip=d)
            diff = (fine - D.crop(F[L][d])) * (damp * dt / D.dx[L][d]).reshape(-1, 1, 1, 1)
            inner = torch.ones_like(D.leaf[L])       # no coarse/fine face across an outflow boundary
            ax = inner.dim() - 1 - d
            if D.prob.bc[d][1] != 0:
                inner.narrow(ax, inner.shape[ax] - 1, 1).fill_(False)
            high = D.leaf[L] & _at(D.finer[L], d, 1) & inner
            low = _at(D.finer[L] & inner, d, -1) & D.leaf[L]
            U[L] = U[L] - torch.where(high, diff, torch.zeros_like(diff))
            U[L] = U[L] + torch.where(low, _at(diff, d, -1), torch.zeros_like(diff))
    return U


def _conduct(c, u, dx, dims, dt):
    """Subcycled thermal conduction on one periodic level."""
    gamma, k0 = _gamma(c), 1e-3
    T = lambda: _pressure(u, gamma).clamp(min=0.0) / u[RHO]  # noqa: E731
    return_to = u
    kmax = c["_kmax"]
    dtc = C_CFL * min(dx[d] for d in dims) ** 2 / (len(dims) * kmax)
    n = math.ceil(dt / dtc) if dtc < dt else 1
    u = return_to.clone()
    for _ in range(n):
        t = T()
        kap = k0 * t * t * torch.sqrt(t)
        rate = torch.zeros_like(t)
        for d in dims:
            gn = (_at(t, d, 1) - t) / dx[d]
            kf = torch.sqrt(kap * _at(kap, d, 1))
            if c["conduction"] == "isotropic":
                F = kf * gn
            else:
                B = 0.5 * (u[BX:EN] + _at(u[BX:EN], d, 1))
                b2 = (B ** 2).sum(0)
                bg = B[d] * gn
                for q in dims:
                    if q != d:
                        g = _cd(t, q, dx)
                        bg = bg + B[q] * 0.5 * (g + _at(g, d, 1))
                F = torch.where(b2 > 0, kf * B[d] * bg / torch.where(b2 > 0, b2, torch.ones_like(b2)), torch.zeros_like(b2))
            rate = rate + (F - _at(F, d, -1)) / dx[d]
        u[EN] = u[EN] + dt / n * rate
    return u


def _one_step(c, D, U):
    dims, gamma = list(D.dims), _gamma(c)
    U = D.fill(U)
    ag, kmax = 0.0, 0.0
    for L in range(D.top + 1):
        if D.leaf[L].any():
            p = _pressure(U[L], gamma)
            for d in dims:
                ag = max(ag, float(_speed(U[L], d, p, gamma)[D.leaf[L]].max()))
            if c["conduction"] != "off":
                t = p.clamp(min=0.0) / U[L][RHO]
                kmax = max(kmax, float((1e-3 * t * t * torch.sqrt(t) / U[L][RHO])[D.leaf[L]].max()))
    least = min(D.dx[D.top][d] for d in dims)
    dt = C_CFL * least / (len(dims) * ag)
    if c["eta"]:
        dt = min(dt, C_CFL * least * least / (2.0 * len(dims) * c["eta"]))
    ch, F, new = ag, [], []
    if c["scheme"] == "weno":
        mid = []
        for L in range(D.top + 1):
            v = D.pad(U[L])
            f, s = _rates(c, v, dims, D.dx[L], dt, ch)
            F.append({d: 0.5 * f[d] for d in dims})
            mid.append(D.crop(_update(v, f, s, dims, D.dx[L], dt)))
        mid = D.fill(mid)
        for L in range(D.top + 1):
            v = D.pad(mid[L])
            f, s = _rates(c, v, dims, D.dx[L], dt, ch)
            F[L] = {d: F[L][d] + 0.5 * f[d] for d in dims}
            new.append(0.5 * (U[L] + D.crop(_update(v, f, s, dims, D.dx[L], dt))))
    else:
        for L in range(D.top + 1):
            v = D.pad(U[L])
            f, s = _rates(c, v, dims, D.dx[L], dt, ch)
            F.append(f)
            new.append(D.crop(_update(v, f, s, dims, D.dx[L], dt)))
    for u in new:
        u[PSI] *= C_D
    new = _reflux(D, new, F, dt)
    if c["conduction"] != "off":
        new[0] = _conduct(dict(c, _kmax=kmax), new[0], D.dx[0], dims, dt)
    return new, dt


def _estimate(c, D, U, out):
    """Block maxima of |J| dx / (|B| + 0.1) over each leaf and one layer around it."""
    for L in range(D.top + 1):
        v = D.pad(U[L])
        J, B = _curl(v[BX:EN], list(D.dims), D.dx[L]), v[BX:EN]
        e = (J ** 2).sum(0).sqrt() * min(D.dx[L]) / ((B ** 2).sum(0).sqrt() + 0.1)
        e = D.crop(e, 1)[None, None]
        blocks = torch.nn.functional.max_pool3d(e, D.nb + 2, stride=D.nb)[0, 0]
        for i in D.mine:
            if D.leaves[i][1] == L:
                _, _, bi, bj, bk = D.leaves[i]
                out[i] = blocks[bk, bj, bi]


def exact(case, seed):
    c, mesh = case, _the_mesh(case)
    u0 = _inputs(c, seed, mesh)
    if c["do"] == "snapshot":
        return u0.double().cpu().numpy()
    if c["riemann"] == "hlld" and c["do"] in ("advance", "step"):
        return None                     # its 64-bit form is as long as the solver itself
    out = torch.zeros(u0.shape, dtype=torch.float64, device=u0.device)
    if c["do"] == "flags":
        D = _Domain(mesh, 0)
        est = torch.zeros(mesh.nleaves, dtype=torch.float64, device=u0.device)
        _estimate(c, D, D.fill(D.load(u0)), est)
        return {"flags": None, "est": est, "plan": None}
    if c["do"] == "regrid":
        moved = _the_mesh(c, moved=True)
        D, M = _Domain(mesh, 0), _Domain(moved, 0)
        other = torch.zeros((moved.nleaves,) + tuple(u0.shape[1:]), dtype=torch.float64, device=u0.device)
        M.store(D.fill(D.load(u0)), other)
        D.store(M.fill(M.load(other)), out)
        return {"moved": other, "back": out}
    dts = []
    for p in range(len(mesh.problems)):
        D = _Domain(mesh, p)
        U = D.load(u0)
        for _ in range(c["steps"]):
            U, dt = _one_step(c, D, U)
            dts.append(dt)
        D.store(U, out)
    return {"u": out, "dt": np.array(dts)} if c["do"] == "step" else out
