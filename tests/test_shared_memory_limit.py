"""Resistive and ideal steps of one kernel take turns in one process: the resistive form needs
more shared memory, and an ideal step in between must not lower the limit under it."""

from __future__ import annotations

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# (a process of its own: the limits are set once per process and kernel)
_CODE = """
import sys
sys.path.insert(0, {root!r})
import workloads as w
from paper_1204_5849_gb300 import Pool
for prec in (0, 1):
    for ndim, nb, base in ((2, 16, (2, 2)), (2, 8, (2, 2)), (3, 16, (1, 1, 1)), (3, 8, (2, 1, 1))):
        if prec == 0 and ndim == 3 and nb == 16:
            continue                    # no room for the current density there, refused as such
        mesh = w.uniform_mesh(ndim, nb, base)
        U = w.evaluate_on_mesh(mesh, w.orszag_tang if ndim == 2 else w.alfven_wave)
        for scheme in ("mmc", "lf", "weno"):
            pool = Pool(mesh, prec)
            pool.write_leaves(U)
            for eta in (1e-3, 0.0, 1e-3, 0.0, 1e-3):
                pool.advance(dict(gamma=5 / 3, c_cfl=0.3, scheme=scheme, limiter="minmod", eta=eta), 1)
            assert pool.check() == 0
            pool.close()
print("all steps ran")
"""


def test_resistive_steps_after_ideal_ones(gpulib):
    r = subprocess.run([sys.executable, "-c", _CODE.format(root=ROOT)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "all steps ran" in r.stdout, r.stderr[-2000:]
