"""The FP64 limiters' bit forms on signed zeros, subnormals, infinities and NaN, on the host
(tests/host/limiter_bits.cpp), without undefined behaviour."""

from __future__ import annotations

import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_fp64_limiters_on_special_values(tmp_path):
    from paper_1204_5849_gb300 import _build
    try:
        cuda = _build._cuda_home(_build._nvcc())
    except RuntimeError as e:
        pytest.skip(str(e))
    exe = str(tmp_path / "limiter_bits")
    cmd = ["g++", "-O1", "-std=c++17", "-w", "-ffp-contract=off", "-fsanitize=undefined", "-fsanitize-undefined-trap-on-error",
           "-I", os.path.join(cuda, "include"), os.path.join(HERE, "host", "limiter_bits.cpp"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip().endswith("0 wrong"), r.stdout + r.stderr
