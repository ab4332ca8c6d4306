"""State copies between the pool and a caller's device buffer: bitwise for every block shape,
whether or not the buffer's address allows the wide accesses."""

from __future__ import annotations

import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ndim,nb,nbase", [(2, 8, (3, 5, 1)), (2, 16, (5, 2, 1)), (3, 8, (2, 3, 1)), (3, 16, (1, 2, 1))])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("shift", [0, 1, 2])
@pytest.mark.parametrize("order", ["forward", "reversed", "part"])
def test_pack_and_unpack_at_any_element_offset(gpulib, ndim, nb, nbase, prec, shift, order):
    import torch
    from paper_1204_5849_gb300 import Pool
    mesh = w.uniform_mesh(ndim, nb, nbase)
    dt = torch.float64 if prec == 0 else torch.float32
    ids = np.arange(mesh.nleaves, dtype=np.int32)                  # the whole state in leaf order
    if order == "reversed":
        ids = ids[::-1].copy()
    elif order == "part":
        ids = ids[1:].copy()
    shape = (len(ids), 9) + mesh.block_shape()
    n = int(np.prod(shape))
    g = torch.Generator().manual_seed(1204 + shift)
    src = torch.empty(n + 4, dtype=dt, device="cuda")
    src[shift:shift + n] = torch.rand(n, generator=g, dtype=dt).cuda()
    dst = torch.full((n + 4,), -1.0, dtype=dt, device="cuda")
    pool = Pool(mesh, prec)
    torch.cuda.synchronize()
    pool.unpack_leaves(ids, src.data_ptr() + shift * src.element_size())
    pool.pack_leaves(ids, dst.data_ptr() + shift * dst.element_size())
    torch.cuda.synchronize()
    want = src[shift:shift + n].cpu().numpy().reshape(shape)
    np.testing.assert_array_equal(pool.read_leaves()[ids], want.astype(np.float64))
    np.testing.assert_array_equal(dst[shift:shift + n].cpu().numpy().reshape(shape), want)
    edges = torch.cat([dst[:shift], dst[shift + n:]])
    assert bool((edges == -1.0).all())                              # nothing outside the buffer
