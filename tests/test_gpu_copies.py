"""Batch transfers between device memory and pinned arrays packed one after
another, at every offset to the 16-byte words the gather kernel moves: inputs
and results arrive entry for entry, and nothing outside them is written."""
from types import SimpleNamespace

import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2210_03356_gb300 as sg
    from paper_2210_03356_gb300 import build
    build.build()
    sg.load()
    return sg


def _pinned(n, dtype):
    import torch
    return torch.zeros(n, dtype=dtype, pin_memory=True).numpy()


@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_packed_arrays_at_every_offset(sg, offset):
    import torch
    mats = [w.banded(n, b, 5 + n) for n, b in
            ((2, 1), (3, 1), (7, 2), (64, 3), (65, 3), (257, 5), (30001, 4))]
    rows, ents = sum(a.n + 1 for a in mats), sum(a.nnz for a in mats)
    rp = _pinned(rows + 4, torch.int64)
    col, val = _pinned(ents + 8, torch.int32), _pinned(ents + 8, torch.float64)
    packed, r0, e0 = [], offset % 2, offset
    for a in mats:
        rp[r0:r0 + a.n + 1], col[e0:e0 + a.nnz], val[e0:e0 + a.nnz] = a.rowptr, a.col, a.val
        packed.append(SimpleNamespace(n=a.n, rowptr=rp[r0:r0 + a.n + 1], col=col[e0:e0 + a.nnz],
                                      val=val[e0:e0 + a.nnz]))
        r0, e0 = r0 + a.n + 1, e0 + a.nnz
    o = sg.default_opts(tol=1e-8)
    batch = sg.Batch(packed)
    batch.solve(o)
    nnz = batch.result_nnz()
    orp = _pinned(rows + 4, torch.int64)
    ocol, oval = _pinned(sum(nnz) + 8, torch.int32), _pinned(sum(nnz) + 8, torch.float64)
    orp[:], ocol[:], oval[:] = -7, -7, -7.0
    outs, r0, e0 = [], offset % 2, offset
    for a, k in zip(mats, nnz):
        outs.append((orp[r0:r0 + a.n + 1], ocol[e0:e0 + k], oval[e0:e0 + k]))
        r0, e0 = r0 + a.n + 1, e0 + k
    batch.results(outs)
    batch.close()
    for a, (orow, oc, ov) in zip(mats, outs):
        ref = sg.solve(a, tol=1e-8)
        assert np.array_equal(orow, ref.rowptr) and np.array_equal(oc, ref.col)
        assert np.array_equal(ov, ref.val)
    assert np.all(orp[:offset % 2] == -7) and np.all(orp[r0:] == -7)
    assert np.all(ocol[:offset] == -7) and np.all(ocol[e0:] == -7)
    assert np.all(oval[:offset] == -7.0) and np.all(oval[e0:] == -7.0)
