"""Calls whose counts pass the limits of a launch's grid (65535 in y and z)."""
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


@pytest.mark.parametrize("count", [3, 65600])
def test_many_dense_blocks(sg, count):
    """Matrices of order 5 and 40 on the FP32 dense path, one row group each or two."""
    base = [w.banded(5, 2, 11), w.banded(40, 3, 12), w.banded(5, 1, 13)]
    mats = [base[0]] * (count - 2) + base[1:]
    opts = sg.default_opts(tol=1e-8, filter="exact", prec=1, dense_frac=0.0)
    b = sg.Batch(mats)
    out = b.solve(opts)
    for i in (0, count // 2, count - 3, count - 2, count - 1):
        ref = sg.solve(mats[i], opts)
        assert out[i][0] == ref.status == sg.SIGN_OK and out[i][1] == ref.iters
        rp, col, val = b.handles[i].result()
        assert np.array_equal(col, ref.col)
        assert np.array_equal(val.view(np.uint64), ref.val.view(np.uint64))
    b.close()


@pytest.mark.parametrize("m,n,k", [(4, 4, 64), (5, 4, 4194300), (3, 68, 4194312)])
def test_long_fp32_product(sg, m, n, k):
    """Entries of -1, 0 and 1: every partial sum is an integer below 2^24, exact."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(k)
    a = torch.randint(-1, 2, (m, k), device="cuda", generator=g).float()
    b = torch.randint(-1, 2, (k, n), device="cuda", generator=g).float()
    assert torch.equal(sg.dense_product(a, b).double(), a.double() @ b.double())
