"""A result does not depend on what else is in the launch: products of some
rows against the same rows among others, and solves alone against the same
matrix in batches, bit for bit."""
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


# ---------------------------------------------------------------- dense tiles
@pytest.mark.parametrize("k", [512, 2048, 2052, 2744, 4096])
@pytest.mark.parametrize("m", [40, 1000, 2500])
def test_rows_of_the_fp64_dense_product(sg, m, k):
    """The last wave's tiles are cut into parts, the others run whole; which
    ones follows from the number of rows (2744 x 2744: 152 of 242 whole)."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(m + k)
    a = torch.randn(2744, k, dtype=torch.float64, device="cuda", generator=g)
    b = torch.randn(k, 2744, dtype=torch.float64, device="cuda", generator=g)
    full = sg.dense_product_f64(a, b)
    some = sg.dense_product_f64(a[:m].contiguous(), b)
    assert torch.equal(full[:m], some)


@pytest.mark.parametrize("m", [40, 1000, 4000])
def test_rows_of_the_fp32_dense_product(sg, m):
    """Whole tiles and the last wave's halves (4100 x 4096: 152 x 3 whole)."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(m)
    a = torch.randn(4100, 1000, device="cuda", generator=g)
    b = torch.randn(1000, 4096, device="cuda", generator=g)
    full = sg.dense_product(a, b)
    some = sg.dense_product(a[:m].contiguous(), b)
    assert torch.equal(full[:m], some)


def test_fp64_dense_path_alone_and_in_a_batch(sg):
    """n = 2209: 162 tiles alone, more beside another dense matrix."""
    mats = [w.laplacian(47, 2), w.laplacian(40, 2)]
    kw = dict(tol=1e-8, filter="exact", prec=0, max_iter=100)
    out = sg.solve_batch(mats, **kw)
    for a, res in zip(mats, out):
        alone = sg.solve(a, **kw)
        assert res.status == alone.status and res.iters == alone.iters
        assert np.array_equal(res.col, alone.col)
        assert np.array_equal(res.val.view(np.uint64), alone.val.view(np.uint64))
