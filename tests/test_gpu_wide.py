"""Rows wider than one warp's accumulator: one and several warps per row, one
and several windows, with the column-block table and without it. Iterates,
patterns and results are the oracle's bit for bit, as for every other row."""
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


def _check(sg, a, max_iter, mixed, filt):
    import oracle
    oracle.build()
    f = {"none": 0, "exact": 1}[filt]
    res = sg.solve(a, tol=1e-8, filter=f, prec=int(mixed), dense_frac=2.0, max_iter=max_iter)
    ref = oracle.nsf(a, tol=1e-8, filter=filt, mixed=mixed, max_iter=max_iter)
    assert res.status == ref.status and res.iters == ref.iters
    assert np.array_equal(res.rowptr, ref.rowptr) and np.array_equal(res.col, ref.col)
    assert np.array_equal(res.val, ref.val)
    np.testing.assert_allclose(res.trace["resid_k"], ref.trace["resid"], rtol=1e-9)
    assert np.array_equal(res.trace["nnz_t"], ref.trace["nnz_t"])


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("filt,max_iter", [("exact", 4), ("none", 3)])
def test_laplacian(sg, mixed, filt, max_iter):
    _check(sg, w.laplacian(40, 2), max_iter, mixed, filt)


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("n,density", [(1025, 0.004), (1500, 0.006)])
def test_scattered(sg, mixed, n, density):
    _check(sg, w.sprand_like(n, density, seed=77 + n), 1, mixed, "exact")


def test_batch_of_wide_and_narrow(sg):
    """Windows are counted from each matrix's own first column."""
    import oracle
    oracle.build()
    mats = [w.tridiagonal(301), w.sprand_like(1200, 0.004, seed=5), w.banded(777, 3, 9),
            w.laplacian(34, 2)]
    out = sg.solve_batch(mats, tol=1e-8, filter=1, dense_frac=2.0, max_iter=1)
    for a, res in zip(mats, out):
        ref = oracle.nsf(a, tol=1e-8, filter="exact", max_iter=1)
        assert np.array_equal(res.col, ref.col) and np.array_equal(res.val, ref.val)
