"""Edges of the blocked inverse of NMF: orders around the panel and strip
widths (8, 4, 2 and 1 columns), pivots on and off the diagonal. Bit for bit
against the oracle's NMF, which factors column by column."""
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


@pytest.mark.parametrize("n", [1, 2, 3, 7, 8, 9, 15, 31, 33, 65, 130])
@pytest.mark.parametrize("pivoting", [False, True])
def test_inverse_edges(sg, n, pivoting):
    import oracle
    oracle.build()
    rng = np.random.default_rng(n)
    d = np.diag(np.where(rng.random(n) < 0.5, -1.0, 1.0) * (1.0 + rng.random(n)))
    d += np.where(rng.random((n, n)) < 0.2, rng.uniform(-0.3, 0.3, (n, n)), 0.0)
    if pivoting and n > 1:  # an ODE-like block: zero diagonal, every column swaps rows
        h = n // 2
        d = np.zeros((n, n))
        d[:h, n - h:] = np.eye(h) + 0.1 * rng.random((h, h))
        d[n - h:, :h] = np.eye(h)
        if n % 2:
            d[h, h] = 1.5
    a = w.csr_from_dense(d)
    res = sg.solve(a, tol=1e-10, filter="exact", method="nmf", max_iter=12)
    ref = oracle.nmf(a, tol=1e-10, filter="exact", max_iter=12)
    assert res.status == ref.status and res.iters == ref.iters
    assert np.array_equal(res.rowptr, ref.rowptr) and np.array_equal(res.col, ref.col)
    assert np.array_equal(res.val, ref.val)
