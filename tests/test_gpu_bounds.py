"""The bounds of a product's rows over batches around the sizes where their
passes change: few rows, many short rows and many long rows, in matrices that
end inside a tile of rows, with band tiles (FP32) and without. Every result
equals the oracle's bit for bit (rows that fill in stay on the sparse path:
the dense one agrees to a tolerance)."""
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


def _long_rows(n, seed):
    """A tridiagonal matrix with a few rows of several hundred entries and a few
    rows of the diagonal alone."""
    rng = np.random.default_rng(seed)
    i, j = np.indices((n, n))
    d = np.where(np.abs(i - j) <= 1, 0.3, 0.0)
    d[rng.integers(0, n, 3)] = rng.uniform(-0.01, 0.01, (3, n))
    d[rng.integers(0, n, 5)] = 0.0
    d[np.arange(n), np.arange(n)] = 2.0
    return w.csr_from_dense(d)


def _check(sg, mats, prec, distinct):
    """mats repeats its first `distinct` matrices."""
    import oracle
    oracle.build()
    for it in (1, 3):
        out = sg.solve_batch(mats, tol=1e-8, filter="exact", prec=prec, dense_frac=2.0,
                             max_iter=it)
        refs = [oracle.nsf(a, tol=1e-8, filter="exact", mixed=bool(prec), max_iter=it)
                for a in mats[:distinct]]
        for k, res in enumerate(out):
            ref = refs[k % distinct]
            assert res.status == ref.status and res.iters == ref.iters
            assert np.array_equal(res.rowptr, ref.rowptr) and np.array_equal(res.col, ref.col)
            assert np.array_equal(res.val.view(np.uint64), ref.val.view(np.uint64))


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("rows", [17, 4000, 9727, 9728, 30011])
@pytest.mark.parametrize("kind", ["short", "long"])
def test_rows_of_a_batch(sg, kind, rows, prec):
    if kind == "short":  # 1 to 7 entries a row; some rows of hundreds
        base = [w.tridiagonal(131), w.banded(97, 3, 5), w.tridiagonal(1), _long_rows(700, 6)]
    else:  # about 25 entries a row
        base = [w.banded(203, 12, 7), w.banded(111, 14, 8), w.banded(16, 10, 9)]
    if rows < 200:
        base = [w.tridiagonal(rows)] if kind == "short" else [w.banded(rows, 5, 3)]
    mats, n = [], 0
    while n < rows:
        a = base[len(mats) % len(base)]
        mats.append(a)
        n += a.n
    _check(sg, mats, prec, min(len(base), len(mats)))
