"""Rows without output, stored nowhere or filtered away, at every place of a
group of 16 rows and in the ragged last group: beside rows of band tiles (FP32)
and of the row-wise kernels, with every other row listed for a kernel or not.
Iterates, patterns and per-iteration entries are the oracle's bit for bit."""
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


def _gaps(n, rows, seed, scale=None):
    """A banded matrix whose given rows are not stored, or (scale) scaled."""
    d = w.banded(n, 6, seed).to_dense()
    if scale is None:
        d[rows] = 0.0
    else:
        d[rows] *= scale
        d[:, rows] *= scale
    return w.csr_from_dense(d)


PLACES = {"first": lambda n: [0], "middle": lambda n: [n // 2 + 3], "group_end": lambda n: [15],
          "last": lambda n: [n - 1], "several": lambda n: [1, 16, 17, 31, n - 1],
          "group": lambda n: list(range(16, 32))}


def _equal(res, ref):
    assert res.status == ref.status and res.iters == ref.iters
    assert np.array_equal(res.rowptr, ref.rowptr) and np.array_equal(res.col, ref.col)
    assert np.array_equal(res.val.view(np.uint64), ref.val.view(np.uint64))
    assert np.array_equal(res.trace["nnz_t"], ref.trace["nnz_t"])
    # sums of squares in other orders, in FP64 or as FP32 pairs of 48 bits
    np.testing.assert_allclose(res.trace["resid_k"], ref.trace["resid"], rtol=1e-9)


@pytest.mark.parametrize("scale", [None, 1e-14])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n", [64, 75])
@pytest.mark.parametrize("place", sorted(PLACES))
def test_alone(sg, place, n, prec, scale):
    import oracle
    oracle.build()
    a = _gaps(n, PLACES[place](n), 7 + n, scale)
    res = sg.solve(a, tol=1e-8, filter="exact", prec=prec, dense_frac=2.0, max_iter=6)
    ref = oracle.nsf(a, tol=1e-8, filter="exact", mixed=bool(prec), max_iter=6)
    _equal(res, ref)


@pytest.mark.parametrize("count", [3, 60])
@pytest.mark.parametrize("prec", [0, 1])
def test_in_a_batch(sg, prec, count):
    """Few rows (3 matrices) and many (60), matrices beginning inside groups."""
    import oracle
    oracle.build()
    base = [_gaps(75, [3, 15, 74], 1), w.banded(64, 6, 2), _gaps(91, [0, 40], 3, 1e-14)]
    mats = [base[i % 3] for i in range(count)]
    out = sg.solve_batch(mats, tol=1e-8, filter="exact", prec=prec, dense_frac=2.0, max_iter=6)
    refs = [oracle.nsf(a, tol=1e-8, filter="exact", mixed=bool(prec), max_iter=6) for a in base]
    for i, res in enumerate(out):
        _equal(res, refs[i % 3])
