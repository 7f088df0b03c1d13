"""Rows of more than 8192 columns, whose kernel looks through the k by the first
and last columns of their B rows: full rows among narrow ones, with the
column-block table and without it, bit for bit with the oracle."""
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


def _border(a, rows, every, seed):
    """a with the given rows replaced by rows that store every `every`-th column."""
    n = a.n
    r = np.repeat(np.arange(n), np.diff(a.rowptr))
    keep = ~np.isin(r, rows)
    r, c, v = [r[keep]], [a.col[keep].astype(np.int64)], [a.val[keep]]
    rng = np.random.default_rng(seed)
    for i in rows:
        cols = np.union1d(np.arange(i % every, n, every), [i])
        x = rng.uniform(-0.3, 0.3, cols.size) / n
        x[cols == i] = 1.3
        r.append(np.full(cols.size, i))
        c.append(cols)
        v.append(x)
    return w.csr_from_coo(n, np.concatenate(r), np.concatenate(c), np.concatenate(v))


CASES = {
    "one_full": lambda: _border(w.tridiagonal(8193), [0], 1, 1),        # one window more
    "below": lambda: _border(w.tridiagonal(8192), [4000], 1, 2),        # not a long row yet
    "several": lambda: _border(w.banded(17000, 2, 5), [3, 9000, 16999], 3, 3),
    "table": lambda: _border(w.banded(9001, 21, 6), [0, 8000], 2, 4),   # rows of 43 entries
    "gaps": lambda: _border(w.csr_from_coo(9999, np.arange(0, 9999, 2), np.arange(0, 9999, 2),
                                           np.full(5000, 1.5)), [1, 500], 1, 5),  # empty B rows
}


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("name", sorted(CASES))
def test_long_rows(sg, name, mixed):
    import oracle
    oracle.build()
    a = CASES[name]()
    kw = dict(tol=1e-8, filter="exact", max_iter=3)
    res = sg.solve(a, prec=int(mixed), dense_frac=2.0, **kw)
    ref = oracle.nsf(a, mixed=mixed, **kw)
    assert res.status == ref.status and res.iters == ref.iters
    assert np.array_equal(res.rowptr, ref.rowptr) and np.array_equal(res.col, ref.col)
    assert np.array_equal(res.val.view(np.uint64), ref.val.view(np.uint64))
    assert np.array_equal(res.trace["nnz_t"], ref.trace["nnz_t"])
    np.testing.assert_allclose(res.trace["resid_k"], ref.trace["resid"], rtol=1e-9)


def test_long_rows_in_a_batch(sg):
    """Beside other matrices the checks' sums are the same bits."""
    a = CASES["several"]()
    kw = dict(tol=1e-8, filter="exact", max_iter=3, dense_frac=2.0)
    alone = sg.solve(a, **kw)
    res = sg.solve_batch([w.laplacian(40, 2), a, w.tridiagonal(300)], **kw)[1]
    assert np.array_equal(res.val.view(np.uint64), alone.val.view(np.uint64))
    for k in ("resid_k", "xnorm_k", "beta_k", "fnorm_k"):
        assert np.array_equal(res.trace[k].view(np.uint64), alone.trace[k].view(np.uint64))
