"""FP64 products whose B rows run as one stream: row lengths around one pass and
around where neighbours' heads and tails meet, full and ragged bands, mixed
with short and empty-ended rows. Bit for bit against the oracle."""
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


def _check(sg, a, max_iter):
    import oracle
    oracle.build()
    res = sg.solve(a, tol=1e-10, filter=0, max_iter=max_iter)
    ref = oracle.nsf(a, tol=1e-10, filter="none", max_iter=max_iter)
    assert res.status == ref.status and res.iters == ref.iters
    assert np.array_equal(res.rowptr, ref.rowptr) and np.array_equal(res.col, ref.col)
    assert np.array_equal(res.val, ref.val)


@pytest.mark.parametrize("b", [15, 16, 30, 31, 32, 40, 63, 64])
def test_full_bands(sg, b):
    _check(sg, w.banded(500, b, 40 + b), 1)


@pytest.mark.parametrize("density", [0.35, 0.6, 0.95])
@pytest.mark.parametrize("half", [40, 75, 110])
def test_ragged_bands(sg, density, half):
    """Random holes: some runs of k stream, others fall back."""
    n = 420
    rng = np.random.default_rng(int(100 * density) + half)
    d = rng.uniform(-1, 1, (n, n)) * (rng.random((n, n)) < density)
    i, j = np.indices((n, n))
    d[np.abs(i - j) > half] = 0.0
    d[rng.integers(0, n, 12)] = 0.0  # rows with the diagonal only
    d[np.arange(n), np.arange(n)] = 2.0
    _check(sg, w.csr_from_dense(d), 1)


def test_neighbours_with_distant_columns(sg):
    """Long B rows whose columns lie elsewhere: heads above their predecessor's
    tail must not share a pass."""
    n = 600
    rng = np.random.default_rng(3)
    d = np.zeros((n, n))
    for r in range(n):
        c0 = [0, 250, 120, 480][r % 4]
        d[r, c0:c0 + 100] = rng.uniform(-1, 1, 100)
        d[r, r] = 2.0
    _check(sg, w.csr_from_dense(d), 1)
