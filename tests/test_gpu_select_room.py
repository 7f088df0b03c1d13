"""The threshold select of filters above 2^28 slots, whose room for candidates is
a fraction of the slots shared by all matrices: matrices with most of their
entries in the crossing bucket, all of them within the room or not."""
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
    yield sg
    sg.trim_memory()


TOL, C4 = 1e-8, 1e-4


def _arrow(n, equal):
    """Diagonal, first row and first column: the square and the first update are
    full (n^2 slots). The update's entries off them have magnitude about c4 tol,
    all the same (equal) or spread over half an octave, so that the budget
    sqrt(n) c4 tol lies above each of them and far below their sum: the crossing."""
    d = np.full(n, 0.9) if equal else np.random.default_rng(n).uniform(0.8, 0.95, n)
    eps = np.sqrt(C4 * TOL / (1.5 * 0.9))
    i, j = np.arange(n), np.arange(1, n)
    z = np.zeros(n - 1, dtype=np.int64)
    return w.csr_from_coo(n, np.concatenate([i, z, j]), np.concatenate([i, j, z]),
                          np.concatenate([d, np.full(2 * (n - 1), eps)]))


KW = dict(tol=TOL, filter="exact", prec=0, scale_1norm=0, max_iter=1)


def _device_solve(sg, mats):
    n0 = sg.kernel_launches()
    out = sg.solve_batch(mats, device_out=True, **KW)
    return out, sg.kernel_launches() - n0


def test_crossing_bucket_within_the_room(sg):
    """n^2 = 2^28 + 32769 slots, (n - 1)(n - 2) < 2^28 candidates of one magnitude: no
    second select, so as many launches as when few are candidates."""
    import torch
    n = 16385
    (r,), launches = _device_solve(sg, [_arrow(n, True)])
    assert r.nnz == n * n and r.trace["fnorm_k"][0] == 0.0
    assert r.trace["tau_k"][0] == float(torch.as_tensor(r.val).abs().min())
    del r
    (r2,), launches2 = _device_solve(sg, [_arrow(n, False)])
    assert 0 < n * n - r2.nnz < n * n // 64
    assert launches == launches2


def test_crossing_bucket_beyond_the_room(sg):
    """(n - 1)(n - 2) > 2^28 candidates: selected again with room for every value."""
    import torch
    n = 16400
    (r,), _ = _device_solve(sg, [_arrow(n, True)])
    assert r.nnz == n * n and r.trace["fnorm_k"][0] == 0.0
    assert r.trace["tau_k"][0] == float(torch.as_tensor(r.val).abs().min())


def test_small_matrix_beside_a_large_one(sg):
    """8 x 8 with 42 of its 64 entries in the crossing bucket, and one of 2 x 2."""
    import oracle
    oracle.build()
    big = _arrow(16400, False)
    small = [_arrow(8, True), _arrow(2, False)]
    out, launches = _device_solve(sg, [big] + small)
    _, launches2 = _device_solve(sg, [big, _arrow(8, False), small[1]])
    assert launches == launches2
    for a, r in zip(small, out[1:]):
        ref = oracle.nsf(a, tol=TOL, filter="exact", scale_1norm=0, max_iter=1)
        assert r.nnz == ref.nnz and r.trace["tau_k"][0] == ref.trace["tau"][0]
        assert np.array_equal(np.asarray(r.val.cpu()).view(np.uint64), ref.val.view(np.uint64))
    alone = sg.solve(big, device_out=True, **KW)
    assert bool((alone.val == out[0].val).all()) and bool((alone.col == out[0].col).all())
