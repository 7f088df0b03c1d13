"""Edges of the dense path's kernels: K around the exact blocks and the steps
that share an accumulator, ragged tiles and odd leading dimensions of the FP64
product; row groups and column chunks of the densify pass."""
from fractions import Fraction

import numpy as np
import pytest

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


@pytest.mark.parametrize("m,n,k", [(1, 2, 1), (129, 258, 127), (127, 254, 512), (40, 34, 513),
                                   (130, 60, 2048), (33, 300, 2049), (20, 20, 4095),
                                   (17, 258, 4097), (16, 30, 8200)])
def test_f64_product_edges(sg, m, n, k):
    """Sampled entries against exact rational products, within the splitting's
    bound 2^-41 max(1, K/4096) 2^(e_i + f_j)."""
    import torch
    rng = np.random.default_rng(m + 3 * n + 7 * k)
    a = rng.standard_normal((m, k)) * np.exp2(rng.integers(-12, 3, (m, k)))
    b = rng.standard_normal((k, n)) * np.exp2(rng.integers(-12, 3, (k, n)))
    pad = torch.zeros(m, k + 3, dtype=torch.float64, device="cuda")  # odd leading dimension
    pad[:, :k] = torch.from_numpy(a)
    c = sg.dense_product_f64(pad[:, :k], torch.from_numpy(b).cuda()).cpu().numpy()
    ea = np.frexp(np.abs(a).max(axis=1))[1]
    fb = np.frexp(np.abs(b).max(axis=0))[1]
    cells = [(0, 0), (m - 1, n - 1), (0, n - 1), (m - 1, 0)]
    cells += list(zip(rng.integers(0, m, 8), rng.integers(0, n, 8)))
    for i, j in cells:
        exact = sum(Fraction(x) * Fraction(y) for x, y in zip(a[i], b[:, j]))
        bound = Fraction(2.0 ** -41 * max(1.0, k / 4096)) * Fraction(2) ** int(ea[i] + fb[j])
        assert abs(Fraction(c[i, j]) - exact) <= bound


@pytest.mark.parametrize("n", [5, 31, 33, 127, 130, 259])
def test_densify_edges(sg, n):
    """Every round on the dense path (dense_frac = 0): the result is the
    oracle's mixed result to the FP32 stage's accuracy."""
    import oracle
    import workloads as w
    oracle.build()
    a = w.banded(n, 3, 900 + n)
    res = sg.solve(a, tol=1e-8, filter="exact", prec=1, dense_frac=0.0)
    ref = oracle.nsf(a, tol=1e-8, filter="exact", mixed=True)
    assert res.status == ref.status == sg.SIGN_OK
    S = np.zeros((n, n))
    S[np.repeat(np.arange(n), np.diff(res.rowptr)), res.col] = res.val
    R = ref.to_dense(n)
    assert np.linalg.norm(S - R) / np.linalg.norm(R) < 1e-5
