"""Edges of the threshold select: chunk and row boundaries of a flat array,
one and several CTAs per matrix in the digit search, candidates that crowd one
bucket, ties, and magnitudes at the ends of the range. The threshold is the
oracle's exactly, as it is decided on exact sums of squares."""
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


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.build()
    return oracle


def _tau_ref(orc, x, b):
    """tau of the oracle's EXACT filter for an array (one CSR row per value)."""
    n = len(x)
    _, tau, _ = orc.filter_csr(n, (np.arange(n + 1, dtype=np.int64), np.zeros(n, np.int32), x),
                               "exact", b)
    return tau


def _check(sg, orc, x, b):
    import torch
    tau = sg.threshold_exact(torch.from_numpy(x).cuda(), b)
    assert tau == _tau_ref(orc, x, b)
    assert tau == sg.threshold_exact(x, b)  # host input


@pytest.mark.parametrize("n", [1, 2, 31, 33, 1023, 1024, 1025, 8191, 8193, 70001])
@pytest.mark.parametrize("frac", [0.0, 1e-6, 0.3, 0.999])
def test_sizes(sg, orc, n, frac):
    rng = np.random.default_rng(n)
    x = rng.standard_normal(n) * 10.0 ** rng.uniform(-9, 0, n)
    x[rng.random(n) < 0.05] = 0.0
    _check(sg, orc, x, float(np.sqrt(frac * np.sum(x * x))))


@pytest.mark.parametrize("n", [4000, 5000, 300000])
def test_one_bucket(sg, orc, n):
    """Every value in one top-16-bit bucket, with ties: few candidates (one CTA),
    more (eight), and more survivors of the first digit than fit on chip."""
    rng = np.random.default_rng(n)
    x = 1.0 + rng.integers(0, 4096, n) * 2.0 ** -17
    _check(sg, orc, x, float(np.sqrt(0.4 * np.sum(x * x))))
    _check(sg, orc, 1.0 + rng.random(n) * 2.0 ** -13, float(np.sqrt(0.7 * n)))


def test_all_equal_and_extreme_magnitudes(sg, orc):
    n = 20000
    _check(sg, orc, np.full(n, 0.25), 0.25 * np.sqrt(n / 2))
    _check(sg, orc, np.full(n, 1e-150), 1e-150 * np.sqrt(n / 2))
    x = np.concatenate([np.full(100, 1e150), np.full(n, 1e100), [5e-324, 0.0]])
    _check(sg, orc, x, 1e100 * np.sqrt(n / 3))
    _check(sg, orc, x, 1e152)  # everything fits: +inf
