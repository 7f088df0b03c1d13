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


# ---------------------------------------------------------------- checks of the iterates
def _long_rows(n, per, seed):
    """n <= 1024 rows of about `per` entries each, within one warp's accumulator."""
    rng = np.random.default_rng(seed)
    d = np.where(rng.random((n, n)) < per / n, rng.uniform(-0.2, 0.2, (n, n)) / per, 0.0)
    d[np.arange(n), np.arange(n)] = rng.choice([-1.0, 1.0], n) * (1.0 + rng.random(n))
    return w.csr_from_dense(d)


SUMS = ("resid_k", "xnorm_k", "beta_k")
MATS = {
    "tridiagonal": lambda: w.tridiagonal(500),      # 8 lanes a row, or 32 when rows are few
    "banded": lambda: w.banded(700, 9, 41),         # 16 and 32 lanes
    "long": lambda: _long_rows(600, 220, 5),        # several warps a row when rows are few
    "wide": lambda: w.laplacian(40, 2),             # rows of several warps, windows
    "scattered": lambda: w.sprand_like(1500, 0.006, seed=3),
}


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("name", sorted(MATS))
def test_checks_alone_and_in_batches(sg, name, prec):
    """Alone, beside a few rows (2432 in all or less) and beside many, among
    matrices of shorter and of longer rows: the sums behind the residual are the
    same bits. (Without band tiles, whose sums go by 4 columns from a multiple
    of 4 of the launch.)"""
    a = MATS[name]()
    kw = dict(tol=1e-8, filter="exact", prec=prec, dense_frac=2.0, max_iter=8, fp32_band=0)
    alone = sg.solve(a, **kw)
    small, long, wide = w.tridiagonal(301), _long_rows(500, 400, 8), w.laplacian(36, 2)
    for rest in ([small], [long], [w.tridiagonal(5000)], [wide, long, wide]):
        for mats, at in (([a] + rest, 0), (rest + [a], len(rest))):
            res = sg.solve_batch(mats, **kw)[at]
            assert res.status == alone.status and res.iters == alone.iters
            assert np.array_equal(res.val.view(np.uint64), alone.val.view(np.uint64))
            for k in SUMS:
                assert np.array_equal(res.trace[k].view(np.uint64),
                                      alone.trace[k].view(np.uint64)), (k, len(rest))


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("filt", ["exact", "bound"])
@pytest.mark.parametrize("name", ["tridiagonal", "banded", "long"])
def test_dropped_norms_alone_and_in_a_batch(sg, name, filt, prec):
    """The filter's passes take 32 lanes a row up to 9727 rows, 8 beyond."""
    a = MATS[name]()
    kw = dict(tol=1e-8, filter=filt, prec=prec, dense_frac=2.0, fp32_band=0)
    alone = sg.solve(a, **kw)
    res = sg.solve_batch([w.tridiagonal(12001), a], **kw)[1]
    if filt == "exact":
        assert (alone.trace["fnorm_k"] > 0).any()
    for k in SUMS + ("tau_k", "fnorm_k"):
        assert np.array_equal(res.trace[k].view(np.uint64), alone.trace[k].view(np.uint64)), k


@pytest.mark.parametrize("kw", [dict(filter="exact"), dict(filter="exact", prec=1, fp32_band=0),
                                dict(filter="bound"), dict(filter="none", max_iter=2),
                                dict(filter="exact", budget_norm=1)], ids=str)
def test_many_matrices(sg, kw):
    """From 1024 matrices on a cluster has eight of them, a CTA for each when all are
    small; those with larger ones (2049 and 3000 rows, thousands of candidates) are taken by
    the whole cluster, and the last one has fewer. Every matrix as alone."""
    kw = dict(tol=1e-8, dense_frac=2.0, **kw)
    base = [w.tridiagonal(16), w.banded(40, 3, 5), w.tridiagonal(1), _long_rows(60, 30, 2)]
    mats = [base[i % 4] for i in range(1030)]
    special = {0: w.tridiagonal(2048), 9: w.banded(3000, 9, 7), 10: w.tridiagonal(2049),
               17: w.laplacian(20, 2), 1029: w.banded(2500, 10, 8)}
    for i, a in special.items():
        mats[i] = a
    out = sg.solve_batch(mats, **kw)
    alone = {i: sg.solve(a, **kw) for i, a in special.items()}
    alone.update({100 + i: sg.solve(base[i], **kw) for i in range(4)})
    for i, ref in alone.items():
        same = [i] if i in special else [j for j in range(i % 4, 1030, 4) if j not in special]
        for j in same:
            res = out[j]
            assert res.status == ref.status and res.iters == ref.iters
            assert np.array_equal(res.col, ref.col)
            assert np.array_equal(res.val.view(np.uint64), ref.val.view(np.uint64))
            for k in SUMS + ("tau_k", "fnorm_k"):
                assert np.array_equal(res.trace[k].view(np.uint64),
                                      ref.trace[k].view(np.uint64)), (i, j, k)
            for k in ("nnz_t", "nnz_bar"):
                assert np.array_equal(res.trace[k], ref.trace[k])
