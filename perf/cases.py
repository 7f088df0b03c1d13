"""Performance cases of the sign solver: the work its users have it do.

Every case goes through the public entry points of the package (solve, Batch,
threshold_exact, dense_product, dense_product_f64) at sizes of the workloads
this repository names: tridiagonal and banded matrices, the ODE block matrix,
shifted Laplacians, random sparse matrices for Newton's method, and the two
building blocks that can be called alone.

A case is a dict with a "kind" and its sizes:

  tridiag    one symmetric tridiagonal matrix, n 500 .. 262144
  ode        one nonsymmetric block matrix [[0, B], [I, 0]], order 2n, unscaled
  banded     one banded matrix, half-bandwidth b 1 .. 10
  batch      many banded matrices solved together, n in [200, 8000], b 1 .. 10,
             from pinned host arrays into pinned host arrays
  laplacian  one shifted 2-D or 3-D grid Laplacian, whose sign fills in
  nmf        one random sparse matrix by Newton's method with filtering
  threshold  the element threshold of one array of values
  gemm32     the dense product of FP32 accuracy
  gemm64     the dense product of FP64 accuracy

Results are the stored CSR of sign(A) where it stays sparse, and the dense
matrix where it fills in (a user of a filled-in sign takes it dense).
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2210_03356_gb300 as sg

FILTERS = {"none": 0, "exact": 1, "bound": 2}
PRECS = {"fp64": 0, "mixed": 1}


def listed():
    return [
        # the smallest call: one small system solved at a time inside a host program
        # (numpy CSR in and out), where launches and waits are the cost
        {"name": "tridiag_500_fp64", "kind": "tridiag", "n": 500, "prec": "fp64",
         "filter": "exact", "tol": 1e-8, "where": "host"},
        # the largest tridiagonal of the served mix, matrix already on the GPU
        {"name": "tridiag_262144_mixed", "kind": "tridiag", "n": 262144, "prec": "mixed",
         "filter": "exact", "tol": 1e-8, "where": "device"},
        # the ODE block matrix at the largest order of its published table:
        # nonsymmetric, unscaled, tight tolerance, the default FP64
        {"name": "ode_5000_fp64", "kind": "ode", "n": 5000, "prec": "fp64", "filter": "exact",
         "tol": 1e-12, "where": "host"},
        # one mid-size banded request with the cheaper BOUND filter, odd order
        {"name": "banded_6001_bound", "kind": "banded", "n": 6001, "b": 7, "prec": "mixed",
         "filter": "bound", "tol": 1e-8, "where": "device"},
        # the benchmark's batch: 512 banded matrices, end to end
        {"name": "batch_512_mixed", "kind": "batch", "count": 512, "nmin": 200, "nmax": 8000,
         "prec": "mixed", "filter": "exact", "tol": 1e-8},
        # a smaller batch for users who need full FP64 results (wider bands, FP64 products only)
        {"name": "batch_32_fp64", "kind": "batch", "count": 32, "nmin": 200, "nmax": 8000,
         "prec": "fp64", "filter": "exact", "tol": 1e-12},
        # a fill-in request of the served mix: wide sparse rows first, then the dense path
        {"name": "laplacian2d_45_mixed", "kind": "laplacian", "dim": 2, "m": 45, "prec": "mixed",
         "filter": "exact", "tol": 1e-8},
        # the 3-D Laplacian at its smallest named size: dense path in FP32 and in FP64
        {"name": "laplacian3d_16_mixed", "kind": "laplacian", "dim": 3, "m": 16, "prec": "mixed",
         "filter": "exact", "tol": 1e-8},
        # Newton's method with filtering (dense inverse) at the paper's small size
        {"name": "nmf_500", "kind": "nmf", "n": 500, "filter": "exact", "tol": 1e-12},
        # the threshold alone over the values of a large update, ragged count
        {"name": "threshold_16777219", "kind": "threshold", "nnz": 16777219, "where": "device"},
        # the dense products alone; 2744 = 14^3 is a grid Laplacian's order
        {"name": "gemm32_4096", "kind": "gemm32", "m": 4096, "n": 4096, "k": 4096},
        {"name": "gemm64_2744", "kind": "gemm64", "m": 2744, "n": 2744, "k": 2744},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tridiag", "ode", "banded", "banded", "batch", "batch", "laplacian",
                       "laplacian", "nmf", "threshold", "gemm32", "gemm64"])
    prec = rng.choice(["fp64", "mixed"])
    filt = rng.choice(["exact", "exact", "exact", "bound"])
    where = rng.choice(["host", "device"])
    tol = rng.choice([1e-8, 1e-8, 1e-10, 1e-12]) if prec == "fp64" else 1e-8
    if kind == "tridiag":
        return {"kind": kind, "n": _log(rng, 500, 262144), "prec": prec, "filter": filt,
                "tol": tol, "where": where}
    if kind == "ode":
        return {"kind": kind, "n": _log(rng, 250, 5000), "prec": "fp64", "filter": "exact",
                "tol": 1e-12, "where": where}
    if kind == "banded":
        return {"kind": kind, "n": _log(rng, 200, 8000), "b": rng.randint(1, 10), "prec": prec,
                "filter": filt, "tol": tol, "where": where}
    if kind == "batch":
        # FP64 throughout costs several times the mixed mode per matrix
        return {"kind": kind, "count": _log(rng, 2, 512 if prec == "mixed" else 48), "nmin": 200,
                "nmax": 8000, "prec": prec, "filter": filt, "tol": tol}
    if kind == "laplacian":
        dim = rng.choice([2, 3])
        return {"kind": kind, "dim": dim, "m": rng.randint(20, 48) if dim == 2 else
                rng.randint(8, 16), "prec": "mixed", "filter": "exact", "tol": 1e-8}
    if kind == "nmf":
        return {"kind": kind, "n": rng.randint(150, 500), "filter": "exact", "tol": 1e-12}
    if kind == "threshold":
        return {"kind": kind, "nnz": _log(rng, 1000, 64 << 20), "where": "device"}
    if kind == "gemm32":
        return {"kind": kind, "m": _log(rng, 300, 6000), "n": 4 * _log(rng, 75, 1500),
                "k": 4 * _log(rng, 75, 1500)}
    return {"kind": kind, "m": _log(rng, 300, 4000), "n": 2 * _log(rng, 150, 2000),
            "k": _log(rng, 300, 5000)}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _rand(g, *shape):
    return torch.rand(*shape, dtype=torch.float64, device="cuda", generator=g)


def _csr_of_diagonals(n, offs, diags):
    """CSR of the matrix whose entry (i, i + offs[j]) is diags[i, j]; offs ascend."""
    offs = torch.tensor(offs, device="cuda")
    col = torch.arange(n, device="cuda")[:, None] + offs[None, :]
    ok = (col >= 0) & (col < n)
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(ok.sum(1), 0, out=rowptr[1:])
    return SimpleNamespace(n=n, rowptr=rowptr, col=col[ok].to(torch.int32), val=diags[ok])


def _banded(n, b, g, off_scale=None):
    """Symmetric banded matrix: diagonal +-(1 + U[0,1)); off-diagonals U[-1,1] scaled so that
    every row's off-diagonal sum is at most 0.8 (or, with off_scale, just scaled by it)."""
    b = min(b, n - 1)
    diag = torch.where(_rand(g, n) < 0.5, -1.0, 1.0) * (1.0 + _rand(g, n))
    up = torch.zeros(n, b, dtype=torch.float64, device="cuda")  # up[i, d-1] = a(i, i+d)
    if b:
        up = 2.0 * _rand(g, n, b) - 1.0
        d = torch.arange(1, b + 1, device="cuda")
        i = torch.arange(n, device="cuda")[:, None]
        up = torch.where(i + d < n, up, torch.zeros_like(up))
        if off_scale is not None:
            up = up * off_scale
        else:
            pad = torch.zeros(b, b, dtype=torch.float64, device="cuda")
            src = torch.cat([pad, up])  # row i + b - d of column d-1 is a(i-d, i)
            low = src[i + b - d, d - 1]
            s = torch.clamp(0.8 / (up.abs().sum(1) + low.abs().sum(1)).clamp_min(1e-300), max=1.0)
            sp = torch.cat([s, torch.ones(b, dtype=torch.float64, device="cuda")])
            up = up * torch.minimum(s[:, None], sp[i + d])
        src = torch.cat([torch.zeros(b, b, dtype=torch.float64, device="cuda"), up])
        low = src[i + b - d, d - 1]
        diags = torch.cat([low.flip(1), diag[:, None], up], 1)
    else:
        diags = diag[:, None]
    return _csr_of_diagonals(n, list(range(-b, b + 1)), diags)


def _ode(n, lam):
    """[[0, B], [I, 0]] of order 2n with B = tridiag(lam, 1 - 2 lam, lam)."""
    dg = torch.zeros(2 * n, 4, dtype=torch.float64, device="cuda")
    offs = [-n, n - 1, n, n + 1]
    dg[:n, 1], dg[:n, 2], dg[:n, 3] = lam, 1.0 - 2.0 * lam, lam
    dg[n:, 0] = 1.0
    col = torch.arange(2 * n, device="cuda")[:, None] + torch.tensor(offs, device="cuda")
    ok = (col >= 0) & (col < 2 * n)
    ok[:n, 0] = False
    ok[n:, 1:] = False
    ok[:n, 1:] &= col[:n, 1:] >= n  # B's own first column
    rowptr = torch.zeros(2 * n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(ok.sum(1), 0, out=rowptr[1:])
    return SimpleNamespace(n=2 * n, rowptr=rowptr, col=col[ok].to(torch.int32), val=dg[ok])


def _laplacian(m, dim, frac):
    """Dirichlet grid Laplacian minus sigma I, sigma at the fraction frac of the spectral gap at
    the centre of the spectrum."""
    e = 2.0 - 2.0 * np.cos(np.arange(1, m + 1) * math.pi / (m + 1))
    lam = e[:, None] + e[None, :]
    if dim == 3:
        lam = lam[:, :, None] + e[None, None, :]
    lam = np.sort(lam.ravel())
    c = 2.0 * dim
    above = lam[lam > c + 1e-9][0]
    below = c if np.abs(lam - c).min() < 1e-9 else lam[lam < c - 1e-9][-1]
    sigma = below + frac * (above - below)
    n = m ** dim
    idx = torch.arange(n, device="cuda")
    offs = sorted([0] + [s * m ** a for a in range(dim) for s in (-1, 1)])
    dg = torch.full((n, len(offs)), -1.0, dtype=torch.float64, device="cuda")
    ok = torch.ones(n, len(offs), dtype=torch.bool, device="cuda")
    for j, o in enumerate(offs):
        if o == 0:
            dg[:, j] = c - sigma
        else:
            x = (idx // abs(o)) % m + (1 if o > 0 else -1)
            ok[:, j] = (x >= 0) & (x < m)
    col = idx[:, None] + torch.tensor(offs, device="cuda")
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(ok.sum(1), 0, out=rowptr[1:])
    return SimpleNamespace(n=n, rowptr=rowptr, col=col[ok].to(torch.int32), val=dg[ok])


def _sprand(n, density, g):
    """Nonsymmetric random sparse matrix, off-diagonal U[0,1) at about density n^2 places, a
    diagonal +-(1 + U[0,1))."""
    a = torch.where(_rand(g, n, n) < density, _rand(g, n, n), torch.zeros(1, dtype=torch.float64,
                                                                          device="cuda"))
    a.diagonal().copy_(torch.where(_rand(g, n) < 0.5, -1.0, 1.0) * (1.0 + _rand(g, n)))
    ok = a != 0
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(ok.sum(1), 0, out=rowptr[1:])
    col = torch.arange(n, device="cuda").expand(n, n)[ok]
    return SimpleNamespace(n=n, rowptr=rowptr, col=col.to(torch.int32), val=a[ok])


def _batch_shapes(case):
    """(n, b) of each matrix: orders spread over the logarithm of [nmin, nmax], half-bandwidths
    over 1 .. 10, the same for every seed."""
    out = []
    for k in range(case["count"]):
        u = (0.5 + k * 0.6180339887498949) % 1.0
        n = int(round(case["nmin"] * (case["nmax"] / case["nmin"]) ** u))
        out.append((n, 1 + (7 * k + 3) % 10))
    return out


def _row_room(b, tol):
    """Room per row of a banded result's CSR in the caller's buffers (their tails stay zero)."""
    return 24 + 16 * b if tol >= 1e-9 else 35 + 30 * b


def _single(case, seed):
    g, kind = _gen(seed), case["kind"]
    if kind == "tridiag":
        return _banded(case["n"], 1, g, off_scale=0.3)
    if kind == "ode":
        return _ode(case["n"], float((0.5 + _rand(g, 1)) / 16.0))
    if kind == "banded":
        return _banded(case["n"], case["b"], g)
    if kind == "laplacian":
        return _laplacian(case["m"], case["dim"], float(0.45 + 0.1 * _rand(g, 1)))
    return _sprand(case["n"], 0.01, g)


def _opts(case):
    kw = {"tol": case["tol"], "filter": FILTERS[case["filter"]]}
    if "prec" in case:
        kw["prec"] = PRECS[case["prec"]]
    if case["kind"] == "ode":
        kw["scale_1norm"] = 0
    if case["kind"] == "nmf":
        kw["method"] = 1
    return kw


def _host(a):
    return SimpleNamespace(n=a.n, rowptr=a.rowptr.cpu().numpy(), col=a.col.cpu().numpy(),
                           val=a.val.cpu().numpy())


def _threshold_input(case, seed):
    """Magnitudes of an update: most of them far below the diagonal, over twelve decades; the
    budget drops the smaller part of them."""
    g = _gen(seed)
    n = case["nnz"]
    mag = torch.pow(10.0, -12.0 * _rand(g, n)) * torch.where(_rand(g, n) < 0.5, -1.0, 1.0)
    return mag, 1e-7 * math.sqrt(n)


def _gemm_input(case, seed):
    g = _gen(seed)
    dt = torch.float32 if case["kind"] == "gemm32" else torch.float64
    # entries of filled-in iterates: all magnitudes up to about 1, no structure left
    a = torch.randn(case["m"], case["k"], dtype=dt, device="cuda", generator=g)
    b = torch.randn(case["k"], case["n"], dtype=dt, device="cuda", generator=g)
    return a / math.sqrt(case["k"]), b


def prepare(case, seed):
    st = SimpleNamespace(case=dict(case), kind=case["kind"])
    if st.kind == "threshold":
        st.x, st.b = _threshold_input(case, seed)
        return st
    if st.kind in ("gemm32", "gemm64"):
        st.a, st.b = _gemm_input(case, seed)
        st.out = torch.empty(case["m"], case["n"], dtype=st.a.dtype, device="cuda")
        return st
    st.opts = sg.default_opts(**_opts(case))
    if st.kind != "batch":
        a = _single(case, seed)
        host = case.get("where") == "host"
        st.a = _host(a) if host else a
        if st.kind not in ("laplacian", "nmf"):  # the caller's own result arrays, kept across calls
            room = a.n * min(a.n, _row_room(case.get("b", 2), case["tol"]))
            st.col, st.val = ((np.zeros(room, np.int32), np.zeros(room)) if host else
                              (torch.zeros(room, dtype=torch.int32, device="cuda"),
                               torch.zeros(room, dtype=torch.float64, device="cuda")))
        return st
    # a batch: CSR arrays in pinned host memory, results into pinned host buffers
    g = _gen(seed)
    shapes = _batch_shapes(case)
    mats = [_banded(n, b, g) for n, b in shapes]
    rp = torch.cat([m.rowptr for m in mats]).cpu().pin_memory().numpy()
    col = torch.cat([m.col for m in mats]).cpu().pin_memory()
    val = torch.cat([m.val for m in mats]).cpu().pin_memory()
    st.keep = (rp, col, val)
    col, val = col.numpy(), val.numpy()
    st.mats, r0, e0 = [], 0, 0
    for n, b in shapes:
        nz = int(rp[r0 + n])
        st.mats.append(SimpleNamespace(n=n, rowptr=rp[r0:r0 + n + 1], col=col[e0:e0 + nz],
                                       val=val[e0:e0 + nz]))
        r0, e0 = r0 + n + 1, e0 + nz
    room = sum(n * min(n, _row_room(b, case["tol"])) for n, b in shapes)
    st.rp = torch.zeros(r0, dtype=torch.int64, pin_memory=True)
    st.col = torch.zeros(room, dtype=torch.int32, pin_memory=True)
    st.val = torch.zeros(room, dtype=torch.float64, pin_memory=True)
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    if st.kind == "threshold":
        return {"tau": sg.threshold_exact(st.x, st.b)}
    if st.kind == "gemm32":
        return {"c": sg.dense_product(st.a, st.b, out=st.out)}
    if st.kind == "gemm64":
        return {"c": sg.dense_product_f64(st.a, st.b, out=st.out)}
    if st.kind == "batch":
        return _run_batch(st)
    dev = st.case.get("where") != "host"
    r = sg.solve(st.a, opts=st.opts, device_out=dev)
    if st.kind in ("laplacian", "nmf"):  # filled in: taken dense
        n = st.a.n
        s = torch.sparse_csr_tensor(r.rowptr, r.col.to(torch.int64), r.val, size=(n, n),
                                    check_invariants=False)
        return {"sign": s.to_dense(), "iters": r.iters, "status": r.status}
    nnz = len(r.col)
    st.col[:nnz], st.val[:nnz] = r.col, r.val
    return {"rowptr": r.rowptr, "col": st.col, "val": st.val, "iters": r.iters,
            "status": r.status}


def _run_batch(st):
    batch = sg.Batch(st.mats)
    try:
        info = batch.solve(st.opts)
        nnz = batch.result_nnz()
        rp, col, val = st.rp.numpy(), st.col.numpy(), st.val.numpy()
        outs, r0, e0 = [], 0, 0
        for m, nz in zip(st.mats, nnz):
            outs.append((rp[r0:r0 + m.n + 1], col[e0:e0 + nz], val[e0:e0 + nz]))
            r0, e0 = r0 + m.n + 1, e0 + nz
        batch.results(outs)
    finally:
        batch.close()
    return {"rowptr": st.rp, "col": st.col, "val": st.val,
            "iters": np.array([i[1] for i in info]), "status": np.array([i[0] for i in info])}


# ------------------------------------------------------------------ work
def _band_work(n, b, prec, tol):
    """(result entries per row, multiply-adds per row of all products) of a banded solve, from
    the entries per row that the iterates of such matrices have: X fills to about w of 15 b + 12
    (FP32 stage 2/3 of it) after two updates and stays there, X^2 has twice as many."""
    w = min(n, (15 * b + 12) * (1.0 if tol >= 1e-9 else 1.4))
    if prec == "mixed":
        s = w * 2 / 3
        return w, 4 * (s * s + s * 2 * s) + (s * s + s * 2 * s) + w * w
    return w, 5 * (w * w + w * 2 * w) + w * w


def work(case):
    kind = case["kind"]
    if kind == "threshold":
        return {"bytes": 8 * case["nnz"], "flops": 0}
    if kind in ("gemm32", "gemm64"):
        m, n, k = case["m"], case["n"], case["k"]
        e = 4 if kind == "gemm32" else 8
        return {"bytes": e * (m * k + k * n + m * n), "flops": 2 * m * n * k}
    if kind == "laplacian":
        n = case["m"] ** case["dim"]
        # about ten updates once it has filled in, two products each
        return {"bytes": 12 * (2 * case["dim"] + 1) * n + 8 * n * n, "flops": 20 * 2 * n ** 3}
    if kind == "nmf":
        n = case["n"]
        return {"bytes": 12 * (0.01 * n + 1) * n + 8 * n * n, "flops": 8 * 2 * n ** 3}
    if kind == "batch":
        shapes = _batch_shapes(case)
    elif kind == "ode":
        shapes = [(2 * case["n"], 1)]
    else:
        shapes = [(case["n"], case.get("b", 1))]
    by = fl = 0.0
    for n, b in shapes:
        w, madds = _band_work(n, b, case["prec"], case["tol"])
        by += 12 * n * (2 * b + 1 + w) + 16 * (n + 1)
        fl += 2 * n * madds
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------ 64-bit values
def _dense(a):
    d = torch.zeros(a.n, a.n, dtype=torch.float64, device="cuda")
    rows = torch.repeat_interleave(torch.arange(a.n, device="cuda"), a.rowptr[1:] - a.rowptr[:-1])
    d[rows, a.col.long()] = a.val
    return d


def exact(case, seed):
    kind = case["kind"]
    if kind == "threshold":
        x, b = _threshold_input(case, seed)
        s = torch.sort(x.abs())[0]
        over = torch.cumsum(s * s, 0) > b * b
        return {"tau": float(s[int(over.to(torch.int8).argmax())]) if bool(over[-1]) else math.inf}
    if kind in ("gemm32", "gemm64"):
        a, b = _gemm_input(case, seed)
        return {"c": a.double() @ b.double()}
    if kind == "laplacian":
        lam, v = torch.linalg.eigh(_dense(_single(case, seed)))
        return {"sign": (v * torch.sign(lam)) @ v.T, "iters": None, "status": None}
    if kind == "nmf":
        # Newton's iteration in 64 bits to its fixed point
        x = _dense(_single(case, seed))
        for _ in range(60):
            y = 0.5 * (x + torch.linalg.inv(x))
            if float((y - x).norm()) <= 1e-14 * float(y.norm()):
                break
            x = y
        return {"sign": y, "iters": None, "status": None}
    # Which entries a sparse result stores is decided by the filter during the iteration: there is
    # no 64-bit value laid out like it without this method's own steps.
    return None
