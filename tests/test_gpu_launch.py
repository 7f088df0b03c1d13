"""Kernels placed before their predecessors have ended: every one of them waits
for the one before it, whatever launched that. Checked through the sources, and
by solves queued between copies and on several streams at once."""
import pathlib
import re
import threading

import numpy as np
import pytest

import workloads as w

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2210_03356_gb300" / "csrc"


def test_every_early_kernel_waits_first():
    """A kernel that launch_next launches has after_previous() as its first
    statement, before any early return."""
    text = "\n".join(p.read_text() for p in sorted(CSRC.glob("*.cu")))
    early = set(re.findall(r"launch_next\((k_\w+)", text))
    # launched through a name of their own
    early |= {"k_bounds", "k_lu_trail"}
    assert "k_publish" in early and len(early) > 30
    for name in early:
        bodies = re.findall(r"\b%s\((?:const |unsigned |int|double|float|T |Rows|SelRows|ScanJobs)"
                            r"[^{;]*\)\s*\{\s*([^\n]*)" % name, text)
        assert bodies and all(b.strip() == "after_previous();" for b in bodies), (name, bodies)


@pytest.mark.gpu
def test_solves_on_several_streams():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    import paper_2210_03356_gb300 as sg
    from paper_2210_03356_gb300 import build
    build.build()
    sg.load()
    oracle.build()
    mats = [w.tridiagonal(500), w.banded(700, 4, 11), w.banded(300, 9, 12), w.tridiagonal(1)]
    refs = [oracle.nsf(a, tol=1e-8, filter="exact") for a in mats]
    bad = []

    def work(k):
        a, ref = mats[k], refs[k]
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(20):
                r = sg.solve(a, tol=1e-8, filter="exact", dense_frac=2.0)
                if not (r.iters == ref.iters and np.array_equal(r.col, ref.col)
                        and np.array_equal(r.val.view(np.uint64), ref.val.view(np.uint64))):
                    bad.append(k)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(mats))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
