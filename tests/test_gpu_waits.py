"""How a solve waits for the device: many matrices' readbacks are copies, and a
process that asked for blocking waits gets them."""
import os
import pathlib
import subprocess
import sys

import pytest

import workloads as w

pytestmark = pytest.mark.gpu

ROOT = pathlib.Path(__file__).resolve().parent.parent


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


def test_large_readbacks_are_copies(sg):
    """The readback kernel is launched for the values of 700 matrices, not for
    those of 6000; otherwise the launches of a solve are the same."""
    launches, iters = {}, {}
    for count in (700, 6000):
        b = sg.Batch([w.tridiagonal(16)] * count)
        n0 = sg.kernel_launches()
        out = b.solve(sg.default_opts(tol=1e-8, filter="exact", dense_frac=2.0))
        launches[count] = sg.kernel_launches() - n0
        assert all(o == out[0] for o in out)
        iters[count] = out[0]
        b.close()
    assert iters[700] == iters[6000]
    # an iteration's check, its filter and (6000 alone) its two products
    assert launches[6000] <= launches[700] - 2 * iters[700][1]


CHILD = """
import ctypes, time
cu = ctypes.CDLL("libcuda.so.1")
assert cu.cuInit(0) == 0 and cu.cuDevicePrimaryCtxSetFlags(0, {flags}) == 0
import paper_2210_03356_gb300 as sg, workloads as w
b = sg.Batch([w.banded(4000, 10, i) for i in range(24)])
o = sg.default_opts(tol=1e-12, filter="exact")
b.solve(o)
t, c = time.perf_counter(), time.thread_time()
for _ in range(3):
    b.solve(o)
print((time.thread_time() - c) / (time.perf_counter() - t))
"""


@pytest.mark.parametrize("flags,most", [(4, 0.5), (0, 1.1), (2, 1.1)])
def test_scheduling_flags(sg, flags, most):
    """4: blocking waits, the waiting thread sleeps (mostly: the products' kernels are
    long); 0 and 2, the default and yield: the same results, whatever the load."""
    r = subprocess.run([sys.executable, "-c", CHILD.format(flags=flags)], cwd=ROOT,
                       env=dict(os.environ, PYTHONPATH=str(ROOT)), capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr
    assert float(r.stdout) < most
