"""A solve reads nothing of its scratch memory that it has not written: the bits
of the results are the same whatever the stream-ordered pool's memory held.

The pool is primed by a block larger than the solve's, filled with 1.0 in every
other stretch of two scratch arrays (so that, of two arrays two apart in the
layout, one holds 1.0 and the other 0) and freed on the stream just before the
solve; a second run has the stretches swapped.  Inputs: outermost eigenvalues and
openings that need a further model step, sums that cancel.
"""
import ctypes

import numpy as np
import pytest

from paper_1302_7203_gb300 import workloads as W
from test_zz_no_alloc import _cudart

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ae():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1302_7203_gb300 import arrowhead, build
    build.build()
    return arrowhead


def t(x):
    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


def data(case):
    if case == "uniform900":
        return W.uniform_arrow(900, seed=3)
    if case == "graded1000":
        return W.graded_arrow(1000, seed=4)
    rng = np.random.default_rng(5)
    d = np.sort(np.linspace(1.0, -1.0, 800) + rng.uniform(-1e-4, 1e-4, 800))[::-1].copy()
    return d, 10.0 ** rng.uniform(-6, 0, 800), 0.0


def prime(ae, rt, n, swap):
    words = 32 << 17                                       # 32 MB
    p = ctypes.c_void_p()
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert rt.cudaMallocAsync(ctypes.byref(p), ctypes.c_size_t(8 * words), s) == 0
    view = torch.as_tensor(ae._DeviceView(p.value, (words,)), device="cuda")
    stretch = 2 * ((8 * n + 255) // 256 * 32)              # two arrays of n doubles
    odd = torch.arange(words, device="cuda") // stretch % 2 == (0 if swap else 1)
    view.copy_(odd.to(torch.float64))
    torch.cuda.synchronize()
    del view
    assert rt.cudaFreeAsync(p, s) == 0


@pytest.mark.parametrize("form", [{}, {"precision": 1, "finish": 1, "bgate": 1}])
@pytest.mark.parametrize("case", ["uniform900", "graded1000", "cancelling"])
def test_results_do_not_depend_on_old_memory(ae, case, form):
    rt = _cudart()
    d, z, a = data(case)
    n = len(d) + 1
    dt, zt = t(d), t(z)
    runs = []
    for swap in (False, True):
        out = {"lam": torch.empty(n, dtype=torch.float64, device="cuda"),
               "V": torch.empty((n, n), dtype=torch.float64, device="cuda")}
        prime(ae, rt, n, swap)
        ae.arrow_eig(dt, zt, a, opts=ae.default_opts(**form), out=out)
        torch.cuda.synchronize()
        runs.append(out)
    assert torch.equal(runs[0]["lam"], runs[1]["lam"])
    assert torch.equal(runs[0]["V"], runs[1]["V"])
