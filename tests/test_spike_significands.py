"""zeta^2 whose rounded value is a power of two with a negative low part.

Spikes of unit modulus (Hermitian), products zc (1 / zc) (non-symmetric) and
d (1 / d) (SVD) give many of them: the significand then lies just below its
leading bit.
CPU: the 64-bit significand against exact integers, at powers of two and their
neighbours with low parts of both signs up to half a last place.
GPU: eigenpairs of such inputs against the oracle at the suite's bar, 10 n eps64,
with and without far poles taken as moments (768 poles and more).
"""
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_1302_7203_gb300 import workloads as W
from parity import assert_parity

HARNESS = r"""
#include "ae_fixed.cuh"
#include <cmath>
#include <cstdio>
using namespace ae;
int main() {
    int bad = 0, n = 0;
    for (int e = -300; e <= 300; e += 7)
        for (int s = -2; s <= 2; ++s) {             // a power of two and its neighbours
            double hi = std::ldexp(1.0, e);
            for (int i = 0; i < std::abs(s); ++i) hi = std::nextafter(hi, s > 0 ? 1e308 : 0.0);
            const int eh = std::ilogb(hi);
            // half the gap below a power of two is half of the one above
            const long long below = s == 0 ? 512 : 1024;
            for (long long lo = -below; lo <= 1024; lo += 64) {
                const unsigned __int128 want =
                    (unsigned __int128)(long long)std::ldexp(hi, 52 - eh) * 2048 + (__int128)lo;
                bad += (unsigned __int128)fix_mant(hi, lo) != want;
                ++n;
            }
        }
    std::printf("%d %d\n", n, bad);
    return 0;
}
"""


def test_significand_on_the_host(tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    src = tmp_path / "h.cpp"
    src.write_text(HARNESS)
    exe = tmp_path / "h"
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I",
                           os.path.join(root, "paper_1302_7203_gb300", "csrc"), str(src), "-o",
                           str(exe)])
    n, bad = subprocess.check_output([str(exe)]).split()
    assert int(n) > 10000 and int(bad) == 0


@pytest.fixture(scope="module")
def ae():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1302_7203_gb300 import arrowhead, build
    build.build()
    return arrowhead


def t(x):
    import torch
    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


@pytest.mark.gpu
@pytest.mark.parametrize("n", [3, 300, 900])
def test_unit_moduli(ae, n):
    rng = np.random.default_rng(n)
    d, _, a = W.uniform_arrow(n, seed=n)
    z = np.exp(1j * rng.uniform(0.0, 2.0 * np.pi, n - 1))
    o = oracle.herm_eig(d, z, a)
    r = ae.herm_arrow_eig(t(d), t(z), a)
    assert_parity(r["lam"].cpu().numpy(), r["U"].cpu().numpy(), {**o, "V": o["U"]}, n,
                  what="herm, unit moduli")
    zc = np.where(rng.random(n - 1) < 0.5, -1.0, 1.0) * rng.uniform(0.2, 5.0, n - 1)
    o = oracle.nsym_eig(d, zc, 1.0 / zc, a)
    r = ae.nsym_arrow_eig(t(d), t(zc), t(1.0 / zc), a)
    for key in ("X", "Y"):
        assert_parity(r["lam"].cpu().numpy(), r[key].cpu().numpy(), {**o, "V": o[key]}, n,
                      what=f"nsym, zr = 1 / zc, {key}")
    d, _, a = W.uniform_tsvd(n, seed=n)
    o = oracle.tsvd(d, 1.0 / d, a)
    r = ae.tri_arrow_svd(t(d), t(1.0 / d), a)
    for key in ("V", "U"):
        assert_parity(r["s"].cpu().numpy(), r[key].cpu().numpy(),
                      {"lam": o["s"], "abserr": np.zeros(n), "V": o[key]}, n,
                      what=f"svd, z = 1 / d, {key}")
