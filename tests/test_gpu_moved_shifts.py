"""Eigenvalues far nearer the remedy's shift than the shift pole: moved by a
subtraction, they need the zero beyond double precision.  A DPR1's last eigenvalue
next to its last pole (small u: the offset is about rho u^2; below 1e-7 the corner
of the arrowhead, a double-double, limits it for every solver), an arrowhead's
eigenvalue next to zero.  Small orders, so that 10 n eps64 is a sharp bar."""
import numpy as np
import pytest

import oracle
from parity import assert_parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FORMS = [{}, {"precision": 1, "finish": 1, "bgate": 1}]


@pytest.fixture(scope="module")
def ae():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1302_7203_gb300 import arrowhead, build
    build.build()
    return arrowhead


def t(x):
    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("size", [1e-3, 1e-6, 1e-7])
@pytest.mark.parametrize("n", [3, 5, 17])
def test_dpr1_next_to_its_last_pole(ae, n, size, form):
    for seed in range(12):
        rng = np.random.default_rng([n, seed])
        d = np.sort(rng.uniform(-1, 3, n))[::-1].copy()
        u = size * rng.uniform(0.1, 1.0, n)
        for rho in (0.5, -0.5):
            ref = oracle.dpr1_eig(d, u, rho)
            r = ae.dpr1_eig(t(d), t(u), rho, opts=ae.default_opts(**form))
            assert_parity(r["lam"].cpu().numpy(), r["Q"].cpu().numpy(),
                          {"lam": ref["lam"], "abserr": np.zeros(n), "V": ref["Q"]}, n,
                          what=f"dpr1 n={n} u={size} seed {seed} rho {rho}")


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("off", [1e-3, 1e-6, 1e-9, 1e-12])
@pytest.mark.parametrize("n", [4, 9, 33])
def test_eigenvalue_next_to_zero(ae, n, off, form):
    for seed in range(12):
        rng = np.random.default_rng([n, seed])
        d = np.sort(rng.choice([-1.0, 1.0], n - 1) * rng.uniform(0.5, 3, n - 1))[::-1].copy()
        z = rng.uniform(0.1, 1.0, n - 1)
        a = float(np.sum(z * z / d)) * (1 + off) + off
        o = oracle.arrow_eig(d, z, a)
        r = ae.arrow_eig(t(d), t(z), a, opts=ae.default_opts(**form))
        assert_parity(r["lam"].cpu().numpy(), r["V"].cpu().numpy(), o, n,
                      what=f"near zero n={n} off={off} seed {seed}")
