"""Poles closer to one another than FP32's range below the largest (1e-40 to 1e-60
against 1): the FP32 opening cannot tell them apart, but their terms count for the
eigenvalues further off.  All eigenpairs against the oracle, 10 n eps64."""
import numpy as np
import pytest

import oracle
from parity import assert_parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ae():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1302_7203_gb300 import arrowhead, build
    build.build()
    return arrowhead


def tiny_poles(k, sign, equal):
    rng = np.random.default_rng(k)
    d = np.sort(sign * np.append(10.0 ** -rng.uniform(40, 60, k), [1.0, 0.5, 0.7]))[::-1].copy()
    return d, np.ones(k + 3) if equal else rng.uniform(0.1, 1.0, k + 3)


@pytest.mark.parametrize("form", [{}, {"precision": 1, "finish": 1, "bgate": 1}])
@pytest.mark.parametrize("alpha", [0.5, 0.0, 3.0])
@pytest.mark.parametrize("k, sign, equal", [(2, -1, False), (2, -1, True), (900, 1, True)])
def test_poles_below_the_fp32_range(ae, k, sign, equal, alpha, form):
    d, z = tiny_poles(k, sign, equal)
    t = lambda x: torch.as_tensor(x, device="cuda")
    r = ae.arrow_eig(t(d), t(z), alpha, opts=ae.default_opts(**form))
    assert_parity(r["lam"].cpu().numpy(), r["V"].cpu().numpy(), oracle.arrow_eig(d, z, alpha),
                  k + 4, what=f"{k} tiny poles, alpha {alpha}")


@pytest.mark.parametrize("form", [{}, {"precision": 1, "finish": 1, "bgate": 1}])
@pytest.mark.parametrize("alpha", [-1e6, -0.5])
@pytest.mark.parametrize("ratio", [1.006, 1.2])
def test_last_eigenvalue_far_below_crowded_poles(ae, ratio, alpha, form):
    # (at the last pole itself FP32 sums of squares come near its largest number)
    m = 942
    d = np.maximum(ratio ** -np.arange(m, dtype=float), 1e-40)
    d = np.sort(d * (1 + 1e-3 * np.random.default_rng(3).random(m)))[::-1].copy()
    t = lambda x: torch.as_tensor(x, device="cuda")
    r = ae.arrow_eig(t(d), t(np.ones(m)), alpha, opts=ae.default_opts(**form))
    assert_parity(r["lam"].cpu().numpy(), r["V"].cpu().numpy(),
                  oracle.arrow_eig(d, np.ones(m), alpha), m + 1,
                  what=f"crowded poles, ratio {ratio} alpha {alpha}")
