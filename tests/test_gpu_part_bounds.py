"""A part of a split solve writes inside its own block, whatever the input: rows that
are not finite leave eigenvalues NaN, which compare with no deflated value."""
import numpy as np
import pytest

from paper_1302_7203_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ae():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1302_7203_gb300 import arrowhead, build
    build.build()
    return arrowhead


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("max_iter", [99, 1000])
def test_bad_input_stays_in_the_block(ae, value, max_iter):
    n, guard = 301, 400
    d, z, a = W.uniform_arrow(n, seed=3)
    d, z = d.copy(), z.copy()
    z[::4] = 0.0                                  # 75 deflated rows before the last part
    d[7] = value
    t = lambda x: torch.as_tensor(x, device="cuda")
    for part in range(3):
        p0, cnt = ae.arrow_eig_part_size(t(d), t(z), part, 3)
        assert 0 <= p0 and 0 < cnt <= n
        lam = torch.full((cnt + 2 * guard,), 7.0, dtype=torch.float64, device="cuda")
        V = torch.full((cnt + 2 * guard, n), 7.0, dtype=torch.float64, device="cuda")
        with pytest.raises(ae.AeError) as e:
            ae.arrow_eig_part(t(d), t(z), a, part, 3, info=True,
                              opts=ae.default_opts(max_iter=max_iter),
                              out={"lam": lam[guard:guard + cnt], "V": V[guard:guard + cnt]})
        assert e.value.status == ae.AE_ERR_INPUT
        for x in (lam, V):
            assert bool((x[:guard] == 7.0).all()) and bool((x[guard + cnt:] == 7.0).all())
