"""Eigenpairs the fixed-point passes refuse and the FP64 solver takes: inputs whose
exponents they do not serve (scaled by 2^500), poles 2^-40 apart, spikes over 20
decades.  Such an eigenpair has the same bits in a solve alone, a part and a batch
or merged pass with many of them, remedied ones excepted (10 n eps64)."""
import numpy as np
import pytest

import oracle
from paper_1302_7203_gb300 import workloads as W
from parity import assert_parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FORMS = {"plain": {}, "fast": dict(precision=1, finish=1, bgate=1)}
REMEDY = 2 | 4 | 8


@pytest.fixture(scope="module")
def ae():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1302_7203_gb300 import arrowhead, build
    build.build()
    return arrowhead


def t(x):
    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


def data(case, n, seed=0):
    rng = np.random.default_rng(1000 * n + seed)
    d, z, a = W.uniform_arrow(n, seed=n + seed)
    if case == "scaled":
        s = 2.0 ** 500
        return d * s, z * s, a * s
    if case == "clusters":
        c = np.linspace(-5, 5, (n - 1 + 9) // 10)
        d = np.sort((c[:, None] * (1 + 2.0 ** -40 * np.arange(1, 11))).ravel())[::-1]
        return d[:n - 1].copy(), z, a
    if case == "one":
        z = z.copy()
        z[(n - 1) // 2] = 1e-18
        return d, z, a
    return d, 10.0 ** rng.uniform(-20, 0, n - 1), a


def alone(ae, d, z, a, form):
    r = ae.arrow_eig(t(d), t(z), a, opts=ae.default_opts(**FORMS[form]), diag=True)
    return r["lam"], r["V"], (r["diag"]["flags"] & REMEDY) == 0


def same(lam, V, ref, n):
    rl, rV, keep = ref
    assert torch.equal(lam[keep], rl[keep]) and torch.equal(V[:, keep], rV[:, keep])
    tol = 10 * n * 2.0 ** -53
    assert torch.all((lam - rl).abs() <= tol * rl.abs())
    assert torch.all((V - rV).abs() <= tol * rV.abs() + 1e-300)


@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("case", ["scaled", "clusters", "spikes", "one"])
@pytest.mark.parametrize("n", [2, 200, 769, 1100])
def test_refused_pairs(ae, n, case, form):
    d, z, a = data(case, n)
    ref = alone(ae, d, z, a, form)
    assert_parity(ref[0].cpu().numpy(), ref[1].cpu().numpy(), oracle.arrow_eig(d, z, a), n,
                  what=f"refused {case} n={n} {form}")
    parts = [ae.arrow_eig_part(t(d), t(z), a, p, 3, opts=ae.default_opts(**FORMS[form]))
             for p in range(3)]
    same(torch.cat([p["lam"] for p in parts]), torch.cat([p["V"] for p in parts], dim=1), ref, n)


@pytest.mark.parametrize("form", sorted(FORMS))
def test_refused_pairs_of_a_batch(ae, form):
    # over 9000 of them in one pass, and orders on both sides of every team rule
    inst = [data("scaled", 500, seed=i) for i in range(16)]
    inst += [data(c, n, seed=7) for c in ("clusters", "spikes", "one") for n in (60, 900)]
    b = ae.Batch(inst, opts=ae.default_opts(**FORMS[form]))
    b.run()
    torch.cuda.synchronize()
    for i in (0, 15, 16, 17, 18, 19, 20, 21):
        same(b.lam(i), b.V(i), alone(ae, *inst[i], form), len(inst[i][0]) + 1)
    b.close()


def test_refused_pairs_of_a_merged_pass(ae):
    srv = ae.Server(budget_bytes=64 << 30, max_inflight=1)
    D, Z, A = W.graded_arrow(8000, seed=2)
    small = [data(c, n, seed=3) for c in ("scaled", "clusters", "spikes", "one")
             for n in (90, 300, 900)]
    dev = [(t(d), t(z), a) for d, z, a in small]
    Dt, Zt = t(D), t(Z)
    torch.cuda.synchronize()
    srv.submit(0, Dt, Zt, A, vectors=False)
    tk = [srv.submit(0, *x) for x in dev]
    for k, (d, z, a) in zip(tk, small):
        assert srv.wait(k)[0] == ae.REQ_DONE
        got = srv.result(k)
        same(got["lam"], got["V"], alone(ae, d, z, a, "plain"), len(d) + 1)
    assert srv.stats()["merged"] >= 2
    srv.close()
