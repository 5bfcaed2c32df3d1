"""The FP64 solver by itself (csrc/ae_solver.cuh): an iteration cap below 100 sends
every eigenpair of every kind to it, in each of its forms -- Algorithm 3's
bisection or the Newton finish, all-FP64 or with FP32 openings, b in double-double
or under Algorithm 5's gate -- and in batched plans and one-shot batches.  Inputs
have deflated rows, runs of equal poles and eigenpairs that remedies move, so that
columns written with the solve have to be written again.  Against the oracle at the
suite's bar, 10 n eps64.  What the options choose is visible in the counters here:
bisection takes many steps an eigenpair, fewer after an FP32 bracket, and a Newton
finish a handful.
"""
import numpy as np
import pytest

import oracle
from paper_1302_7203_gb300 import workloads as W
from parity import assert_parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FORMS = {"bisect": dict(), "bisect32": dict(precision=1), "newton": dict(finish=1),
         "gated": dict(precision=1, finish=1, bgate=1)}


@pytest.fixture(scope="module")
def ae():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1302_7203_gb300 import arrowhead, build
    build.build()
    return arrowhead


def t(x):
    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


def messy(d, z, seed):
    """Zero spikes, equal poles, rows in no order."""
    rng = np.random.default_rng(seed)
    d, z = d.copy(), z.copy()
    m = d.size
    z[rng.random(m) < 0.1] = 0.0
    tie = np.nonzero(rng.random(m) < 0.1)[0]
    d[tie] = d[rng.integers(0, m, tie.size)]
    p = rng.permutation(m)
    return d[p], z[p]


def arrow(case, n):
    if case == "graded":
        return W.graded_arrow(n, seed=n)
    d, z, a = W.uniform_arrow(n, seed=n)
    if case == "messy":
        d, z = messy(d, z, n)
    return d, z, a


def check(r, lam, pairs, n, what):
    for got, want in pairs:
        assert_parity(r[lam[0]].cpu().numpy(), r[got].cpu().numpy(),
                      {"abserr": np.zeros(n), **lam[1], "V": want}, n, what=f"{what} {got}")
    assert r["info"]["n_capped"] == 0


# (bisection of a graded matrix may need more than 99 steps)
CASES = [(c, f) for c in ("uniform", "messy") for f in sorted(FORMS)] + \
    [("graded", "newton"), ("graded", "gated")]


@pytest.mark.parametrize("case, form", CASES)
@pytest.mark.parametrize("n", [5, 33, 300])
def test_arrow(ae, n, case, form):
    d, z, a = arrow(case, n)
    r = ae.arrow_eig(t(d), t(z), a, opts=ae.default_opts(max_iter=99, **FORMS[form]), info=True)
    o = oracle.arrow_eig(d, z, a)
    check(r, ("lam", o), [("V", o["V"])], n, f"arrow {case} {form}")
    steps = r["info"]["total_iter"] - r["info"]["fix_iter"]
    pairs = r["info"]["n_reduced"]
    if form == "bisect":
        assert steps > 25 * pairs
    elif form == "bisect32":
        assert steps < 40 * pairs
    else:
        assert steps < 10 * pairs


@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("kind", ["dpr1", "dpr1-", "svd", "herm", "nsym"])
@pytest.mark.parametrize("case", ["uniform", "messy"])
def test_other_kinds(ae, kind, case, form):
    n = 301
    o = ae.default_opts(max_iter=99, **FORMS[form])
    what = f"{kind} {case} {form}"
    if kind.startswith("dpr1"):
        d, u, rho = W.uniform_dpr1(n, seed=5)
        if case == "messy":
            d, u = messy(d, u, 5)
        rho = -rho if kind == "dpr1-" else rho
        ref = oracle.dpr1_eig(d, u, rho)
        r = ae.dpr1_eig(t(d), t(u), rho, opts=o, info=True)
        check(r, ("lam", {"lam": ref["lam"]}), [("Q", ref["Q"])], n, what)
    elif kind == "svd":
        d, z, a = W.uniform_tsvd(n, seed=5)
        ref = oracle.tsvd(d, z, a)
        if case == "messy":                  # (the oracle takes distinct d in order)
            p = np.random.default_rng(5).permutation(n - 1)
            d, z, q = d[p], z[p], np.append(p, n - 1)
            ref["U"], ref["V"] = ref["U"][q], ref["V"][q]
        r = ae.tri_arrow_svd(t(d), t(z), a, opts=o, info=True)
        check(r, ("s", {"lam": ref["s"]}), [("V", ref["V"]), ("U", ref["U"])], n, what)
    elif kind == "herm":
        d, z, a = W.uniform_herm(n, seed=5)
        if case == "messy":
            d, z = messy(d, z, 5)
        ref = oracle.herm_eig(d, z, a)
        r = ae.herm_arrow_eig(t(d), t(z), a, opts=o, info=True)
        check(r, ("lam", ref), [("U", ref["U"])], n, what)
    else:
        d, zc, zr, a = W.uniform_nsym(n, seed=5)
        if case == "messy":
            f = zr / zc
            d, zc = messy(d, zc, 5)
            zr = zc * f
        ref = oracle.nsym_eig(d, zc, zr, a)
        r = ae.nsym_arrow_eig(t(d), t(zc), t(zr), a, opts=o, info=True)
        check(r, ("lam", ref), [("X", ref["X"]), ("Y", ref["Y"])], n, what)


@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("graph", [True, False])
def test_batches(ae, graph, form):
    inst = [arrow(c, n) for c, f in CASES if f == form for n in (2, 7, 40, 300)]
    b = ae.Batch(inst, opts=ae.default_opts(max_iter=99, **FORMS[form]), graph=graph)
    b.run()
    torch.cuda.synchronize()
    for i, (d, z, a) in enumerate(inst):
        o = oracle.arrow_eig(d, z, a)
        assert_parity(b.lam(i).cpu().numpy(), b.V(i).cpu().numpy(), o, len(d) + 1,
                      what=f"batch {i} {form}")
    b.close()


@pytest.mark.parametrize("form", sorted(FORMS))
def test_parts(ae, form):
    d, z, a = arrow("messy", 301)
    o = oracle.arrow_eig(d, z, a)
    parts = [ae.arrow_eig_part(t(d), t(z), a, p, 3,
                               opts=ae.default_opts(max_iter=99, **FORMS[form]))
             for p in range(3)]
    assert_parity(torch.cat([p["lam"] for p in parts]).cpu().numpy(),
                  torch.cat([p["V"] for p in parts], dim=1).cpu().numpy(), o, 301,
                  what=f"parts {form}")
