"""The work that users of this framework have it do, as measurable cases.

A case is one call (or one burst of calls) through the public entry points of
``paper_1302_7203_gb300.arrowhead``.  Inputs follow the recipes of the
package's ``workloads`` module (uniform, graded, quantum-dot-like spectra; the
DPR1, SVD, Hermitian, non-symmetric and batched sets), drawn here from the
case's seed.  Two forms are in earnest use: ``plain`` (the library defaults:
Algorithm 3's bisection, b in double-double) and ``fast`` (FP32 opening,
Algorithm 5's gates, bracketed Newton finish), the form of the benchmark.
"""
import math

import numpy as np
import torch

from paper_1302_7203_gb300 import arrowhead as ae

FORMS = {"plain": {}, "fast": {"precision": 1, "finish": 1, "bgate": 1}}
DEV = "cuda"


def listed():
    return [
        # one small matrix in a caller's loop: latency and launches
        {"name": "arrow-64-plain", "kind": "arrow", "spectrum": "uniform", "n": 64,
         "form": "plain", "vectors": True},
        # the plain method on the order-1000 uniform arrowhead
        {"name": "arrow-1000-plain", "kind": "arrow", "spectrum": "uniform", "n": 1000,
         "form": "plain", "vectors": True},
        # the plain method on a graded matrix of odd order
        {"name": "arrow-graded-4097-plain", "kind": "arrow", "spectrum": "graded", "n": 4097,
         "form": "plain", "vectors": True},
        # the benchmark: graded, all eigenpairs and the 2 GiB V
        {"name": "arrow-graded-16384", "kind": "arrow", "spectrum": "graded", "n": 16384,
         "form": "fast", "vectors": True},
        # eigenvalues alone of unsorted input with zero spikes and equal poles
        {"name": "arrow-values-6001-messy", "kind": "arrow", "spectrum": "messy", "n": 6001,
         "form": "fast", "vectors": False},
        # the rank-one update of a divide-and-conquer merge
        {"name": "dpr1-8192", "kind": "dpr1", "spectrum": "uniform", "n": 8192, "form": "fast",
         "vectors": True},
        # singular triplets of a triangular arrowhead (SVD updating)
        {"name": "svd-8192", "kind": "svd", "spectrum": "uniform", "n": 8192, "form": "fast",
         "vectors": True},
        # Hermitian arrowhead, complex vectors, odd order
        {"name": "herm-3001", "kind": "herm", "spectrum": "uniform", "n": 3001, "form": "fast",
         "vectors": True},
        # non-symmetric arrowhead of the quantum-dot order, right and left vectors
        {"name": "nsym-2501", "kind": "nsym", "spectrum": "graded", "n": 2501, "form": "fast",
         "vectors": True},
        # host arrays in, page-locked host arrays out (a caller without device data)
        {"name": "host-4096", "kind": "host", "spectrum": "uniform", "n": 4096, "form": "fast",
         "vectors": True},
        # a captured plan over many arrowheads of uneven order
        {"name": "batch-512", "kind": "batch", "spectrum": "uniform", "count": 512, "lo": 32,
         "hi": 4096, "form": "fast", "graph": True, "vectors": True},
        # a burst of mixed requests through the serving loop
        {"name": "serve-burst-20", "kind": "serve", "spectrum": "uniform", "count": 20, "lo": 64,
         "hi": 8192, "form": "fast", "vectors": True},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["arrow", "arrow", "arrow", "dpr1", "svd", "herm", "nsym", "host", "batch",
                       "serve"])
    form = rng.choice(["plain", "fast", "fast"])
    case = {"kind": kind, "spectrum": "uniform", "form": form, "vectors": True}
    if kind == "batch":
        lo = _log_int(rng, 16, 256)
        hi = _log_int(rng, 2 * lo, 16 * lo)
        case.update(lo=lo, hi=hi, count=_log_int(rng, 16, max(16, min(2048, (1 << 28) // (hi * hi)))),
                    graph=rng.random() < 0.7)
        return case
    if kind == "serve":
        lo = _log_int(rng, 48, 256)
        case.update(form="fast", lo=lo, hi=_log_int(rng, 2 * lo, 4096), count=rng.randint(8, 20))
        return case
    top = 6000 if form == "plain" else 16384 if kind == "arrow" else 9000
    case["n"] = _log_int(rng, 40, top)
    if kind in ("arrow", "host"):
        case["spectrum"] = rng.choice(["uniform", "graded", "qdot", "messy"])
    elif kind in ("herm", "nsym"):
        case["spectrum"] = rng.choice(["uniform", "graded"])
    if kind == "arrow":
        case["vectors"] = rng.random() < 0.75
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _desc_distinct(f, count, rng):
    v = f(count)
    for _ in range(100):
        v = np.sort(v)[::-1].copy()
        dup = np.nonzero(v[1:] == v[:-1])[0]
        if not dup.size:
            return v
        v[dup + 1] = f(dup.size)
    return v


def _arrow(spectrum, n, rng):
    """(d, z, alpha) of order n."""
    m = n - 1
    if spectrum == "graded":
        d = _desc_distinct(lambda c: np.where(rng.random(c) < 0.5, -1.0, 1.0) *
                           10.0 ** rng.uniform(-15, 0, c), m, rng)
        return d, 10.0 ** rng.uniform(-10, 0, m), 1e3
    if spectrum == "qdot":
        d = _desc_distinct(lambda c: rng.uniform(5.87e14, 1.38e15, c), m, rng)
        z = 10.0 ** rng.uniform(math.log10(1.05e4), math.log10(1.10e7), m)
        return d, z, 9.7949881500060375e14
    d = _desc_distinct(lambda c: rng.uniform(-10, 10, c), m, rng)
    z = 1.0 - rng.random(m)
    if spectrum == "messy":
        # rows in no order, signs mixed, a tenth of the spikes zero and a tenth
        # of the rows sharing another row's pole
        d = rng.permutation(d)
        z = z * np.where(rng.random(m) < 0.5, -1.0, 1.0)
        z[rng.random(m) < 0.1] = 0.0
        tie = np.nonzero(rng.random(m) < 0.1)[0]
        d[tie] = d[rng.integers(0, m, tie.size)]
    return d, z, float(rng.standard_normal())


def _inputs(kind, spectrum, n, rng):
    if kind == "dpr1":
        d = _desc_distinct(lambda c: rng.uniform(0, 1, c), n, rng)
        u = rng.standard_normal(n)
        return d, u / np.linalg.norm(u), 0.5
    if kind == "svd":
        d = _desc_distinct(lambda c: 1.0 - rng.random(c), n - 1, rng)
        return d, rng.standard_normal(n - 1), float(1.0 - rng.random())
    d, z, alpha = _arrow(spectrum, n, rng)
    if kind == "herm":
        return d, z * np.exp(1j * rng.uniform(0, 2 * np.pi, n - 1)), alpha
    if kind == "nsym":
        zc = np.where(rng.random(n - 1) < 0.5, -1.0, 1.0) * z
        return d, zc, zc * 10.0 ** rng.uniform(-2, 2, n - 1), alpha
    return d, z, alpha


def _sizes(case, rng):
    lo, hi = case["lo"], case["hi"]
    if case["kind"] == "serve":
        # the orders are part of the workload, not of the data: evenly spread
        q = (np.arange(case["count"]) * 7 % case["count"] + 0.5) / case["count"]
    else:
        q = (rng.permutation(case["count"]) + 0.5) / case["count"]
    return np.clip(np.rint(lo * (hi / lo) ** q).astype(int), lo, hi)


def _many(case, seed):
    """[(kind, d, z, alpha)] of a batch or a burst."""
    rng = np.random.default_rng(seed)
    kinds = ("arrow", "dpr1", "svd") if case["kind"] == "serve" else ("arrow",)
    return [(kinds[i % len(kinds)],) + _inputs(kinds[i % len(kinds)], case["spectrum"], int(n), rng)
            for i, n in enumerate(_sizes(case, rng))]


def _one(case, seed):
    return _inputs(case["kind"], case["spectrum"], case["n"], np.random.default_rng(seed))


def _up(x):
    return torch.as_tensor(np.ascontiguousarray(x), device=DEV)


def prepare(case, seed):
    kind = case["kind"]
    opts = ae.default_opts(**FORMS[case["form"]])
    if kind == "batch":
        inst = [x[1:] for x in _many(case, seed)]
        return {"case": case, "batch": ae.Batch(inst, opts=opts, graph=case["graph"])}
    if kind == "serve":
        reqs = [(k, _up(d), _up(z), a) for k, d, z, a in _many(case, seed)]
        return {"case": case, "reqs": reqs,
                "server": ae.Server(64 << 30, max_inflight=16, opts=opts)}
    x = _one(case, seed)
    n = case["n"]
    st = {"case": case, "opts": opts}
    if kind == "host":
        st["in"] = tuple(torch.as_tensor(v).pin_memory() for v in x[:2]) + (x[2],)
        st["out"] = {"lam": torch.empty(n, dtype=torch.float64).pin_memory(),
                     "V": torch.empty((n, n), dtype=torch.float64).pin_memory()}
        return st
    st["in"] = tuple(_up(v) for v in x[:-1]) + (x[-1],)
    # the output buffers that a caller with a steady stream of solves reuses
    dt = torch.complex128 if kind == "herm" else torch.float64
    names = {"arrow": ("lam", "V"), "dpr1": ("lam", "Q"), "svd": ("s", "U", "V"),
             "herm": ("lam", "U"), "nsym": ("lam", "X", "Y")}[kind]
    st["out"] = {names[0]: torch.empty(n, dtype=torch.float64, device=DEV)}
    if case["vectors"]:
        st["out"].update({k: torch.empty((n, n), dtype=dt, device=DEV) for k in names[1:]})
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        b = state["batch"]
        b.run()
        return {"lam": b.lam_all, "V": b.V_all, "status": b.status}
    if kind == "serve":
        s = state["server"]
        code = {"arrow": ae.KIND_ARROW, "dpr1": ae.KIND_DPR1, "svd": ae.KIND_SVD}
        tickets = [s.submit(code[k], d, z, a) for k, d, z, a in state["reqs"]]
        res = []
        for t in tickets:
            s.wait(t)
            res.append(s.result(t))
            s.release(t)
        return res
    fn = {"arrow": ae.arrow_eig, "dpr1": ae.dpr1_eig, "svd": ae.tri_arrow_svd,
          "herm": ae.herm_arrow_eig, "nsym": ae.nsym_arrow_eig, "host": ae.arrow_eig_host}[kind]
    return fn(*state["in"], vectors=case["vectors"], opts=state["opts"], out=state["out"])


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _work_one(kind, n, vectors):
    """Inputs and outputs once; per eigenpair and row the element b (3 flops),
    one evaluation of the secular function (3) and one vector component (6; a
    second vector 2 more, a complex one 1 more)."""
    ins = {"herm": 3, "nsym": 3}.get(kind, 2)
    mats = {"herm": 2, "nsym": 2, "svd": 2}.get(kind, 1) if vectors else 0
    flops = 6 + (6 + 2 * (mats - 1) if vectors else 0)
    return 8.0 * (ins * n + n + mats * n * n), float(flops) * n * n


def work(case):
    if case["kind"] in ("batch", "serve"):
        ns = _sizes(case, np.random.default_rng(0))
        kinds = ("arrow", "dpr1", "svd") if case["kind"] == "serve" else ("arrow",)
        w = [_work_one(kinds[i % len(kinds)], int(n), case["vectors"]) for i, n in enumerate(ns)]
    else:
        w = [_work_one(case["kind"], case["n"], case["vectors"])]
    return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}


# ---------------------------------------------------------------------------
# the same results by plain torch in 64 bits
# ---------------------------------------------------------------------------
def _bits(x):
    return x.view(torch.int64)


def _zeros(diff, z2, corner, rho, hi_first, hi_last, count):
    """Offsets (pole index i, mu) of the `count` eigenvalues from their nearest
    poles, by bisection on the bits of |mu|.

    diff(j): column vector p - p_j for a row of pole indices j.  f falls through
    each eigenvalue: arrowhead (rho None) corner(j) - mu - sum z2 / (diff - mu),
    DPR1 -(1 + rho sum z2 / (diff - mu))."""
    m = z2.numel()
    poles, mus = [], []
    chunk = max(1, min(count, (1 << 27) // max(1, m)))
    for c0 in range(0, count, chunk):
        k = torch.arange(c0, min(count, c0 + chunk), device=DEV)

        def f(j, mu):
            s = (z2[:, None] / (diff(j) - mu[None, :])).sum(0)
            return corner(j) - mu - s if rho is None else -(1.0 + rho * s)

        first, last = k == 0, k == m
        lower = k.clamp(max=m - 1)                 # the pole below eigenvalue k
        upper = (k - 1).clamp(min=0)               # the pole above it
        gap = diff(lower)[upper, torch.arange(k.numel(), device=DEV)]
        half = 0.5 * gap
        inner = ~(first | last)
        fm = f(lower, torch.where(inner, half, torch.full_like(half, hi_first)))
        side = torch.where(first | (inner & (fm < 0)), 1.0, -1.0)
        j = torch.where(side > 0, lower, upper)
        top = torch.where(inner, half, torch.where(first, hi_first, hi_last))
        a = torch.zeros_like(_bits(top))
        b = _bits(top).clone()
        for _ in range(64):
            mid = a + torch.div(b - a, 2, rounding_mode="floor")
            mu = side * mid.view(torch.float64)
            up = f(j, mu) * side > 0               # the zero lies farther from the pole
            a, b = torch.where(up, mid, a), torch.where(up, b, mid)
        poles.append(j)
        mus.append(side * b.view(torch.float64))
    return torch.cat(poles), torch.cat(mus)


def _exact_one(kind, x, vectors):
    d, z, alpha = _up(x[0]), _up(x[1]), x[-1]
    m = d.numel()
    if kind == "dpr1":
        rho, z2 = alpha, z * z
        j, mu = _zeros(lambda i: d[:, None] - d[i][None, :], z2, None, rho,
                       float(rho * z2.sum()) * (1 + 1e-12), 0.0, m)
        lam = d[j] + mu
        if not vectors:
            return {"lam": lam}
        q = z[:, None] / ((d[:, None] - d[j][None, :]) - mu[None, :])
        return {"lam": lam, "Q": q / q.norm(dim=0, keepdim=True)}
    zr = _up(x[2]) if kind == "nsym" else z
    if kind == "svd":
        sp2, c = (d * z) ** 2, float(alpha * alpha + (z * z).sum())

        def diff(i):
            return (d[:, None] - d[i][None, :]) * (d[:, None] + d[i][None, :])

        p = d * d
    else:
        sp2, c, p = (z.abs() ** 2 if kind == "herm" else z * zr), alpha, d

        def diff(i):
            return d[:, None] - d[i][None, :]

    s = float(sp2.sum().sqrt())
    j, mu = _zeros(diff, sp2, lambda i: c - p[i], None,
                   max(c - float(p[0]), 0.0) + 2 * s + 1e-300,
                   max(float(p[-1]) - c, 0.0) + 2 * s + 1e-300, m + 1)
    lam = p[j] + mu
    if kind == "svd":
        lam = lam.sqrt()
    name = "s" if kind == "svd" else "lam"
    if not vectors:
        return {name: lam}
    t = 1.0 / (diff(j) - mu[None, :])
    inv = 1.0 / (1.0 + (sp2[:, None] * t * t).sum(0)).sqrt()
    last = -inv[None, :]
    spk = d * z if kind == "svd" else z
    V = torch.cat([spk[:, None] * t * inv[None, :], last.to(spk.dtype)])
    if kind == "svd":
        U = torch.cat([lam[None, :] * V[:-1] / d[:, None], alpha * last / lam[None, :]])
        return {"s": lam, "U": U, "V": V}
    if kind == "herm":
        return {"lam": lam, "U": V}
    if kind == "nsym":
        return {"lam": lam, "X": V, "Y": torch.cat([zr[:, None] * t * inv[None, :], last])}
    return {"lam": lam, "V": V}


def _dense_values(x):
    d, z, alpha = _up(x[0]), _up(x[1]), x[2]
    A = torch.diag(torch.cat([d, torch.tensor([alpha], dtype=torch.float64, device=DEV)]))
    A[-1, :-1] = z
    A[:-1, -1] = z
    return torch.linalg.eigvalsh(A).flip(0)


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        out = []
        for k, d, z, a in _many(case, seed):
            e = _exact_one(k, (d, z, a), True)
            out.append({"lam": e["s" if k == "svd" else "lam"],
                        "V": e["Q" if k == "dpr1" else "V"]} | ({"U": e["U"]} if k == "svd" else {}))
        return out
    if kind == "batch":
        lam, V = [], []
        for _, d, z, a in _many(case, seed):
            e = _exact_one("arrow", (d, z, a), True)
            lam.append(e["lam"])
            V.append(e["V"].t().reshape(-1))
        return {"lam": torch.cat(lam), "V": torch.cat(V), "status": None}
    x = _one(case, seed)
    if case["spectrum"] == "messy":
        res = {"lam": _dense_values(x)}
        return res | ({"V": None} if case["vectors"] else {})
    res = _exact_one("arrow" if kind == "host" else kind, x, case["vectors"])
    return {k: v.cpu() for k, v in res.items()} if kind == "host" else res
