"""The fixed-point passes (csrc/ae_fixed.cuh, csrc/ae_fast.cuh).

CPU: the reciprocal, the modular tail and the high product, compiled for the
host, against exact integers; the bounds are those the header derives (2^-56
for the quadratic reciprocal, 2^-58.5 for the cubic one, 2^-60 for the columns'
one, 2 units for the product), seeds off by an ulp included.
GPU: eigenpairs at the passes' edges -- tile and chunk boundaries, outermost
eigenvalues far from all poles, poles in tight clusters, a DPR1 whose last pole
lies far out, spectra that need the 128-bit evaluations, inputs whose exponents
the passes refuse, an iteration cap that sends a solve to the FP64 kernels, far poles taken
as moments and their rows' components (768 poles and more, groups of 32) --
against the oracle at the suite's bar, 10 n eps64.
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
#include <random>
using namespace ae;
typedef unsigned __int128 u128;
typedef __int128 i128;
static double dbl(uint32_t h, uint32_t l) {
    uint64_t u = ((uint64_t)h << 32) | l;
    double d;
    memcpy(&d, &u, 8);
    return d;
}
static i128 fix128(double x) {          // floor(x 2^106)
    int e;
    const i128 m = (i128)std::ldexp(std::frexp(x, &e), 53);
    const int sh = e - 53 + 106;
    return sh >= 0 ? m << sh : sh < -120 ? (m < 0 ? -1 : 0) : m >> -sh;
}
int main() {
    std::mt19937_64 g(7);
    std::uniform_real_distribution<> U(-0.5, 0.5);
    double w2 = 0, w3 = 0, w6 = 0;
    int prod = 0, n = 0;
    for (int it = 0; it < 2000000; ++it) {
        const double sc = std::ldexp(1.0, -(int)(g() % 40));
        const double p = U(g) * (it % 3 ? 1 : sc);
        double lh = U(g) * sc;
        if (it % 5 == 0) lh = p * (1 + std::ldexp((double)(g() % 1000) - 500, -14 - (int)(g() % 12)));
        const double ll = 0.999 * U(g) * std::ldexp(std::fabs(lh), -53);
        const double D = p - lh;
        const uint64_t b = f64_bits(D);
        const uint32_t dh = (uint32_t)(b >> 32), dl = (uint32_t)b, eb = (dh << 1) >> 21;
        const uint32_t el = (uint32_t)((f64_bits(lh) << 1) >> 53);
        if (eb < kFixMinExp || eb + kTailSpan < el) continue;
        ++n;
        const uint64_t L = fix_mod(lh) + fix_mod(ll);
        const int tl = tail_of(fix_mod(p) - L, dh, dl, eb);
        // the exact difference in units of 2^-106
        i128 x = fix128(p) - fix128(lh) - fix128(ll);
        if (x < 0) x = -x;
        const uint32_t hm = (dh & 0xfffffu) | 0x3ff00000u;
        const double r = (1.0 / dbl(hm, 0)) * (1 + ((int)(g() % 3) - 1) * std::ldexp(1.0, -21));
        const uint32_t seed = (uint32_t)(f64_bits(r) >> 32);
        const uint64_t R2 = recip63<false>(dh, dl, tl, seed), R3 = recip63<true>(dh, dl, tl, seed);
        // relative error = R m / 2^63 - 1, m = x 2^-106 / 2^(eb - 1023), in long double
        const int sh = (int)eb - 1023 + 106;
        for (int c = 0; c < 2; ++c) {
            const uint64_t R = c ? R3 : R2;
            // (x R) / 2^(sh + 63) - 1 exactly: x < 2^107, R <= 2^63
            const u128 lo = (u128)(uint64_t)x * R, hi = (u128)(uint64_t)(x >> 64) * R;
            const i128 top = (i128)(hi + (lo >> 64)) - ((i128)1 << (sh - 1));
            const double e = std::fabs((double)top / std::ldexp(1.0, sh - 1));
            if (c) w3 = std::fmax(w3, e); else w2 = std::fmax(w2, e);
        }
        const uint64_t z = g() | (1ull << 63);
        const uint64_t ex = (uint64_t)(((u128)z * R3) >> 64);
        const int64_t df = (int64_t)(ex - mul_hi3(z, R3));
        if (df < 0 || df > 2) ++prod;
        // recip62 from an FP32 reciprocal an ulp off
        const uint64_t mm = (uint64_t)((0.872 + 1.384 * (double)(g() >> 11) * 0x1p-53) * 0x1p62);
        float r1 = 1.0f / (float)(uint32_t)(mm >> 32);
        uint32_t rb;
        memcpy(&rb, &r1, 4);
        rb += (int)(g() % 3) - 1;
        memcpy(&r1, &rb, 4);
        const uint32_t R0 = (uint32_t)std::lrint((double)r1 * 0x1p52);
        const i128 pr = (i128)((u128)mm * recip62(mm, R0)) - ((i128)1 << 124);
        w6 = std::fmax(w6, std::fabs((double)pr / 0x1p124));
    }
    std::printf("%d %.3f %.3f %d %.3f\n", n, std::log2(w2), std::log2(w3), prod, std::log2(w6));
    return 0;
}
"""


def test_fixed_point_arithmetic_on_the_host(tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    src = tmp_path / "h.cpp"
    src.write_text(HARNESS)
    exe = tmp_path / "h"
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I",
                           os.path.join(root, "paper_1302_7203_gb300", "csrc"), str(src), "-o",
                           str(exe)])
    n, w2, w3, prod, w6 = subprocess.check_output([str(exe)]).split()
    assert int(n) > 500000
    assert float(w2) <= -55.5 and float(w3) <= -58.5 and int(prod) == 0
    assert float(w6) <= -60.0


FORMS = {"plain": {}, "fast": dict(precision=1, finish=1, bgate=1)}


def data(case):
    rng = np.random.default_rng(5)
    if case[1:].isdigit():
        return W.uniform_arrow(int(case[1:]), seed=int(case[1:]))
    if case == "far_corner":             # outermost eigenvalues beyond all poles
        d, z, _ = W.graded_arrow(300, seed=3)
        return d, z, -1e6
    if case == "long_spikes":
        d, z, a = W.uniform_arrow(300, seed=4)
        return d, z * 1e3, a
    if case == "clusters":               # relative gaps down to 1e-10
        c = rng.uniform(-5, 5, 12)
        d = np.unique((c[:, None] * (1 + 1e-10 * np.arange(1, 26))).ravel())[::-1].copy()
        return d, 1.0 - rng.random(d.size), 0.5
    if case == "zero_pole":
        d, z, a = W.uniform_arrow(129, seed=9)
        d[64] = 0.0
        return np.sort(d)[::-1].copy(), z, a
    if case == "near_zero":              # many eigenvalues next to zero
        d, z, a = W.graded_arrow(500, seed=8)
        return d * 1e-3, z, 0.0
    if case == "tiny_spikes":            # mu far below the pole's last place
        d, z, a = W.uniform_arrow(400, seed=6)
        return d, z * 10.0 ** rng.uniform(-14, 0, z.size), a
    if case == "cancelling":             # b's sum cancels: the 128-bit evaluations
        d = np.linspace(1.0, -1.0, 400) + rng.uniform(-1e-4, 1e-4, 400)
        z = 10.0 ** rng.uniform(-6, 0, 400)
        return np.sort(d)[::-1].copy(), z, 0.0
    d, z, a = W.uniform_arrow(200, seed=2)
    s = 2.0 ** (500 if case == "huge" else -500)   # squares stay finite, scaling refused
    return d * s, z * s, a * s


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
@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("case", ["n3", "n32", "n33", "n34", "n256", "n257", "n258", "n514", "n700",
                                  "far_corner", "long_spikes", "clusters", "zero_pole",
                                  "near_zero", "tiny_spikes", "cancelling", "huge", "small"])
def test_edges_of_the_passes(ae, case, form):
    d, z, a = data(case)
    r = ae.arrow_eig(t(d), t(z), a, opts=ae.default_opts(**FORMS[form]), info=True)
    o = oracle.arrow_eig(d, z, a)
    assert_parity(r["lam"].cpu().numpy(), r["V"].cpu().numpy(), o, len(d) + 1,
                  what=f"{case} {form}")
    # the diagnostics change nothing
    q = ae.arrow_eig(t(d), t(z), a, opts=ae.default_opts(**FORMS[form]), diag=True)
    assert np.array_equal(q["lam"].cpu().numpy(), r["lam"].cpu().numpy())
    assert np.array_equal(q["V"].cpu().numpy(), r["V"].cpu().numpy())


@pytest.mark.gpu
def test_iteration_cap_takes_the_fp64_solver(ae):
    d, z, a = W.uniform_arrow(150, seed=1)
    o = oracle.arrow_eig(d, z, a)
    r = ae.arrow_eig(t(d), t(z), a, opts=ae.default_opts(finish=1, max_iter=99), info=True)
    assert_parity(r["lam"].cpu().numpy(), r["V"].cpu().numpy(), o, 151, what="max_iter 99")
    with pytest.raises(ae.AeError) as ei:
        ae.arrow_eig(t(d), t(z), a, opts=ae.default_opts(max_iter=5), info=True)
    assert ei.value.status == ae.AE_ERR_NOCONV


@pytest.mark.gpu
@pytest.mark.parametrize("rho", [0.5, -0.5])
def test_dpr1_with_a_far_last_pole(ae, rho):
    d, u, _ = W.uniform_dpr1(300, seed=12)
    d = d.copy()
    d[-1 if rho > 0 else 0] = -1e3 if rho > 0 else 1e3
    ref = oracle.dpr1_eig(d, u, rho)
    for kw in FORMS.values():
        r = ae.dpr1_eig(t(d), t(u), rho, opts=ae.default_opts(**kw))
        assert_parity(r["lam"].cpu().numpy(), r["Q"].cpu().numpy(),
                      {"lam": ref["lam"], "abserr": np.zeros(300), "V": ref["Q"]}, 300,
                      what="dpr1, far last pole")


@pytest.mark.gpu
@pytest.mark.parametrize("n", [3, 33, 257])
def test_svd_edges(ae, n):
    d, z, a = W.uniform_tsvd(n, seed=n)
    ref = oracle.tsvd(d, z, a)
    r = ae.tri_arrow_svd(t(d), t(z), a, opts=ae.default_opts(**FORMS["fast"]))
    for key in ("V", "U"):
        assert_parity(r["s"].cpu().numpy(), r[key].cpu().numpy(),
                      {"lam": ref["s"], "abserr": np.zeros(n), "V": ref[key]}, n,
                      what=f"svd {n} {key}")


@pytest.mark.gpu
@pytest.mark.parametrize("m", [200, 800])
def test_svd_columns_of_close_squares(ae, m):
    # squares down to 1e-80: differences below the rows' fixed-point unit
    d, z = 10.0 ** -np.linspace(0, 40, m), np.random.default_rng(m).standard_normal(m)
    ref = oracle.tsvd(d, z, 0.5)
    r = ae.tri_arrow_svd(t(d), t(z), 0.5)
    for key in ("V", "U"):
        assert_parity(r["s"].cpu().numpy(), r[key].cpu().numpy(),
                      {"lam": ref["s"], "abserr": np.zeros(m + 1), "V": ref[key]}, m + 1,
                      what=f"svd, close squares, {m} {key}")


def far_case(case):
    rng = np.random.default_rng(6)
    if case[1:].isdigit():
        return W.uniform_arrow(int(case[1:]), seed=int(case[1:]))
    if case == "graded":
        return W.graded_arrow(900, seed=31)
    if case == "gap":                    # a group straddles a gap: no pole is far from it
        d = np.concatenate([rng.uniform(4, 5, 432), rng.uniform(-3, -2, 433)])
    elif case == "clusters":             # one group's poles agree to 1e-10
        c = np.linspace(-5, 5, 30) + rng.uniform(-0.1, 0.1, 30)
        d = (c[:, None] * (1 + 1e-10 * np.arange(1, 33))).ravel()
    else:                                # "zero": eigenvalues next to 0 and large spikes
        d = np.concatenate([rng.uniform(-5, 5, 800), 10.0 ** rng.uniform(-9, -1, 100)])
    d = np.sort(d)[::-1].copy()
    z = 1.0 - rng.random(d.size)
    return d, z * (100.0 if case == "zero" else 1.0), 0.5


@pytest.mark.gpu
@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("case", ["n768", "n769", "n770", "n800", "n801", "n802", "n1025",
                                  "graded", "gap", "clusters", "zero"])
def test_far_poles_as_moments(ae, case, form):
    d, z, a = far_case(case)
    r = ae.arrow_eig(t(d), t(z), a, opts=ae.default_opts(**FORMS[form]), info=True)
    assert_parity(r["lam"].cpu().numpy(), r["V"].cpu().numpy(), oracle.arrow_eig(d, z, a),
                  len(d) + 1, what=f"far poles {case} {form}")


@pytest.mark.gpu
def test_far_poles_dpr1_and_svd(ae):
    d, u, rho = W.uniform_dpr1(900, seed=5)
    ref = oracle.dpr1_eig(d, u, rho)
    r = ae.dpr1_eig(t(d), t(u), rho)
    assert_parity(r["lam"].cpu().numpy(), r["Q"].cpu().numpy(),
                  {"lam": ref["lam"], "abserr": np.zeros(900), "V": ref["Q"]}, 900, what="dpr1")
    d, z, a = W.uniform_tsvd(900, seed=5)
    ref = oracle.tsvd(d, z, a)
    r = ae.tri_arrow_svd(t(d), t(z), a)
    for key in ("V", "U"):
        assert_parity(r["s"].cpu().numpy(), r[key].cpu().numpy(),
                      {"lam": ref["s"], "abserr": np.zeros(900), "V": ref[key]}, 900,
                      what=f"svd {key}")


@pytest.mark.gpu
@pytest.mark.parametrize("order", ["sorted", "permuted"])
def test_columns_of_far_rows(ae, order):
    # zero and tiny spikes among the far rows (components of 0 and down to 1e-140),
    # a last segment of few rows; permuted: no 32 rows are far together
    rng = np.random.default_rng(8)
    d, z, a = W.uniform_arrow(933, seed=8)
    z = z.copy()
    z[[3, 40, 500, 931]] = 0.0
    z[100:140] *= 1e-130
    p = rng.permutation(d.size) if order == "permuted" else np.arange(d.size)
    r = ae.arrow_eig(t(d[p]), t(z[p]), a)
    assert_parity(r["lam"].cpu().numpy(), r["V"].cpu().numpy(), oracle.arrow_eig(d[p], z[p], a),
                  933, what=f"far rows {order}")
    zr = z * (0.5 + rng.random(d.size))
    r = ae.nsym_arrow_eig(t(d[p]), t(z[p]), t(zr[p]), a)
    ref = oracle.nsym_eig(d[p], z[p], zr[p], a)
    for key in ("X", "Y"):
        assert_parity(r["lam"].cpu().numpy(), r[key].cpu().numpy(), {**ref, "V": ref[key]}, 933,
                      what=f"far rows, {key} {order}")
