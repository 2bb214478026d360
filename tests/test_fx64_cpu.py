"""The fixed-point FP64 functions of csrc/fx64.cuh, compiled as plain C++,
against extended precision, over their ordinary ranges and at the edges of
their reductions.  Tolerances: 0.51 ulp of the result (0.5 of the final
rounding plus 2^-60 relative for the 62-bit evaluation and the reference), and for the functions that pass through zero an
absolute 2^-60 beside it."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LD = np.longdouble

HARNESS = """
#include "fx64.cuh"
using namespace synax;
extern "C" void fx_eval(int op, int n, const double* a, const double* b, double* r, double* r2) {
    for (int i = 0; i < n; ++i) {
        switch (op) {
        case 0: r[i] = fx::exp_any<true>(a[i]); break;
        case 1: r[i] = fx::exp_any<false>(a[i]); break;
        case 2: r[i] = fx::log_any<true>(a[i]); break;
        case 3: r[i] = fx::log_any<false>(a[i]); break;
        case 4: r[i] = fx::sqrt(a[i]); break;
        case 5: r[i] = fx::rsqrt(a[i]); break;
        case 6: r[i] = fx::rcp(a[i]); break;
        case 7: r[i] = fx::div(a[i], b[i]); break;
        case 8: fx::sincos_any<false>(a[i], r + i, r2 + i); break;
        case 9: fx::sincos_any<true>(a[i], r + i, r2 + i); break;
        case 10: r[i] = fx::atan2(a[i], b[i]); break;
        case 11: fx::sech2_tanh(a[i], r[i], r2[i]); break;
        case 12: r[i] = fx::exp_radial<false>(a[i]); r2[i] = fx::exp_radial<true>(a[i]); break;
        }
    }
}
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx64")
    src, so = d / "h.cpp", d / "h.so"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_2410_01136_gb300", "csrc"), str(src), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))

    def call(op, a, b=None):
        a = np.ascontiguousarray(a, dtype=np.float64)
        b = np.zeros_like(a) if b is None else np.ascontiguousarray(b, dtype=np.float64)
        r, r2 = np.empty_like(a), np.empty_like(a)
        p = [v.ctypes.data_as(ctypes.c_void_p) for v in (a, b, r, r2)]
        lib.fx_eval(op, a.size, *p)
        return r, r2

    return call


def edges(v):
    v = np.asarray(v, dtype=np.float64)
    return np.concatenate([v, np.nextafter(v, np.inf), np.nextafter(v, -np.inf)])


def draw(op):
    g = np.random.default_rng(op)
    n = 40000
    if op in (0, 1):
        near = edges(np.arange(-60, 61) * (np.log(2) / 2 if op == 0 else 0.5))
        return np.concatenate([g.uniform(-40, 40, n), g.uniform(-690, 690, n), near,
                               10.0 ** g.uniform(-300, 0, n) * g.choice([-1, 1], n)]), None
    if op in (2, 3, 4, 5, 6):
        pos = np.concatenate([2.0 ** g.uniform(-100, 100, n), g.uniform(0.9, 1.1, n), g.uniform(0, 30, n) + 1e-9,
                              edges([1, 2, 4, 0.5, np.sqrt(2), np.sqrt(0.5)])])
        return (pos * np.where(g.random(pos.size) < 0.5, -1, 1) if op == 6 else pos), None
    if op == 7:
        return g.normal(size=n) * 10.0 ** g.uniform(-50, 50, n), g.normal(size=n) * 10.0 ** g.uniform(-50, 50, n)
    if op == 8:
        return np.concatenate([g.uniform(-7, 7, n), g.uniform(-500, 500, n), g.uniform(-1e6, 1e6, n), edges(np.arange(-40, 41) * (np.pi / 4)),
                               10.0 ** g.uniform(-290, 0, n) * g.choice([-1, 1], n), [0.0, -0.0]]), None
    if op == 9:
        return np.concatenate([g.uniform(-0.5, 0.5, n), g.uniform(-200, 200, n), g.uniform(-1e12, 1e12, n), edges(np.arange(-40, 41) / 8),
                               10.0 ** g.uniform(-290, 0, n) * g.choice([-1, 1], n), [0.0, -0.0]]), None
    if op in (11, 12):
        return np.concatenate([g.uniform(0, 2, n), g.uniform(0, 60, n), g.uniform(0, 250, n),
                               10.0 ** g.uniform(-300, 0, n), [0.0, 255.0]]), None
    s = 10.0 ** g.uniform(-3, 3, n)
    y, x = g.normal(size=n) * s, g.normal(size=n) * s
    ax = np.array([[1, 1], [1, -1], [-1, 1], [-1, -1], [0, 1], [0, -1], [-0.0, -1], [1, 0], [-1, 0], [1e-30, 1],
                   [1, 1e-30], [1e-30, -1], [1, np.nextafter(1, 2)], [np.nextafter(1, 2), 1]])
    return np.concatenate([y, ax[:, 0]]), np.concatenate([x, ax[:, 1]])


def check(got, want, absolute):
    tol = LD(0.51) * np.spacing(np.abs(want.astype(np.float64))).astype(LD) + LD(absolute)
    bad = np.abs(got.astype(LD) - want) > tol
    assert not bad.any(), (int(bad.sum()), float(np.max(np.abs(got.astype(LD) - want) / tol)))


@pytest.mark.parametrize("op", range(13))
def test_against_extended_precision(fx, op):
    a, b = draw(op)
    r, r2 = fx(op, a, b)
    A = a.astype(LD)
    if op == 8:
        check(r, np.sin(A), 2.0 ** -60)
        check(r2, np.cos(A), 2.0 ** -60)
        small = np.abs(a) < 0.5                      # small angles keep their relative accuracy
        check(r[small], np.sin(A[small]), 0.0)
    elif op == 9:
        f = (A - np.rint(A)) * LD("6.283185307179586476925286766559005768")
        check(r, np.sin(f), 2.0 ** -60)
        check(r2, np.cos(f), 2.0 ** -60)
    elif op == 10:
        check(r, np.arctan2(A, b.astype(LD)), 2.0 ** -60)
    elif op == 11:
        check(r, 1 / np.cosh(A) ** 2, 0.0)
        check(r2, np.tanh(A), 2.0 ** -60)
    elif op == 12:
        for got, k in ((r, 20), (r2, 5)):
            q = A / k                                # the quotient's rounding, up to 12 2^-63 of the result, put back
            check(got, np.exp(-q) * (1 - ((A - 4 * (k // 5) * q) - (k // 5) * q) / k), 0.0)
    else:
        want = {0: np.exp, 1: np.exp2, 2: np.log, 3: np.log2, 4: np.sqrt, 5: lambda v: 1 / np.sqrt(v),
                6: lambda v: 1 / v, 7: lambda v: v / b.astype(LD)}[op](A)
        check(r, want, 2.0 ** -60 if op in (2, 3) else 0.0)


def test_special_values(fx):
    inf, nan = np.inf, np.nan
    assert list(fx(0, [0.0, -inf, inf, -1000.0, 1000.0])[0]) == [1.0, 0.0, inf, 0.0, inf]
    assert list(fx(2, [1.0, 0.0, inf])[0]) == [0.0, -inf, inf]
    assert list(fx(4, [0.0, 4.0, inf, 1e-320])[0]) == [0.0, 2.0, inf, np.sqrt(1e-320)]
    assert list(fx(6, [1.0, -2.0, inf, 1e-320])[0]) == [1.0, -0.5, 0.0, inf]
    assert list(fx(7, [0.0, 1.0, 6.0], [3.0, 0.0, 3.0])[0]) == [0.0, inf, 2.0]
    assert list(fx(9, [0.0, 0.25, 0.5])[0]) == [0.0, 1.0, 0.0]
    for op in range(9):
        assert np.isnan(fx(op, [nan], [1.0])[0][0])
    assert np.isnan(fx(2, [-1.0])[0][0]) and np.isnan(fx(4, [-1.0])[0][0]) and np.isnan(fx(8, [inf])[0][0])
