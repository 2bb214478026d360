"""The functions of csrc/fx64.cuh beside their zeros, where the results keep
their relative accuracy as CUDA's functions do: ln and log2 beside 1, atan2 of
a small angle, sine and cosine beside non-zero multiples of pi/2.  Reference:
400-bit arithmetic.  Tolerance 0.53 ulp: 0.5 of the final rounding and 2^-58
relative for the 62-bit evaluation (a few units of 2^-61: seed and Newton step,
quotient, polynomial, product)."""
import numpy as np
import pytest

mp = pytest.importorskip("mpmath")

from .test_fx64_cpu import fx  # noqa: E402,F401  (the compiled header)

mp.mp.prec = 400


def ulps(got, want):
    """|got - want| in units of the last place of want (mpmath reals)."""
    out = []
    for g, w in zip(got, want):
        w64 = float(w)
        out.append(float(abs(mp.mpf(float(g)) - w) / mp.mpf(float(np.spacing(abs(w64)))) if w else abs(g) * 1e300))
    return np.array(out)


@pytest.mark.parametrize("op,fn", [(2, mp.log), (3, lambda v: mp.log(v, 2))])
def test_logarithms_beside_one(fx, op, fn):
    g = np.random.default_rng(op)
    d = np.concatenate([10.0 ** g.uniform(-15.9, -1, 1500), 2.0 ** -np.arange(2.0, 53.0)])
    x = np.concatenate([1 + d, 1 - d / 2])
    x = x[x != 1]
    assert np.max(ulps(fx(op, x)[0], [fn(mp.mpf(float(v))) for v in x])) <= 0.53


def test_small_angles_of_atan2(fx):
    g = np.random.default_rng(10)
    n = 3000
    y = g.normal(size=n) * 10.0 ** -g.uniform(0, 250, n)
    x = np.abs(g.normal(size=n)) * 10.0 ** g.uniform(-40, 40, n)
    y[-60:], x[-60:] = 2.0 ** -np.arange(60.0), 1.0 + 2.0 ** -np.arange(1.0, 61.0)
    want = [mp.atan2(mp.mpf(float(a)), mp.mpf(float(b))) for a, b in zip(y, x)]
    assert np.max(ulps(fx(10, y, x)[0], want)) <= 0.53


# the doubles next to k pi/2 are the angles whose reduction cancels most bits;
# 29 2^j are the worst of them
@pytest.mark.parametrize("op", [8, 9])
def test_sine_and_cosine_beside_multiples_of_a_quarter_turn(fx, op):
    g = np.random.default_rng(op)
    quarter = mp.pi / 2 if op == 8 else mp.mpf(1) / 4
    k = np.concatenate([np.arange(1, 200), g.integers(200, 40000, 400), 29 * 2 ** np.arange(9)])
    base = np.array([float(quarter * int(v)) for v in k])
    near = base * (1 + g.choice([-1, 1], base.size) * 10.0 ** -g.uniform(3, 16, base.size))
    x = np.concatenate([base, np.nextafter(base, 0), np.nextafter(base, np.inf), near])
    x = np.concatenate([x, -x])
    s, c = fx(op, x)
    unit = 1 if op == 8 else 2 * mp.pi
    X = [mp.mpf(float(v)) * unit for v in x]
    if op == 9:                                   # exact quarter turns: exact zeros and ones
        r = np.round(4 * x) == 4 * x
        assert np.all((s[r] == 0) | (np.abs(s[r]) == 1)) and np.all(np.abs(s[r]) + np.abs(c[r]) == 1)
        x, s, c, X = x[~r], s[~r], c[~r], [v for v, z in zip(X, r) if not z]
    assert np.max(ulps(s, [mp.sin(v) for v in X])) <= 0.53
    assert np.max(ulps(c, [mp.cos(v) for v in X])) <= 0.53
