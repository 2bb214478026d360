"""The polynomial coefficients of csrc/fx64.cuh, recomputed: each polynomial
interpolates its function at the Chebyshev nodes of the reduced range (as many
as it has coefficients), in 400-bit arithmetic, truncated to the word."""
import os
import re

import pytest

mp = pytest.importorskip("mpmath")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = open(os.path.join(ROOT, "paper_2410_01136_gb300", "csrc", "fx64.cuh")).read()


def coefficients(start, end, var):
    i = SOURCE.index(start)
    text = SOURCE[i:SOURCE.index(end, i)]
    return [int(x, 16) for x in re.findall(r"\b%s = (0x[0-9A-F]+)ull" % var, text)][::-1]


ROOT2 = "((mp.sqrt(2) - 1) / (mp.sqrt(2) + 1)) ** 2"          # s^2 at m = sqrt 2


# name, where the words stand, the function of f or of u = s^2, w^2, the end of
# its range, fraction bits, alternating signs (kept as subtractions)
@pytest.mark.parametrize("where,fn,hi,bits,alternating", [
    (("u64 exp2m1_core", "return mh(p, f)", "p"), "(mp.power(2, u) - 1) / u", "1", 64, False),
    (("u64 log2_core", "return mh(sn", "p"), "2 / mp.log(2) * mp.atanh(mp.sqrt(u)) / mp.sqrt(u)", ROOT2, 62, False),
    (("void sincos_any", "u64 pc", "ps"), "mp.sin(mp.pi / 4 * mp.sqrt(u)) / mp.sqrt(u)", "1", 64, True),
    (("u64 pc", "an unreduced", "pc"), "(1 - mp.cos(mp.pi / 4 * mp.sqrt(u))) / u", "1", 64, True),
    (("SYNAX_FX_FN double atan2", "u64 t = mh(w", "p"), "mp.atan(mp.sqrt(u)) / mp.sqrt(u)", "1", 63, True)],
    ids=["exp2", "log2", "sin", "cos", "atan"])
def test_coefficients(where, fn, hi, bits, alternating):
    have = coefficients(*where)
    n = len(have)
    with mp.workprec(400):
        f = eval("lambda u: " + fn, {"mp": mp})
        top = mp.mpf(eval(hi, {"mp": mp}))
        nodes = [top / 2 * (1 + mp.cos(mp.pi * (2 * i + 1) / (2 * n))) for i in range(n)]
        p = mp.lu_solve(mp.matrix([[x ** j for j in range(n)] for x in nodes]), mp.matrix([f(x) for x in nodes]))
        words = [int(mp.floor((-v if alternating and j % 2 else v) * mp.mpf(2) ** bits)) for j, v in enumerate(p)]
    assert [hex(w) for w in have] == [hex(w) for w in words]
