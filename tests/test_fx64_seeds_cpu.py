"""Reciprocals and inverse square roots of csrc/fx64.cuh with the worst seeds
that the device may give: rcp.approx and rsqrt.approx are specified to an error
of 1 and 2 units of the FP32 result, where the host build's seeds are correctly
rounded.  With seeds of up to 2 units either way the results keep 0.51 ulp."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from .test_fx64_cpu import HARNESS, LD, ROOT, check, draw, edges


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    """The header with `seed_ulp` added to the bits of both seeds."""
    d = tmp_path_factory.mktemp("fx64s")
    text = open(os.path.join(ROOT, "paper_2410_01136_gb300", "csrc", "fx64.cuh")).read()
    host = text.index("#else", text.index("rsqrt.approx"))
    tail = text[host:].replace("    std::memcpy(&b, &y, 4);\n    return b;", "    std::memcpy(&b, &y, 4);\n    return b + seed_ulp;", 2)
    assert tail.count("b + seed_ulp") == 2
    (d / "fx64.cuh").write_text(text[:host] + tail)
    (d / "h.cpp").write_text("static int seed_ulp = 0;\n" + HARNESS +
                             '\nextern "C" void set_seed_ulp(int k) { seed_ulp = k; }\n')
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", "-I", str(d),
                    str(d / "h.cpp"), "-o", str(d / "h.so")], check=True)
    lib = ctypes.CDLL(str(d / "h.so"))

    def call(ulp, op, a, b=None):
        a = np.ascontiguousarray(a, dtype=np.float64)
        b = np.zeros_like(a) if b is None else np.ascontiguousarray(b, dtype=np.float64)
        r, r2 = np.empty_like(a), np.empty_like(a)
        lib.set_seed_ulp(ulp)
        lib.fx_eval(op, a.size, *[v.ctypes.data_as(ctypes.c_void_p) for v in (a, b, r, r2)])
        return r

    return call


@pytest.mark.parametrize("ulp", [-2, -1, 1, 2])
@pytest.mark.parametrize("op", [4, 5, 6, 7])
def test_worst_seeds(fx, op, ulp):
    a, b = draw(op)
    # mantissas beside the ends of the seeds' ranges, where a seed may leave [1/2, 1)
    ends = np.concatenate([2.0 - np.arange(1, 200) * 2.0 ** -24, 4.0 - np.arange(1, 200) * 2.0 ** -23,
                           1.0 + np.arange(200) * 2.0 ** -24, edges([1.0, 2.0, 4.0])])
    a = np.concatenate([a, ends])
    if op == 7:
        b = np.concatenate([b, ends[::-1]])
    A = a.astype(LD)
    want = {4: lambda: np.sqrt(A), 5: lambda: 1 / np.sqrt(A), 6: lambda: 1 / A, 7: lambda: A / b.astype(LD)}[op]()
    check(fx(ulp, op, a, b), want, 0.0)
