"""csrc/fx64.cuh as the device computes it, with the hardware's reciprocal and
inverse-square-root seeds, against the host build of the same header (which the
CPU tests hold to 0.53 ulp): the integer arithmetic is the same, so only the
seeds differ, and a result may differ by the last place of FP64 where the exact
value lies near the middle of two."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from .test_fx64_cpu import HARNESS, ROOT, draw

pytestmark = pytest.mark.gpu

EXTRA = """
        case 13: r[i] = fx::log_any<true, false>(a[i]); r2[i] = fx::log_any<false, false>(a[i]); break;
        case 14: r[i] = fx::atan2<false>(a[i], b[i]); break;
        case 15: fx::sincos_any<false, false>(a[i], r + i, r2 + i); break;
        case 16: fx::sincos_any<true, false>(a[i], r + i, r2 + i); break;
"""
# the inputs of each operation: those of the CPU tests
INPUTS = list(range(13)) + [2, 10, 8, 9]


@pytest.fixture(scope="module")
def both(tmp_path_factory):
    from paper_2410_01136_gb300.cuda_build import ARCH, nvcc
    d = tmp_path_factory.mktemp("fx64d")
    inc = os.path.join(ROOT, "paper_2410_01136_gb300", "csrc")
    ops = HARNESS[HARNESS.index("        case 0:"):HARNESS.index("        }\n    }\n}")] + EXTRA
    (d / "h.cpp").write_text(HARNESS.replace("        case 12:", EXTRA + "        case 12:"))
    (d / "d.cu").write_text("""
#include "fx64.cuh"
using namespace synax;
__global__ void k_eval(int op, int n, const double* a, const double* b, double* r, double* r2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    switch (op) {
""" + ops + """
    }
}
extern "C" int fx_eval(int op, int n, const double* a, const double* b, double* r, double* r2) {
    k_eval<<<(n + 127) / 128, 128>>>(op, n, a, b, r, r2);
    const int e = (int)cudaGetLastError();
    return e ? e : (int)cudaDeviceSynchronize();
}
""")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", "-I", inc, str(d / "h.cpp"),
                    "-o", str(d / "h.so")], check=True)
    subprocess.run([nvcc(), "-shared", "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-I", inc, str(d / "d.cu"), "-o",
                    str(d / "d.so")] + ARCH, check=True)
    return ctypes.CDLL(str(d / "h.so")), ctypes.CDLL(str(d / "d.so"))


@pytest.mark.parametrize("op", range(17))
def test_device_against_host(both, op):
    import torch
    host, dev = both
    a, b = draw(INPUTS[op])
    if op == 8:
        a = a[np.abs(a) < 2.0 ** 14]          # beyond, CUDA's function and the host's answer
    a = np.ascontiguousarray(a, dtype=np.float64)
    b = np.zeros_like(a) if b is None else np.ascontiguousarray(b, dtype=np.float64)
    want = [np.zeros_like(a), np.zeros_like(a)]
    host.fx_eval(op, a.size, *[ctypes.c_void_p(v.ctypes.data) for v in (a, b, *want)])
    t = [torch.tensor(v, device="cuda") for v in (a, b, np.zeros_like(a), np.zeros_like(a))]
    assert dev.fx_eval(op, a.size, *[ctypes.c_void_p(v.data_ptr()) for v in t]) == 0
    for w, g in zip(want, t[2:]):
        g = g.cpu().numpy()
        assert np.array_equal(np.isfinite(g), np.isfinite(w))
        f = np.isfinite(w)
        # absolute 2^-60 where the short forms and tanh have it beside their zeros
        tol = np.spacing(np.abs(w[f])) + (2.0 ** -60 if op in (11, 13, 14, 15, 16) else 0.0)
        assert np.all(np.abs(g[f] - w[f]) <= tol)
        assert np.array_equal(g[~f], w[~f], equal_nan=True)
        # a seed moves the value by 2^-61 of itself at most, across a rounding boundary for 1 in 2^7
        assert np.mean(g[f] == w[f]) >= 0.98
