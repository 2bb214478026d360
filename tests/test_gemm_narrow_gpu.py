"""Narrow GEMM tiles (32 columns, chosen when few rows leave SMs idle).

The operands are small integers, so every product and partial sum is exact in
FP32 (|sum| <= K * 9 < 2^24) and the results must equal the integer matrix
product whatever the tile width; with random operands the same rows computed
inside a taller product (wider tiles, same order along K) must be bitwise equal.
"""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


def _gemm(a, b):
    import torch
    from paper_2410_01136_gb300._native import check, lib
    m, k = a.shape
    n = b.shape[0]
    c = torch.full((m, n), float("nan"), device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    vp = ctypes.c_void_p
    check(lib().synax_gemm_bf16(vp(a.data_ptr()), k, vp(b.data_ptr()), k, m, n, k, vp(c.data_ptr()), n,
                                vp(err.data_ptr()), vp(torch.cuda.current_stream().cuda_stream)), "synax_gemm_bf16")
    assert int(err.item()) == 0
    return c


# one row, a ragged and a whole row block, two row blocks; outputs below, at
# and beyond one tile of 32 columns; one K tile and the longest product
@pytest.mark.parametrize("m,n,k", [(1, 16, 64), (1, 33, 64), (96, 31, 128), (128, 32, 9216), (129, 1024, 1024),
                                   (96, 1056, 9216), (512, 1000, 64), (127, 2049, 192)])
def test_narrow_tiles_are_exact(m, n, k):
    import torch
    g = torch.Generator(device="cuda").manual_seed(m * 7 + n)
    a = torch.randint(-3, 4, (m, k), generator=g, device="cuda").to(torch.bfloat16)
    b = torch.randint(-3, 4, (n, k), generator=g, device="cuda").to(torch.bfloat16)
    assert torch.equal(_gemm(a, b), (a.double() @ b.double().T).float())


@pytest.mark.parametrize("n,k", [(1024, 1024), (1024, 9216), (9216, 1024), (256, 512)])
def test_rows_do_not_depend_on_the_tile_width(n, k):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n + k)
    a = torch.randn((8192, k), generator=g, device="cuda").to(torch.bfloat16)
    b = torch.randn((n, k), generator=g, device="cuda").to(torch.bfloat16)
    tall = _gemm(a, b)
    assert torch.equal(_gemm(a[:96].contiguous(), b), tall[:96])
    assert torch.equal(_gemm(a[512:1024].contiguous(), b), tall[512:1024])
