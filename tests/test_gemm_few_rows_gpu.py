"""Products of a few rows with a long K.  All CTAs then read the same few lines
of A, and beyond 64 of them the product gets slower with every further one
(1 x 9216 x 4096: 24.7 us on 36 CTAs, 35 us on 144), so narrow tiles stop there."""
import pytest

from .test_gemm_narrow_gpu import _gemm
from .test_gemm_pair_step_gpu import tile

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,k", [(1, 512), (1, 4096), (8, 4096), (1, 8192), (7, 8192), (31, 2048), (63, 1024)])
@pytest.mark.parametrize("n", [64, 1024, 2048, 4096, 6144, 9216])
@pytest.mark.parametrize("output", [0, 1, 2, 3])
def test_few_rows_run_on_few_ctas(m, n, k, output):
    assert tile(m, n, k, output)[2] <= 64


@pytest.mark.parametrize("m,n,k", [(64, 9216, 1024), (32, 9216, 2048), (8, 9216, 8192), (1, 9216, 448), (8, 9216, 960), (64, 9216, 64)])
def test_other_products_use_the_narrow_tiles(m, n, k):
    assert tile(m, n, k, 0)[2] > 64


# either side of the line (65536 elements of A), at the widths that it now chooses
@pytest.mark.parametrize("m,n,k", [(1, 9216, 4096), (15, 4096, 4096), (16, 4096, 4096), (63, 6144, 1024),
                                   (64, 6144, 1024)])
def test_few_rows_are_exact(m, n, k):
    import torch
    g = torch.Generator(device="cuda").manual_seed(m + n)
    a = torch.randint(-3, 4, (m, k), generator=g, device="cuda").to(torch.bfloat16)
    b = torch.randint(-3, 4, (n, k), generator=g, device="cuda").to(torch.bfloat16)
    assert torch.equal(_gemm(a, b), (a.double() @ b.double().T).float())
