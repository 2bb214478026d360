"""GEMM tiles of 256 x 256 shared by two CTAs (chosen for many rows and a long
K: the hidden layers and the output layer's adjoint of a large evaluation).

A set's coefficients and gradient do not depend on the others', and every tile
width sums along K in the same order, so the rows of a large evaluation must be
bitwise those of the same sets evaluated a few at a time by single CTAs.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def surrogate(width, n_basis, rows):
    from paper_2410_01136_gb300 import inputs
    from paper_2410_01136_gb300.surrogate import Surrogate
    lo, hi = inputs.config5_box()
    sign, brows = inputs.surrogate_basis_spec(16, n_basis, seed=5)
    sur = Surrogate(16, lo, hi, sign, brows, width=width, depth=3, nside=16, batch=64, max_eval=rows, map_chunk=1)
    sur.set_params(inputs.mlp_init(sur.widths, seed=3))
    return sur


# one row past a pair's upper CTA, a ragged lower CTA, an even number of pairs,
# several waves of tiles; outputs of whole and ragged columns
@pytest.mark.parametrize("n,width,n_basis", [(8193, 1024, 1024), (16384 + 200, 1024, 704), (20000, 1088, 832),
                                             (6144, 2048, 1024)])
def test_rows_of_large_evaluations(n, width, n_basis):
    import torch
    from paper_2410_01136_gb300 import inputs
    lo, hi = (np.asarray(v) for v in inputs.config5_box())
    u = np.random.default_rng(7).random((n, 16))
    theta = torch.tensor(lo + (hi - lo) * u, dtype=torch.float32, device="cuda")
    g = torch.randn((n, 3, n_basis), generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")
    sur = surrogate(width, n_basis, n)
    c, gt = sur(theta, g)
    for first in (0, 128, 4000, n - 96):
        rows = slice(first, first + 96)
        cs, gs = sur(theta[rows].contiguous(), g[rows].contiguous())
        assert torch.equal(cs, c[rows]) and torch.equal(gs, gt[rows])
    sur.status()

