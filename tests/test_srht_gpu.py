"""The fast Hadamard projection (srht.cu) against the dense FP64 oracle.

Tolerance: a coefficient is a sum of N = 12 Nside^2 products +-x_p / sqrt(N)
formed by 12 + log2(Nside^2) - 1 levels of FP32 additions and one product, each
with relative error 2^-24 of a partial sum; partial sums are at most ||x||_2
sqrt(N) / sqrt(N) after scaling (Cauchy-Schwarz), so |dc| <= 28 * 2^-24 ||x||_2 =
1.7e-6 ||x||_2 for Nside <= 256.
"""
import numpy as np
import pytest

from oracle import surrogate as so
from paper_2410_01136_gb300 import inputs

pytestmark = pytest.mark.gpu


# every transform length (Nside 4 .. 64) and the folded ones (128, 256), each
# number of combinations per CTA (1, 3 and 6: rows * Nside^2 / 4096 around 76
# and 152), a full basis, and maps that start 4 bytes off a 16-byte boundary
@pytest.mark.parametrize("nside,n_basis,rows,offset", [
    (4, 192, 1, 0), (4, 64, 152, 1), (8, 128, 75, 0), (16, 192, 76, 3), (32, 64, 151, 0), (32, 12288, 2, 0),
    (64, 64, 153, 0), (64, 192, 3, 1), (128, 64, 19, 2), (128, 128, 1, 0), (256, 64, 1, 0), (256, 64, 5, 1)])
def test_projection_of_every_shape(nside, n_basis, rows, offset):
    import torch
    from paper_2410_01136_gb300.surrogate import Surrogate
    lo, hi = inputs.config5_box()
    sign, brows = inputs.surrogate_basis_spec(nside, n_basis, seed=nside + n_basis)
    sur = Surrogate(16, lo, hi, sign, brows, width=64, depth=1, nside=nside, batch=64, max_eval=64, map_chunk=8)
    npix = 12 * nside * nside
    g = torch.Generator().manual_seed(rows)
    host = 10.0 + 40.0 * torch.randn(rows * npix, generator=g)
    buf = torch.empty(rows * npix + offset, device="cuda")
    buf[offset:].copy_(host)
    c = sur.project(buf[offset:].reshape(rows, npix)).cpu().numpy()
    x = host.reshape(rows, npix).double().numpy()
    pick = np.arange(n_basis) if n_basis <= 256 else inputs.sample_pixels(n_basis, 64, seed=8)
    ref = so.project(x, nside, sign, brows[pick], chunk=64)
    assert c.shape == (rows, n_basis)
    assert np.max(np.abs(c[:, pick] - ref) / np.linalg.norm(x, axis=1)[:, None]) <= 1.7e-6
    sur.close()
