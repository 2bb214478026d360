"""CTA pairs of the GEMM at every remainder of their operand ring.

The last loads of a tile are released by commits that no later load waits for;
how many of them are outstanding when the pair ends depends on the number of K
tiles modulo the ring's 5 stages, and on whether a pair has one tile or
several.  Widths of 1024 + 64 r give 16 + r K tiles.  A wait that expired is
reported by status(); the rows must be bitwise those of the same sets evaluated
by single CTAs, which sum along K in the same order.
"""
import numpy as np
import pytest

from .test_gemm_pair_gpu import surrogate

pytestmark = pytest.mark.gpu


# one tile per pair (3000 rows), and several with a ragged last row block
@pytest.mark.parametrize("n,width", [(3000, 1024), (8193, 1024), (8193, 1088), (8193, 1152), (8193, 1216),
                                     (8193, 1280), (8193, 1344)])
def test_every_ring_remainder(n, width):
    import torch
    from paper_2410_01136_gb300 import inputs
    lo, hi = (np.asarray(v) for v in inputs.config5_box())
    u = np.random.default_rng(width).random((n, 16))
    theta = torch.tensor(lo + (hi - lo) * u, dtype=torch.float32, device="cuda")
    sur = surrogate(width, 704, n)
    for _ in range(3):                      # back to back: a pair's SMs are taken over by the next kernel at once
        c = sur(theta)
    sur.status()
    for first in (0, 1000, n - 96):
        rows = slice(first, first + 96)
        assert torch.equal(sur(theta[rows].contiguous()), c[rows])
    sur.status()
    sur.close()
