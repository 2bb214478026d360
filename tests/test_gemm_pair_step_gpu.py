"""The training step's output layer on CTA pairs: the squared-error epilogue of
the paired tiles (gradient, its transposed copy, target rows and their
normalisation, per-CTA loss partials).

Reference: the same rows in batches of 64, whose output layer runs on single
CTAs (both asserted), with the gradients summed in FP64.  Every product sums
along K in the same order whatever its tile, so a row's residual d is bitwise
the same; the output gradient is BF16(coef d) with coef = 2 / (rows columns).

Tolerances, norm-wise per 256 x 64 block of a weight gradient (a wrong row,
column or tile changes a block by its whole size):
 * the gradient sums `batch` products in FP32: |error| <= batch 2^-24 sum |term|
   <= batch^1.5 2^-24 (sum term^2)^1/2, and the block's norm is about that of
   (sum term^2)^1/2 for terms of independent sign: 512^1.5 2^-24 = 6.9e-4;
 * unless batch / 64 is a power of two, coef d rounds to BF16 differently
   (2^-9 relative per term, twice), independent per term: 2^-8 in all; the layers
   below round the propagated gradient to BF16 once more each: 2^-7.
Loss: FP32 sums of 9216 x batch squares, at most 2 x 256 deep per thread in
order and then by trees: (512 + 20) 2^-24 = 3.2e-5 relative.
"""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NB = 3072
WIDTH = 1024


def tile(m, n, k, output):
    from paper_2410_01136_gb300._native import check, lib
    v = [ctypes.c_int() for _ in range(3)]
    check(lib().synax_gemm_tile(m, n, k, output, *[ctypes.byref(x) for x in v]), "synax_gemm_tile")
    return tuple(x.value for x in v)


def make(batch, nside=32, **kw):
    from paper_2410_01136_gb300 import inputs
    from paper_2410_01136_gb300.surrogate import Surrogate
    lo, hi = inputs.config5_box()
    sign, rows = inputs.surrogate_basis_spec(nside, NB, seed=5)
    sur = Surrogate(16, lo, hi, sign, rows, width=WIDTH, depth=2, nside=nside, batch=batch, max_eval=64, map_chunk=8,
                    **kw)
    sur.set_params(inputs.mlp_init(sur.widths, seed=3))
    return sur


def data(batch, seed):
    from paper_2410_01136_gb300 import inputs
    lo, hi = (np.asarray(v) for v in inputs.config5_box())
    g = np.random.default_rng(seed)
    theta = (lo + (hi - lo) * g.random((batch, 16))).astype(np.float32)
    coeffs = (2.0 + 3.0 * g.normal(size=(batch, 3, NB))).astype(np.float32)
    return theta, coeffs, (1.0 + g.normal(size=3 * NB)).astype(np.float32)


def blocks(a):
    r, c = (-a.shape[0]) % 256, (-a.shape[1]) % 64
    a = np.pad(a, ((0, r), (0, c)))
    return np.sqrt((a.reshape(a.shape[0] // 256, 256, -1, 64) ** 2).sum((1, 3)))


# 512: whole pairs; 448: the last pair's second CTA holds 64 rows; 320: none
@pytest.mark.parametrize("batch", [512, 448, 320])
def test_step_on_pairs_against_single_ctas(batch):
    import torch
    assert tile(batch, 3 * NB, WIDTH, 3)[:2] == (256, 1) and tile(64, 3 * NB, WIDTH, 3)[1] == 0
    theta, coeffs, mean = data(batch, batch)
    t, c = torch.tensor(theta, device="cuda"), torch.tensor(coeffs, device="cuda")
    big, small = make(batch), make(64)
    for s in (big, small):
        s.set_normalization(mean, 2.5)
    loss = float(big.step(t, c, update=False).item())
    got = big.grads()
    want, losses = None, []
    for k in range(0, batch, 64):
        losses.append(float(small.step(t[k:k + 64].contiguous(), c[k:k + 64].contiguous(), update=False).item()))
        g = [(W.astype(np.float64) * 64 / batch, b.astype(np.float64) * 64 / batch) for W, b in small.grads()]
        want = g if want is None else [(W0 + W, b0 + b) for (W0, b0), (W, b) in zip(want, g)]
    big.status()
    small.status()
    assert abs(loss - np.mean(losses)) <= 3.2e-5 * np.mean(losses)
    exact = (batch // 64) & (batch // 64 - 1) == 0
    for l, ((W, b), (Wr, br)) in enumerate(zip(got, want)):
        tol = 6.9e-4 if exact else (2.0 ** -8 if l == len(want) - 1 else 2.0 ** -7)
        assert np.all(blocks(W - Wr) <= tol * blocks(Wr)), l
        assert np.linalg.norm(b - br) <= tol * np.linalg.norm(br), l
    big.close()
    small.close()


def test_captured_training_on_pairs():
    """train(): target rows in the shuffled order of a stored data set.  With a
    data set of one batch the shuffle is a permutation of its rows, which the
    loss and the gradients do not depend on beyond the order of their sums."""
    import torch
    from paper_2410_01136_gb300 import forward, inputs
    batch, nside = 512, 16
    prob = inputs.config5_problem().replace(nside=nside, n_steps=8)
    thetas = inputs.config5_thetas(batch, seed=50)
    sur, ref = make(batch, nside), make(batch, nside)
    sur.dataset(prob, thetas)
    mean, scale = sur.normalization()
    ref.set_normalization(mean, scale)
    maps = torch.stack([forward(prob.with_theta(th))[0] for th in thetas])
    coeffs = ref.project(maps)
    loss = ref.step(torch.tensor(thetas, dtype=torch.float32, device="cuda"), coeffs, update=False)
    got = sur.train(1, seed=9)
    assert abs(got[0] - float(loss.item())) <= 3.2e-5 * got[0]
    for (W, b), (Wr, br) in zip(sur.grads(), ref.grads()):
        W, Wr = W.astype(np.float64), Wr.astype(np.float64)
        assert np.all(blocks(W - Wr) <= 2 * 6.9e-4 * np.maximum(blocks(Wr), 1e-3 * np.linalg.norm(Wr)))
        assert np.linalg.norm(b - br) <= 2 * 6.9e-4 * np.linalg.norm(br)
    sur.close()
    ref.close()


@pytest.mark.parametrize("m,n,k,output", [(8193, 1024, 1024, 1), (16584, 1024, 1024, 1), (20000, 1088, 1088, 1),
                                          (6144, 2048, 2048, 1), (16584, 1024, 2112, 2), (20000, 1088, 2496, 2),
                                          (3000, 1024, 1024, 1)] + [(8193, w, w, 1) for w in range(1088, 1345, 64)])
def test_the_paired_tests_run_pairs(m, n, k, output):
    """The products of test_gemm_pair_gpu and test_gemm_pair_ring_gpu."""
    assert tile(m, n, k, output)[:2] == (256, 1)
