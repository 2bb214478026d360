"""FP64 maps and gradients at 16 lanes per ray (1216 rays or more) and at 32.

Maps of a ragged pixel range (1501 rays, whose last CTA is part empty) against
the FP64 oracle at 1e-9, the repository's FP64 tolerance.  Gradients, chi^2 and
node gradients are sums over rays, so that the whole range at 16 lanes must be
the sum of shares below 1216 rays, which march at 32: the two differ by the
order of the sums and the rotation of each chunk's phase (1e-13 of a sum of
magnitudes; held to 1e-9 of it, as the maps are).
"""
import numpy as np
import pytest

import oracle
from paper_2410_01136_gb300 import adjoint, adjoint_grid, forward, inputs

from .parity import assert_parity

pytestmark = pytest.mark.gpu

RANGE = dict(pix_begin=37, pix_count=1501)
CUTS = (0, 700, 1499, 1501)                     # shares of 700, 799 and 2 rays


def problem(model, steps=77):
    kw = dict(nside=16, n_steps=steps)
    if model == "jf12":
        p = inputs.config2().replace(freq_hz=(408e6, 1.4e9, 2.3e9), **kw)
    elif model == "wmap":
        p = inputs.config1().replace(freq_hz=(408e6, 2.3e9), **kw)
    elif model == "stack":
        p = inputs.wmap_stack_problem(**kw)
    elif model == "toy":
        p = inputs.toy_problem(**kw)
    else:
        p = inputs.grid_problem(n=(20, 17, 9), **kw)
    return p.replace(f64=True, **RANGE)


def shares(prob):
    for a, b in zip(CUTS, CUTS[1:]):
        yield a, b, prob.replace(pix_begin=prob.pix_begin + a, pix_count=b - a)


def close(whole, parts):
    size = sum(np.abs(p) for p in parts)
    assert np.all(np.abs(whole - sum(parts)) <= 1e-9 * size + 1e-9 * 1e-3 * np.max(size))


@pytest.mark.parametrize("model", ["toy", "wmap", "jf12", "stack", "grid"])
def test_maps(model):
    prob = problem(model)
    whole = forward(prob).cpu().numpy()
    ref = oracle.forward(prob)                        # the whole map
    assert_parity(whole, ref[..., prob.pix_begin:prob.pix_begin + prob.pix_count], 1e-9, 1e-9, model)
    for a, b, p in shares(prob):
        assert_parity(forward(p).cpu().numpy(), whole[..., a:b], 1e-9, 1e-9, model)


# 77 steps: ragged chunks; 9 steps: lanes without a sample
@pytest.mark.parametrize("steps", [77, 9])
@pytest.mark.parametrize("model", ["wmap", "jf12", "stack", "grid"])
def test_gradients(model, steps):
    import torch
    prob = problem(model, steps)
    maps = forward(prob)
    gen = torch.Generator(device="cuda").manual_seed(steps)
    g = torch.randn(maps.shape, generator=gen, device="cuda", dtype=torch.float64)
    target = maps * (1 + 0.1 * g)
    sigma = float(maps.abs().mean())
    out = torch.empty_like(maps)
    vjp = adjoint(prob, gmaps=g, maps_out=out).cpu().numpy()
    assert torch.equal(out, maps)
    chi_grad, chi2 = (v.cpu().numpy() for v in adjoint(prob, target=target, sigma=sigma))
    parts = [[], [], []]
    for a, b, p in shares(prob):
        parts[0].append(adjoint(p, gmaps=g[..., a:b].contiguous()).cpu().numpy())
        cg, c = adjoint(p, target=target[..., a:b].contiguous(), sigma=sigma)
        parts[1].append(cg.cpu().numpy())
        parts[2].append(c.cpu().numpy())
    close(vjp, parts[0])
    close(chi_grad, parts[1])
    close(chi2, parts[2])


def test_node_gradient():
    import torch
    prob = problem("grid")
    g = torch.randn((1, 3, prob.n_pix_out), generator=torch.Generator(device="cuda").manual_seed(4), device="cuda",
                    dtype=torch.float64)
    theta, nodes = (v.cpu().numpy() for v in adjoint_grid(prob, gmaps=g))
    parts = [[v.cpu().numpy() for v in adjoint_grid(p, gmaps=g[..., a:b].contiguous())] for a, b, p in shares(prob)]
    close(theta, [p[0] for p in parts])
    close(nodes, [p[1] for p in parts])
