"""The field angles' reduction classes (FP32 WMAP-type and stacked models): maps
and gradients just below and above the line where the reduction is left out,
with parameters of either sign, against the FP64 oracle at the repository's
FP32 tolerances."""
import numpy as np
import pytest

import oracle
from paper_2410_01136_gb300 import adjoint, forward, inputs

from .parity import assert_parity

pytestmark = pytest.mark.gpu

# psi0 + 0.981 psi1 and chi0 around 0.785, where the class changes
ANGLES = [(0.7, 0.0866, 0.7849), (0.7, 0.0867, 0.7851), (-0.7, 0.0866, -0.7849), (-0.7, -0.0867, 0.7851),
          (2.0, 1.5, 1.6), (-3.0, 0.5, -2.5)]


def problems(psi0, psi1, chi0):
    th = np.array([6.0, psi0, psi1, chi0, 1.0, inputs.N0_EARTH, 3.0, 0.03])
    yield inputs.Problem(nside=4, n_steps=65, freq_hz=(2.4e9, 5e9), model_id=inputs.MODEL_WMAP, theta=th)
    st = inputs.wmap_stack_theta()
    for k in range(4):
        st[4 * k + 1:4 * k + 4] = (psi0, psi1, chi0) if k % 2 else (0.3, 0.1, -0.2)
    yield inputs.wmap_stack_problem(nside=4, n_steps=65, theta=st)


@pytest.mark.parametrize("angles", ANGLES)
def test_maps_and_gradients_at_the_class_edges(angles):
    import torch
    for prob in problems(*angles):
        maps = forward(prob)
        assert_parity(maps.cpu().numpy(), oracle.forward(prob))
        # the gradient of FP32 against that of FP64 for the same seed
        g = torch.ones_like(maps)
        g32 = adjoint(prob, gmaps=g).cpu().numpy()
        g64 = adjoint(prob.replace(f64=True), gmaps=g.double()).cpu().numpy()
        assert np.all(np.abs(g32 - g64) <= 1e-3 * np.abs(g64) + 1e-4 * np.max(np.abs(g64)))
