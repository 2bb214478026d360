"""FP64 field components that are nothing but a function beside its zero.

WMAP-type field on the x axis (y = z = 0, chi = 0): B_y = b0 e^(-rho/8) sin psi and
B_x = b0 e^(-rho/8) cos psi, psi = psi0 + psi1 ln(rho/8).  The points have an
exactly representable rho^2.  Tolerance: 8 roundings and functions of at most
0.53 ulp each, 8 x 2^-53."""
import numpy as np
import pytest

mp = pytest.importorskip("mpmath")

from paper_2410_01136_gb300 import eval_fields, inputs  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = 8 * 2.0 ** -53


def fields(psi0, psi1, rho):
    th = np.array([6.0, psi0, psi1, 0.4, 0.0, inputs.N0_EARTH, 3.0, 0.03])
    prob = inputs.Problem(nside=2, n_steps=4, freq_hz=(2.4e9,), model_id=inputs.MODEL_WMAP, theta=th, f64=True)
    pos = np.zeros((rho.size, 3))
    pos[:, 0] = rho
    return eval_fields(prob, pos, rho).cpu().numpy()


def test_azimuthal_component_beside_8_kpc():
    rho = np.concatenate([8 + 2.0 ** -np.arange(1.0, 24.0), 8 - 2.0 ** -np.arange(1.0, 24.0)])
    with mp.workprec(300):
        want = [float(6 * mp.exp(-mp.mpf(float(r)) / 8) * mp.sin(mp.log(mp.mpf(float(r)) / 8))) for r in rho]
    assert np.max(np.abs(fields(0.0, 1.0, rho)[:, 1] / want - 1)) <= TOL


def test_radial_component_at_a_quarter_turn():
    rho = np.array([4.0, 7.5, 8.0, 16.0])
    for quarter in (1, 3, 29, 58 * 8 + 1):
        psi0 = float(np.float64(quarter) * np.float64(np.pi / 2))
        with mp.workprec(300):
            want = [float(6 * mp.exp(-mp.mpf(float(r)) / 8) * mp.cos(mp.mpf(psi0))) for r in rho]
        assert np.max(np.abs(fields(psi0, 0.0, rho)[:, 0] / want - 1)) <= TOL
