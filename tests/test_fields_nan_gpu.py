"""A position that is not a number has no field in the grid model, in either
precision: its cell index is clamped into the grid (grid_axis_split: fmax and
fmin return the other operand), and the result is NaN, not a blend with
arbitrary weights.  The points beside it are not touched by it."""
import numpy as np
import pytest

from paper_2410_01136_gb300 import eval_fields, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("f64", [False, True])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_nan_position_in_the_grid(f64, axis):
    prob = inputs.grid_problem(nside=2, n_steps=8, n=(8, 6, 4)).replace(f64=f64)
    pos = np.array([[1.0, 2.0, 0.3], [1.0, 2.0, 0.3], [-4.0, 0.5, 1.0]])
    want = eval_fields(prob, pos, np.ones(3)).cpu().numpy()
    assert np.isfinite(want).all()
    pos[1, axis] = np.nan
    got = eval_fields(prob, pos, np.ones(3)).cpu().numpy()
    assert np.isnan(got[1, :3]).all()
    assert np.array_equal(got[[0, 2]], want[[0, 2]])
