"""problem_struct takes box and observer from anything that is indexed by 0, 1, 2,
and parameters and frequencies from anything that is iterated."""
import collections
import types

import numpy as np
import pytest

from paper_2410_01136_gb300 import inputs
from paper_2410_01136_gb300._native import MAX_FREQ, MAX_THETA, problem_struct

FORMS = [tuple, list, np.array, lambda v: np.array(v, dtype=np.float32), collections.deque,
         lambda v: dict(enumerate(v)), lambda v: list(v) + [99.0]]


@pytest.mark.parametrize("form", FORMS)
def test_box_and_observer_forms(form):
    prob = inputs.config2().replace(box_kpc=form([40.0, 24.0, 10.0]), obs_kpc=form([-8.5, 0.25, 0.5]))
    s = problem_struct(prob)
    assert list(s.box_kpc) == [40.0, 24.0, 10.0] and list(s.obs_kpc) == [-8.5, 0.25, 0.5]


@pytest.mark.parametrize("form", [tuple, list, np.array, collections.deque, iter])
def test_parameter_and_frequency_forms(form):
    base = inputs.config2()
    th, fr = [float(x) for x in base.theta], list(base.freq_hz)
    fields = {f: getattr(base, f) for f in base.__dataclass_fields__}
    s = problem_struct(types.SimpleNamespace(**{**fields, "theta": form(th), "freq_hz": form(fr), "n_pix_out": 0}))
    assert s.n_theta == len(th) and list(s.theta[:len(th)]) == th
    assert s.n_freq == len(fr) and list(s.freq_hz[:len(fr)]) == fr


def test_refused():
    base = inputs.config2()
    with pytest.raises((IndexError, ValueError)):
        problem_struct(base.replace(box_kpc=(1.0, 2.0)))
    with pytest.raises(ValueError):
        problem_struct(base.replace(freq_hz=(1e9,) * (MAX_FREQ + 1)))
    with pytest.raises(ValueError):
        problem_struct(base.replace(theta=np.ones(MAX_THETA + 1)))
