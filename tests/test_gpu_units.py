"""An evaluation does not depend on the unit of time: with the durations, frequencies and controls
in units 2^e times larger every result has the same bits (up to the unit of the gradient), for
units in which the controls and their squares leave the range of a float."""
import numpy as np
import pytest

from paper_2407_13950_gb300 import msqoc
from paper_2407_13950_gb300 import synthetic as S

pytestmark = pytest.mark.gpu

SPECS = {"three transmons": (S.transmon_spec(3, 9.0, 601, 4, 6), {}), "QFT-8": (S.paper_qft_spec(3, M=2, nsteps=1501).replace(T=60.0), {}),
         "four transmons, lane pairs": (S.transmon_spec(4, 2.4, 402, 8, 5), dict(layout=msqoc.LAYOUT_PAIR))}


@pytest.mark.parametrize("e", [-90, -70, 70, 90])
@pytest.mark.parametrize("name", list(SPECS))
def test_the_unit_of_time_does_not_matter(name, e):
    spec, kw = SPECS[name]
    u = 2.0 ** e
    scale = lambda x: None if x is None else [scale(y) if isinstance(y, list) else y / u for y in x]  # noqa: E731
    other = spec.replace(T=spec.T * u, xi=scale(spec.xi), xi_cross=scale(spec.xi_cross), omega=scale(spec.omega),
                         detune=scale(spec.detune), jx=scale(spec.jx))
    alpha, W = S.random_alpha(spec, 96), S.random_W(spec, 96)
    with msqoc.Problem(spec, **kw) as p, msqoc.Problem(other, **kw) as o:
        want, got = p.eval_gradient(alpha, W), o.eval_gradient(alpha / u, W)
    assert got["P"] == want["P"]
    np.testing.assert_array_equal(got["grad_W"], want["grad_W"])
    np.testing.assert_array_equal(got["grad_alpha"] / u, want["grad_alpha"])
