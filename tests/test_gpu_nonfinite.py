"""Inputs that are not finite reach the results as NaN, whatever solver, kernel family and history:
a control coefficient that is NaN or infinite gives NaN in P and in the gradient of the evaluation,
and in the roll-out; a window state that is not finite gives NaN in P and in every entry of its
column's dP/dW, and leaves the windows it does not meet as they are.  The evaluation after it is the
one before."""
import numpy as np
import pytest

from paper_2407_13950_gb300 import msqoc
from paper_2407_13950_gb300 import synthetic as S

pytestmark = pytest.mark.gpu

QFT8 = S.paper_qft_spec(3, M=4, nsteps=1203).replace(T=40.0)
CASES = {
    "two transmons, slices": (S.transmon_spec(2, 10.0, 400, 4, 6), {}),
    "two transmons, fine steps, slices": (S.transmon_spec(2, 2.0, 400, 4, 6), {}),
    "two transmons, lane pairs": (S.transmon_spec(2, 10.0, 400, 4, 6), dict(layout=msqoc.LAYOUT_PAIR)),
    "QFT-8, slices": (QFT8, {}),
    "QFT-8, lane quads": (QFT8, dict(layout=msqoc.LAYOUT_QUAD)),
    "QFT-8, FP64": (QFT8, dict(solver=msqoc.SOLVER_FP64)),
    "four transmons, whole windows": (S.config_4q(64).replace(nsteps=640, T=3.84), {}),
    "four transmons, lean build, coarse steps": (S.config_4q(64).replace(nsteps=640, T=16.0), dict(layout=msqoc.LAYOUT_FIBER_LEAN)),
    "four transmons, checkpoints": (S.transmon_spec(4, 1.8, 300, 3, 5), dict(ckpt_interval=32)),
}


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("name", list(CASES))
def test_a_value_that_is_not_finite_reaches_the_results(name, value):
    spec, kw = CASES[name]
    alpha, W = S.random_alpha(spec, 95), S.random_W(spec, 95)
    bad_alpha, bad_W = alpha.copy(), W.copy()
    bad_alpha[2 * (spec.d1 // 2)] = value            # a spline of the first carrier, inside the grid
    col = 2 * spec.N * (spec.E + 1)                  # W^2, column 1
    bad_W[col + 5] = value
    with msqoc.Problem(spec, **kw) as p:
        before, obj = p.eval_gradient(alpha, W), p.eval_objective(alpha, W)
        assert np.isfinite(before["P"])
        assert np.isnan(p.eval_objective(bad_alpha, W)["P"])
        r = p.eval_gradient(bad_alpha, W)
        assert np.isnan(r["P"]) and np.isnan(r["grad_alpha"]).any() and np.isnan(r["grad_W"]).any()
        assert np.isnan(p.rollout(bad_alpha)).any()
        o, r = p.eval_objective(alpha, bad_W), p.eval_gradient(alpha, bad_W)
        assert np.isnan(o["P"]) and np.isnan(r["P"]) and np.isnan(r["grad_alpha"]).any()
        touched = np.array([2, 3]) - 1               # the windows that end and start at W^2
        others = np.setdiff1d(np.arange(spec.M - 1), touched)
        np.testing.assert_array_equal(o["pen"][others], obj["pen"][others])
        assert not np.isfinite(r["grad_W"][col:col + 2 * spec.N]).any()
        after = p.eval_gradient(alpha, W)
    for k in ("P", "grad_alpha", "grad_W"):
        np.testing.assert_array_equal(after[k], before[k])
