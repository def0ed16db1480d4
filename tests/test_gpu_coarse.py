"""Steps on either side of the mixed solver's bounds for its common form (kappa = h max|D| / 2 of 2^-4,
contraction factor rho of 2^-5): few and many steps around them, rotations of up to 0.7 and factors
of up to 0.4 a step, controls that cross the bound within a window, tiles over two windows whose
steps differ, slices, checkpoints and both register builds, against the oracle.

Tolerance, norm-wise: the oracle and the solver each round a state a few times a step, about 2^-53
of its norm, and a window has n steps: 2 n 2^-52 in the worst case for each, 4 n 2^-52 together."""
import numpy as np
import pytest

import oracle
from paper_2407_13950_gb300 import msqoc
from paper_2407_13950_gb300 import synthetic as S

pytestmark = pytest.mark.gpu

FIBER, LEAN = dict(layout=msqoc.LAYOUT_FIBER), dict(layout=msqoc.LAYOUT_FIBER_LEAN)


def qft8(h, nsteps, M):
    return S.paper_qft_spec(3, M=M, nsteps=nsteps).replace(T=h * nsteps, d1=6)


CASES = {   # spec, amplitude of the controls in the workloads' 4 MHz, options
    "kappa just below": (S.transmon_spec(3, 9.0, 308, 3, 5), 1, {}),
    "kappa just above": (S.transmon_spec(3, 9.0, 300, 3, 5), 1, {}),
    "kappa just above, checkpoints": (S.transmon_spec(3, 9.0, 300, 3, 5), 1, dict(ckpt_interval=33)),
    "rho across its bound": (S.transmon_spec(3, 9.0, 300, 3, 5), 20, {}),
    "rho across its bound, two-window tiles": (S.transmon_spec(3, 9.0, 301, 4, 9), 20, dict(col_block=5, ckpt_interval=64)),
    "large rotations": (S.transmon_spec(3, 90.0, 300, 3, 5), 1, {}),
    "large rotations and factors": (S.transmon_spec(3, 90.0, 300, 3, 5), 6, {}),
    "two transmons, large factors": (S.transmon_spec(2, 60.0, 200, 2, 5), 10, {}),
    "four transmons, whole windows": (S.transmon_spec(4, 40.0, 300, 20, 5), 2, {**FIBER, "ckpt_interval": 100}),
    "four transmons, lean, two-window tiles": (S.transmon_spec(4, 60.0, 301, 20, 6), 8, {**LEAN, "col_block": 14, "ckpt_interval": 100}),
    "five transmons": (S.transmon_spec(5, 9.0, 101, 2, 5), 6, dict(ckpt_interval=16)),
    "QFT-8, both": (qft8(0.4, 200, 2), 6, {}),
    "QFT-8, factors of 0.4": (qft8(0.4, 200, 2), 15, {}),
    "one qubit": (S.transmon_spec(1, 200.0, 200, 2, 5, L=2), 8, {}),
}


@pytest.mark.parametrize("name", list(CASES))
def test_coarse_steps_match_the_oracle(name):
    spec, amp, kw = CASES[name]
    alpha, W = amp * S.random_alpha(spec, 97), S.random_W(spec, 97)
    want = oracle.evaluate(spec, alpha, W)
    tol = 4.0 * (-(-spec.nsteps // spec.M)) * 2.0 ** -52
    with msqoc.Problem(spec, **kw) as p:
        obj, got, again = p.eval_objective(alpha, W), p.eval_gradient(alpha, W), p.eval_gradient(alpha, W)
    for r in (obj, got):
        assert abs(r["P"] - want["P"]) <= tol * abs(want["P"])
    for k in ("grad_alpha", "grad_W"):
        err = np.linalg.norm(got[k] - want[k]) / np.linalg.norm(want[k])
        assert err <= tol, (k, err, tol)
        np.testing.assert_array_equal(got[k], again[k])
