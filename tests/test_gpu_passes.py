"""Steps of the mixed solver's common form that take two passes (contraction factors of 0.01 to 0.03
beside rotations of a few hundredths), against the oracle.

Tolerance, norm-wise: as in test_gpu_coarse.py, 2 n 2^-52 for the oracle and for the solver each, n
the steps of a window."""
import numpy as np
import pytest

import oracle
from paper_2407_13950_gb300 import msqoc
from paper_2407_13950_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


def qft8(M, nsteps):
    return S.paper_qft_spec(3, M=M, nsteps=nsteps).replace(T=0.202 * nsteps, d1=16)


CASES = {   # spec, amplitude of the controls in the workloads' 4 MHz, options
    "QFT-8": (qft8(2, 200), 2.5, {}),
    "QFT-8, checkpoints": (qft8(3, 200), 2.5, dict(ckpt_interval=25)),
    "QFT-8, ragged windows, lean build": (qft8(3, 200), 2.5, dict(layout=msqoc.LAYOUT_FIBER_LEAN)),
    "three transmons": (S.transmon_spec(3, 9.0, 308, 2, 6), 12, {}),
}


@pytest.mark.parametrize("name", list(CASES))
def test_steps_of_two_passes_match_the_oracle(name):
    spec, amp, kw = CASES[name]
    alpha, W = amp * S.random_alpha(spec, 98), S.random_W(spec, 98)
    want = oracle.evaluate(spec, alpha, W)
    tol = 4.0 * (-(-spec.nsteps // spec.M)) * 2.0 ** -52
    with msqoc.Problem(spec, **kw) as p:
        got = p.eval_gradient(alpha, W)
    assert abs(got["P"] - want["P"]) <= tol * abs(want["P"])
    for k in ("grad_alpha", "grad_W"):
        err = np.linalg.norm(got[k] - want[k]) / np.linalg.norm(want[k])
        assert err <= tol, (k, err, tol)
