"""The iteration counts of a mixed one-thread step reach their target, the FP64 unit roundoff, for every
contraction factor, rotation and change of the controls from the step before, growing and falling.

The sweeps start from the step before's d = s P w(P U + d), |d| <= rho_prev |U|.  It is off by the change
of the controls, drho >= |rho - rho_prev|, and by rho_prev times the change of the state over a step,
at most 2 (kap + rho_prev) and at most 2 of its norm; never by more than |d| + |d_prev|.  j1 sweeps
multiply that by rho^j1; a pass multiplies the error by its own FP32 roundings and rho^(j2+1) (the
derivation beside step_counts)."""
import numpy as np
import pytest

from paper_2407_13950_gb300 import msqoc

U32, TARGET = 2.0 ** -24, 2.0 ** -53
COARSE, WIDE = 2, 8


def error_of(rho, rho_prev, kap, counts):
    j1, j2, passes, flags = counts
    drho = abs(rho - rho_prev)
    start = min(rho_prev * 2.0 * min(kap + rho_prev, 1.0) + drho, rho + rho_prev)
    f = U32 * ((0.0 if flags & COARSE else 2.0 * kap) + 4.0 * rho)
    return (f + rho ** j1 * start) * (f + rho ** (j2 + 1)) ** passes


@pytest.mark.parametrize("kap", [0.0, 1e-3, 0.017, 0.04, 0.0624, 0.0626, 0.3, 2.0])
def test_counts_reach_the_unit_roundoff_for_growing_and_falling_controls(kap):
    worst = 0.0
    for rho in np.float32(10.0 ** np.linspace(-8, np.log10(0.49), 120)):
        for ratio in (1.0, 0.0, 0.3, 0.9, 1.1, 2.0, 5.0, 30.0, 300.0, 1e4):
            prev = float(rho) * ratio
            if prev > 0.49:
                continue
            drho = abs(float(rho) - prev)
            c = msqoc.selftest_step_counts(msqoc.SOLVER_MIXED, 0, float(rho), kap, drho)
            assert not c[3] & 1 and bool(c[3] & WIDE) == (rho > 2.0 ** -5)
            assert (c[3] & COARSE) or (c[2] == 1 and kap <= 2.0 ** -4 and rho <= 2.0 ** -5)
            worst = max(worst, error_of(float(rho), prev, kap, c) / TARGET)
    assert worst <= 1.01, worst
