"""The quadrature kernel of the gradient at the edges of its layout against the oracle: column
counts of one, not a power of two, exactly 32 and above 32 (several column blocks a step), the
smallest and largest shapes, windows shorter than a group of steps, ragged windows, checkpointed
segments (a chunk cut by a window's end), and both forms of the stored midpoint states (split
by the one-thread families of the mixed solver, FP64 otherwise)."""
import numpy as np
import pytest

import oracle
from paper_2407_13950_gb300 import msqoc
from paper_2407_13950_gb300 import synthetic as S

from gpu_helpers import assert_grad_close, assert_objective_close

pytestmark = pytest.mark.gpu

# (levels, essential levels, subsystems, windows, steps)
SHAPES = [(2, 2, 1, 3, 40), (3, 1, 2, 4, 61), (3, 1, 4, 3, 50), (3, 3, 1, 5, 43), (3, 3, 2, 3, 47), (3, 3, 3, 2, 33),
          (2, 2, 5, 4, 66), (2, 2, 6, 2, 25), (3, 3, 4, 2, 9), (3, 2, 5, 2, 11), (2, 1, 6, 3, 40), (3, 2, 3, 40, 41)]


@pytest.mark.parametrize("L,ness,q,M,nsteps", SHAPES)
@pytest.mark.parametrize("layout,solver,K", [(msqoc.LAYOUT_FIBER, msqoc.SOLVER_MIXED, 0),
                                             (msqoc.LAYOUT_FIBER, msqoc.SOLVER_MIXED, 7),
                                             (msqoc.LAYOUT_AUTO, msqoc.SOLVER_DEFAULT, 0),
                                             (msqoc.LAYOUT_AUTO, msqoc.SOLVER_FP64, 5)])
def test_gradient_products_at_the_edges(L, ness, q, M, nsteps, layout, solver, K):
    spec = S.transmon_spec(q, 0.01 * nsteps, nsteps, M, 5, L=L, ness=ness)
    alpha, W = S.random_alpha(spec, 300 + q), S.random_W(spec, 300 + q)
    # columns of very different magnitudes share a step's sum
    scale = 2.0 ** (13.0 * np.arange(spec.E) / max(1, spec.E - 1)) if spec.E > 1 else np.ones(1)
    W = (W.reshape(spec.M - 1, spec.E, 2 * spec.N) * scale[None, :, None]).reshape(-1)
    want = oracle.evaluate(spec, alpha, W)
    with msqoc.Problem(spec, layout=layout, solver=solver, ckpt_interval=K) as p:
        got = p.eval_gradient(alpha, W)
        again = p.eval_gradient(alpha, W)
    assert_objective_close(got["P"], want["P"])
    assert_grad_close(got["grad_alpha"], want["grad_alpha"], what="grad_alpha")
    assert_grad_close(got["grad_W"], want["grad_W"], what="grad_W")
    np.testing.assert_array_equal(got["grad_alpha"], again["grad_alpha"])
