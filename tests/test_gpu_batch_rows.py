"""A batch of more problems of one shape than a grid's y or z dimension has rows (65535), sliced ones:
its first and last members' gradients are those they have alone, evaluated together and as a subset."""
import numpy as np
import pytest

from paper_2407_13950_gb300 import msqoc
from paper_2407_13950_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


def test_more_members_than_rows_of_a_grid():
    spec = S.transmon_spec(1, 1.0, 20, 2, 5, L=2)
    n = 65535 + 9
    alpha, W = S.random_alpha(spec, 3), S.random_W(spec, 3)
    probs = [msqoc.Problem(spec) for _ in range(n)]
    assert probs[0].tiles * probs[0].col_block > spec.M * spec.E + probs[0].col_block, "not sliced"
    want = probs[0].eval_gradient(alpha, W)
    with msqoc.Batch(probs, gradient=True) as b:
        for i in (0, n - 1):
            b.set_inputs(i, alpha, W)
        b.eval_gradient()
        got = [b.get_gradient(i) for i in (0, n - 1)]
        b.eval_subset(list(range(n)), gradient=True, slot=0)
        got += [b.get_gradient(i) for i in (0, n - 1)]
    for g in got:
        for k in ("P", "grad_alpha", "grad_W"):
            np.testing.assert_array_equal(g[k], want[k])
    for p in probs:
        p.close()
