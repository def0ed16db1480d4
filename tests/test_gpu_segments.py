"""Checkpointed gradients whose segments are recomputed and swept backwards in one launch: the last
segment shorter than the others, windows a step apart, one window, one step a segment, tiles over
two windows, the smallest and the largest shapes, a single column and coarse steps, against the
oracle."""
import numpy as np
import pytest

import oracle
from paper_2407_13950_gb300 import msqoc
from paper_2407_13950_gb300 import synthetic as S

from gpu_helpers import assert_grad_close

pytestmark = pytest.mark.gpu

CASES = {
    "ragged windows and segments": (S.transmon_spec(3, 9.0, 607, 5, 6), 17, {}),
    "one window": (S.transmon_spec(2, 4.0, 201, 1, 5), 64, {}),
    "two steps a segment": (S.transmon_spec(2, 1.0, 41, 3, 5), 2, {}),
    "one qubit": (S.transmon_spec(1, 4.0, 401, 2, 5, L=2), 13, {}),
    "one column": (S.transmon_spec(2, 4.0, 301, 2, 5, ness=1), 64, {}),
    "tiles over two windows": (S.transmon_spec(3, 9.0, 601, 3, 6), 16, dict(col_block=5)),
    "four transmons": (S.transmon_spec(4, 2.4, 402, 3, 5), 64, {}),
    "five transmons": (S.transmon_spec(5, 0.6, 101, 2, 5), 16, {}),
    "six qubits": (S.transmon_spec(6, 3.0, 301, 2, 5, L=2), 50, {}),
    "QFT-8, coarse steps": (S.paper_qft_spec(3, M=2, nsteps=601), 64, {}),
}


@pytest.mark.parametrize("name", list(CASES))
def test_segments_match_the_oracle(name):
    spec, K, kw = CASES[name]
    alpha, W = S.random_alpha(spec, 71), S.random_W(spec, 71)
    want = oracle.evaluate(spec, alpha, W)
    with msqoc.Problem(spec, ckpt_interval=K, layout=msqoc.LAYOUT_FIBER, **kw) as p:
        got, again = p.eval_gradient(alpha, W), p.eval_gradient(alpha, W)
    assert_grad_close(got["grad_alpha"], want["grad_alpha"], what="grad_alpha")
    if W.size:
        assert_grad_close(got["grad_W"], want["grad_W"], what="grad_W")
    assert got["P"] == again["P"] and np.array_equal(got["grad_alpha"], again["grad_alpha"])
    assert np.array_equal(got["grad_W"], again["grad_W"])


def test_a_batch_of_checkpointed_and_whole_histories_equals_its_problems():
    specs = [S.transmon_spec(3, 9.0, 607, 5, 6), S.transmon_spec(3, 6.0, 401, 7, 6), S.transmon_spec(3, 3.0, 203, 2, 6)]
    probs = [msqoc.Problem(s, ckpt_interval=K, layout=msqoc.LAYOUT_FIBER, col_block=4) for s, K in zip(specs, (17, 64, 200))]
    ins = [(S.random_alpha(s, 5 + i), S.random_W(s, 5 + i)) for i, s in enumerate(specs)]
    want = [p.eval_gradient(*x) for p, x in zip(probs, ins)]
    with msqoc.Batch(probs, graph=True) as b:
        for i, x in enumerate(ins):
            b.set_inputs(i, *x)
        for _ in range(2):
            b.eval_gradient()
            for i, w in enumerate(want):
                got = b.get_gradient(i)
                assert all(np.array_equal(got[k], w[k]) for k in ("P", "grad_alpha", "grad_W"))
        b.eval_subset([2, 0])
        for i in (2, 0):
            assert np.array_equal(b.get_gradient(i)["grad_alpha"], want[i]["grad_alpha"])
    for p in probs:
        p.close()
