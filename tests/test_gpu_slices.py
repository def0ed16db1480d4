"""Windows cut into slices that run at the same time (propagators, their chain, then all slices'
sweeps at once), which the library chooses for problems whose columns do not fill the GPU: single
shooting, few and ragged windows, the smallest and largest shapes, one column, coarse steps, tiles
over two slices, shards and batches, against the oracle; and the roll-out, which always runs on
the windows' propagators."""
import numpy as np
import pytest

import oracle
from paper_2407_13950_gb300 import msqoc, shard
from paper_2407_13950_gb300 import synthetic as S

from gpu_helpers import assert_grad_close, assert_objective_close

pytestmark = pytest.mark.gpu

CASES = {
    "one qubit": (S.transmon_spec(1, 4.0, 401, 1, 5, L=2), {}),
    "one transmon, one column": (S.transmon_spec(1, 6.0, 640, 2, 5, ness=1), {}),
    "two transmons, all levels essential": (S.transmon_spec(2, 4.0, 403, 2, 5, ness=3), {}),
    "QFT-8, single shooting": (S.paper_qft_spec(3, M=1, nsteps=19806).replace(nsteps=900, T=22.7), {}),
    "QFT-4, ragged windows": (S.paper_qft_spec(2, M=3, nsteps=1003), {}),
    "QFT-8, coarse steps": (S.paper_qft_spec(3, M=2, nsteps=601), {}),
    "six qubits": (S.transmon_spec(6, 3.0, 301, 1, 5, L=2), {}),
    "four transmons, single shooting": (S.transmon_spec(4, 2.4, 402, 1, 5), {}),
    "three transmons, tiles over two slices": (S.transmon_spec(3, 9.0, 601, 2, 6), dict(col_block=5)),
    "three transmons, lean build": (S.transmon_spec(3, 9.0, 601, 2, 6), dict(layout=msqoc.LAYOUT_FIBER_LEAN)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_sliced_evaluation_and_rollout_match_the_oracle(name):
    spec, kw = CASES[name]
    alpha, W = S.random_alpha(spec, 90), S.random_W(spec, 90)
    want = oracle.evaluate(spec, alpha, W)
    with msqoc.Problem(spec, **kw) as p:
        assert p.tiles * p.col_block > spec.M * spec.E + p.col_block, "the problem is not sliced"
        obj = p.eval_objective(alpha, W)
        got = p.eval_gradient(alpha, W)
        again = p.eval_gradient(alpha, W)
        roll = p.rollout(alpha)
    for r in (obj, got):
        assert_objective_close(r["P"], want["P"])
    assert_objective_close(obj["J"], want["J"])
    np.testing.assert_allclose(obj["pen"], want["pen"], rtol=1e-12)
    assert_grad_close(got["grad_alpha"], want["grad_alpha"], what="grad_alpha")
    assert_grad_close(got["grad_W"], want["grad_W"], what="grad_W")
    for k in ("grad_alpha", "grad_W"):
        np.testing.assert_array_equal(got[k], again[k])
    if spec.M > 1:
        np.testing.assert_allclose(roll, oracle.rollout(spec, alpha), rtol=0, atol=1e-12)


def test_sliced_shards_and_batches_equal_the_whole_problem():
    spec = S.paper_qft_spec(3, M=4, nsteps=1203).replace(T=40.0)
    other = S.transmon_spec(2, 10.0, 801, 3, 6)
    alpha, W = S.random_alpha(spec, 91), S.random_W(spec, 91)
    a2, W2 = S.random_alpha(other, 92), S.random_W(other, 92)
    with msqoc.Problem(spec) as p, msqoc.Problem(spec) as p2, msqoc.Problem(other) as q:
        assert p.tiles * p.col_block > spec.M * spec.E + p.col_block
        whole, second = p.eval_gradient(alpha, W), q.eval_gradient(a2, W2)
        with msqoc.Batch([p, q, p2], gradient=True, graph=True) as b:
            for _ in range(2):
                for i, (a, w) in enumerate(((alpha, W), (a2, W2), (alpha, W))):
                    b.set_inputs(i, a, w)
                b.eval_gradient()
                got = [b.get_gradient(i) for i in range(3)]
            b.eval_subset([1, 2], gradient=True, slot=1)
            got += [b.get_gradient(1), b.get_gradient(2)]
            b.eval_objective()
            objs = [b.get_objective(i) for i in range(3)]
    for g, w in zip(got, (whole, second, whole, second, whole)):
        for k in ("grad_alpha", "grad_W"):
            assert_grad_close(g[k], w[k], rtol=1e-13, floor=1e-15, what=k)
        assert_objective_close(g["P"], w["P"], rtol=1e-14)
    for o, w in zip(objs, (whole, second, whole)):
        assert_objective_close(o["P"], w["P"], rtol=1e-14)
    parts = []
    for first, last in shard.partition(spec.M, 3):
        lo, hi = shard.w_slice(spec, first, last)
        with msqoc.Problem(spec, windows=(first, last)) as s:
            parts.append(((first, last), s.eval_gradient(alpha, W[lo:hi])))
    np.testing.assert_array_equal(shard.combine(spec, parts)["grad_W"], whole["grad_W"])
