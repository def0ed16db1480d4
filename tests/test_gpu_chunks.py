"""Sliced problems whose adjoint midpoint states exceed one chunk (1 GiB): the adjoint then runs
slice by slice in several launches, each from the state the one before left.  dP/dalpha, dP/dW and P
equal those of the same problem with checkpoints every 64 steps, whose windows are not sliced; alone,
and in a batch beside a problem of one chunk."""
import numpy as np
import pytest

from paper_2407_13950_gb300 import msqoc
from paper_2407_13950_gb300 import synthetic as S

from gpu_helpers import assert_grad_close, assert_objective_close

pytestmark = pytest.mark.gpu

SPECS = {
    "six qubits, two chunks": S.transmon_spec(6, 30.0, 17003, 4, 5, L=2),
    "six qubits, single shooting, three chunks": S.transmon_spec(6, 60.0, 35001, 1, 5, L=2),
    "four transmons, the workload's step, 8 windows": S.config_4q(8).replace(nsteps=60000, T=360.0),
}


def inputs(spec, seed):
    return S.random_alpha(spec, seed), S.random_W(spec, seed) if spec.M > 1 else None


def assert_same(got, want):
    assert_objective_close(got["P"], want["P"])
    assert_grad_close(got["grad_alpha"], want["grad_alpha"], what="grad_alpha")
    assert_grad_close(got["grad_W"], want["grad_W"], what="grad_W")


def sliced(p):
    return p.tiles * p.col_block > p.spec.M * p.spec.E + p.col_block


@pytest.mark.parametrize("name", list(SPECS))
def test_chunked_slices_equal_the_checkpointed_gradient(name):
    spec = SPECS[name]
    a, W = inputs(spec, 61)
    with msqoc.Problem(spec, ckpt_interval=64) as p:
        want = p.eval_gradient(a, W)
    with msqoc.Problem(spec) as p:
        assert sliced(p) and spec.nsteps * spec.N * spec.E * 16 > 1 << 30
        assert_same(p.eval_gradient(a, W), want)


def test_a_batch_of_chunked_and_whole_slices_equals_its_problems():
    specs = [SPECS["six qubits, two chunks"], S.transmon_spec(6, 8.0, 5003, 4, 5, L=2)]
    ins = [inputs(s, 62 + i) for i, s in enumerate(specs)]
    probs = [msqoc.Problem(s) for s in specs]
    assert all(sliced(p) for p in probs)
    want = [p.eval_gradient(*x) for p, x in zip(probs, ins)]
    with msqoc.Batch(probs, gradient=True, graph=True) as b:
        for i, x in enumerate(ins):
            b.set_inputs(i, *x)
        for _ in range(2):
            b.eval_gradient()
            got = [b.get_gradient(i) for i in (0, 1)]
        b.eval_subset([1, 0], gradient=True, slot=1)
        got += [b.get_gradient(i) for i in (0, 1)]
    for g, w in zip(got, want + want):
        assert_grad_close(g["grad_alpha"], w["grad_alpha"], rtol=1e-13, floor=1e-15, what="grad_alpha")
        assert np.array_equal(g["grad_W"], w["grad_W"])
    for p in probs:
        p.close()
