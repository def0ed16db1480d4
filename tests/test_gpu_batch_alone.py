"""A member's results in a batch are those it has alone, bit by bit, beside members of any size: small
problems, whose gradient products are formed in FP64, keep them beside larger ones of their shape."""
import numpy as np
import pytest

from paper_2407_13950_gb300 import msqoc
from paper_2407_13950_gb300 import synthetic as S

pytestmark = pytest.mark.gpu

SETS = {
    "two transmons": [S.config_2q(M).replace(nsteps=n, T=0.025 * n) for M, n in ((8, 400), (8, 14000), (32, 4000), (4, 801))],
    "QFT-4": [S.paper_qft_spec(2, M=M, nsteps=n).replace(T=0.084 * n, d1=12) for M, n in ((16, 2252), (16, 30011), (3, 503))],
    "two transmons, lane pairs": [S.config_2q(8).replace(nsteps=n, T=0.025 * n) for n in (400, 14000)],
}


@pytest.mark.parametrize("name", list(SETS))
def test_members_equal_themselves_alone(name):
    specs = SETS[name]
    kw = dict(layout=msqoc.LAYOUT_PAIR) if "pairs" in name else {}
    probs = [msqoc.Problem(s, **kw) for s in specs]
    ins = [(S.random_alpha(s, 21 + i), S.random_W(s, 21 + i)) for i, s in enumerate(specs)]
    want = [p.eval_gradient(*x) for p, x in zip(probs, ins)]
    with msqoc.Batch(probs, gradient=True, graph=True) as b:
        for i, x in enumerate(ins):
            b.set_inputs(i, *x)
        b.eval_gradient()
        got = [b.get_gradient(i) for i in range(len(probs))]
        b.eval_subset([1, 0], gradient=True, slot=1)
        got += [b.get_gradient(i) for i in (0, 1)]
    for g, w in zip(got, want + want[:2]):
        for k in ("P", "grad_alpha", "grad_W"):
            np.testing.assert_array_equal(g[k], w[k])
    for p in probs:
        p.close()
