"""A window's results do not depend on the window that shares its tile, also where one of the two takes
coarse steps and the other does not: the gradients of a problem's shards, whose tiles pair the windows
otherwise, have the bits of the whole problem's."""
import numpy as np
import pytest

from paper_2407_13950_gb300 import msqoc, shard
from paper_2407_13950_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [dict(layout=msqoc.LAYOUT_FIBER), dict(layout=msqoc.LAYOUT_FIBER_LEAN)])
def test_shards_equal_the_whole_problem_beside_coarse_windows(kw):
    # controls that rise and fall over every pair of windows: contraction factors on both sides of
    # 2^-5, rotations below 2^-4, tiles of 5 columns over windows of 8
    spec = S.transmon_spec(3, 9.0, 330, 6, 30)
    alpha, W = S.random_alpha(spec, 99), S.random_W(spec, 99)
    t = np.arange(spec.d1)
    envelope = 1.0 + 24.0 * (np.sin(2 * np.pi * 3 * t / spec.d1) > 0)
    alpha = (alpha.reshape(-1, spec.d1, 2) * envelope[:, None]).reshape(-1)
    opts = dict(col_block=5, ckpt_interval=50, **kw)
    with msqoc.Problem(spec, **opts) as p:
        whole = p.eval_gradient(alpha, W)
    for ranges in ([(1, 1), (2, 6)], [(1, 3), (4, 6)], [(1, 2), (3, 3), (4, 6)]):
        parts = []
        for first, last in ranges:
            lo, hi = shard.w_slice(spec, first, last)
            with msqoc.Problem(spec, windows=(first, last), **opts) as s:
                parts.append(((first, last), s.eval_gradient(alpha, W[lo:hi])))
        np.testing.assert_array_equal(shard.combine(spec, parts)["grad_W"], whole["grad_W"])
