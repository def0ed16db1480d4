"""Inputs that the kernels read in the caller's device memory against the copied ones (host arrays,
device arrays off their alignment), outputs written over the inputs, inputs rewritten right behind
the call, and launches that follow one another without a pause: the same bits every way."""
import numpy as np
import pytest
import torch

from paper_2407_13950_gb300 import msqoc
from paper_2407_13950_gb300 import synthetic as S

pytestmark = pytest.mark.gpu

SPECS = {
    "QFT-4": S.paper_qft_spec(2, M=16),
    "one window": S.transmon_spec(2, 4.0, 403, 1, 5),
    "lane pairs": S.transmon_spec(3, 9.0, 601, 4, 6),
    "four transmons": S.transmon_spec(4, 2.4, 402, 3, 5),
}


def _device(x, off):
    """x on the device, `off` doubles behind an aligned address."""
    buf = torch.zeros(x.size + off, dtype=torch.float64, device="cuda")
    buf[off:] = torch.from_numpy(x).cuda()
    return buf[off:]


@pytest.mark.parametrize("name", list(SPECS))
def test_inputs_in_place_equal_copied_inputs(name):
    spec = SPECS[name]
    kw = dict(layout=msqoc.LAYOUT_PAIR) if name == "lane pairs" else {}
    alpha, W = S.random_alpha(spec, 3), S.random_W(spec, 3)
    with msqoc.Problem(spec, **kw) as p:
        want = p.eval_gradient(alpha, W)
        want_obj = p.eval_objective(alpha, W)["P"]
        for off in (0, 1):                     # W read in place, then (off 16 bytes) copied
            a, w = _device(alpha, off), _device(W, off)
            P = torch.zeros(4, dtype=torch.float64, device="cuda")
            ga, gw = torch.zeros_like(a), torch.zeros(max(1, W.size), dtype=torch.float64, device="cuda")
            P2 = torch.zeros_like(P)
            for _ in range(5):                 # back to back, no pause
                p.eval_gradient_into(a, w if W.size else None, P, ga, gw if W.size else None)
                p.eval_objective_into(a, w if W.size else None, P2)
            keep = a.clone()
            a.zero_()                          # behind the call, on its stream
            torch.cuda.synchronize()
            assert float(P[0]) == want["P"] and float(P2[0]) == want_obj
            assert np.array_equal(ga.cpu().numpy(), want["grad_alpha"])
            if W.size:
                assert np.array_equal(gw.cpu().numpy()[:W.size], want["grad_W"])
            # outputs over the inputs
            a.copy_(keep)
            if off == 0:
                p.eval_gradient_into(a, w if W.size else None, P, a, w if W.size else None)
                torch.cuda.synchronize()
                assert np.array_equal(a.cpu().numpy(), want["grad_alpha"])
                if W.size:
                    assert np.array_equal(w.cpu().numpy(), want["grad_W"])
