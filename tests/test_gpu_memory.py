"""A gradient whose history leaves less device memory than the adjoint's chunk of states takes runs in
smaller chunks, with the same results up to the rounding of the state between two chunks (an FP64
rounding of each entry a chunk, far below 1e-13 of the gradient); whole windows, slices, and
checkpoints whose recomputation and adjoint share a launch otherwise."""
import numpy as np
import pytest

from paper_2407_13950_gb300 import msqoc
from paper_2407_13950_gb300 import synthetic as S

from gpu_helpers import assert_grad_close, assert_objective_close

pytestmark = pytest.mark.gpu

MIB = 1 << 20
CASES = {   # spec, options, MiB left for the adjoint's states (a chunk takes 650 to 1024)
    "whole windows": (S.config_4q(64).replace(nsteps=40000, T=240.0), {}, 300),
    "slices": (S.transmon_spec(6, 20.0, 11003, 4, 5, L=2), {}, 250),
    "checkpoints": (S.config_4q(128).replace(nsteps=100000), dict(ckpt_interval=300), 200),
}


@pytest.mark.parametrize("name", list(CASES))
def test_a_short_device_memory_takes_smaller_chunks(name):
    torch = pytest.importorskip("torch")
    spec, kw, left = CASES[name]
    a, W = S.random_alpha(spec, 63), S.random_W(spec, 63)
    with msqoc.Problem(spec, **kw) as p:
        want = p.eval_gradient(a, W)
    ne = spec.N * spec.E * 16
    K = kw.get("ckpt_interval", 0)
    windows = -(-spec.nsteps // spec.M)
    held = spec.nsteps * ne if not K else spec.M * (min(K, windows) + -(-windows // K)) * ne
    with msqoc.Problem(spec, **kw) as p:
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        filler = torch.empty(free - held - left * MIB, dtype=torch.uint8, device="cuda")
        got = p.eval_gradient(a, W)
        del filler
    torch.cuda.empty_cache()
    assert_objective_close(got["P"], want["P"])
    assert_grad_close(got["grad_alpha"], want["grad_alpha"], rtol=1e-12, floor=1e-13, what="grad_alpha")
    assert_grad_close(got["grad_W"], want["grad_W"], rtol=1e-12, floor=1e-13, what="grad_W")
