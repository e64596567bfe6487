"""pgm_grad with the evidence gradient written over the cotangent: the launches' bits, also where the
one-launch form would hand the call back (a table of -inf)."""
import ctypes

import numpy as np
import pytest

from paper_2202_04110_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_04110_gb300 import build
    build.build()
    from paper_2202_04110_gb300 import binding
    return binding


@pytest.mark.parametrize("shape", [(9, 11), (64, 64), (120, 130)])
@pytest.mark.parametrize("hard", [False, True])
def test_in_place(gpu, shape, hard):
    import torch
    p = W.ising_grid(*shape, seed=1)
    if hard:
        p.log_pot[5] = -np.inf
    cot = np.random.default_rng(2).standard_normal(p.evidence.size).astype(np.float32)
    g = gpu.Graph(p.graph)
    lp, ev, c = (torch.as_tensor(a).cuda() for a in (p.log_pot, p.evidence, cot))
    g.set_option(gpu.OPT_SMALL_RUN, 0)
    want = [t.nan_to_num(7.0) for t in g.grad(lp, ev, 1.0, 0.5, 8, 4, c)]
    g.set_option(gpu.OPT_SMALL_RUN, 1)
    d_lp = torch.empty_like(lp)
    gpu.check(gpu.load_library().pgm_grad(g._h, lp.data_ptr(), ev.data_ptr(), 1.0, 0.5, 8, 4, c.data_ptr(), d_lp.data_ptr(),
                                          c.data_ptr(), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    assert torch.equal(d_lp.nan_to_num(7.0), want[0]) and torch.equal(c.nan_to_num(7.0), want[1])
