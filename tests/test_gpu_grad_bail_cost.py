"""A gradient that the one-launch form hands back for its inputs -- a table with -inf, evidence of -inf
in both states -- costs about what the launches cost, on each form, with their bits."""
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


@pytest.mark.parametrize("shape", [(10, 10), (64, 64), (120, 130)])
@pytest.mark.parametrize("what", ["table", "evidence", "NaN"])
def test_cost(gpu, shape, what):
    """(With the kernel run to its end first 1.22 times.)"""
    import torch
    p = W.ising_grid(*shape, seed=1)
    if what == "table":
        p.log_pot[-3] = -np.inf  # (the last block's)
    else:
        p.evidence[10:12] = -np.inf if what == "evidence" else np.nan
    cot = np.random.default_rng(2).standard_normal(p.evidence.size).astype(np.float32)
    a = [torch.as_tensor(x).cuda() for x in (p.log_pot, p.evidence, cot)]
    times, outs = {}, {}
    for small in (0, 1):
        g = gpu.Graph(p.graph)
        g.set_option(gpu.OPT_SMALL_RUN, small)

        def call():
            return g.grad(a[0], a[1], 1.0, 0.5, 60, 10, a[2])

        for _ in range(3):
            outs[small] = [t.nan_to_num(7.0) for t in call()]
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        best = 1e9
        for _ in range(3):
            e[0].record()
            for _ in range(5):
                call()
            e[1].record()
            torch.cuda.synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
        times[small] = best
    assert all(torch.equal(x, y) for x, y in zip(outs[0], outs[1]))
    assert times[1] <= 1.17 * times[0], times
