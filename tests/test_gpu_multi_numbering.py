"""Many samples of a grid whose variables are numbered at random (several blocks a sample do not pay):
the launches where the samples are few, one block a sample where they are many, the same bits."""
import numpy as np
import pytest

from tests.test_gpu_small_run import _run
from tests.test_lr_run_cpu import random_numbering

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


@pytest.mark.parametrize("side,S", [(45, 3), (60, 8), (60, 24), (97, 8)])
def test_bits(gpu, side, S):
    import torch
    p = random_numbering(side, side, 1)
    ev = np.random.default_rng(2).standard_normal((S, p.evidence.size)).astype(np.float32)
    g = gpu.Graph(p.graph)
    lp, evt = torch.as_tensor(p.log_pot).cuda(), torch.as_tensor(ev).cuda()
    got = g.run_bp_multi(lp, evt, 1.0, 0.5, 11, torch.zeros(S, p.graph.n_edge_states, device="cuda")).cpu().numpy()
    for s in {0, S // 2, S - 1}:
        _, want, _, _, _ = _run(gpu, p.graph, p.log_pot, ev[s], 1.0, 0.5, 11, 0)
        assert np.array_equal(got[s], want), s


def test_few_samples_cost_no_more_than_the_launches(gpu):
    """97 x 97, 8 samples: one block a sample took 2.8 times the launches' time."""
    import torch
    p = random_numbering(97, 97, 1)
    S = 8
    lp = torch.as_tensor(p.log_pot).cuda()
    ev = torch.randn(S, p.evidence.size, device="cuda")
    g = gpu.Graph(p.graph)
    m = torch.zeros(S, p.graph.n_edge_states, device="cuda")
    times = {}
    for small in (1, 0):
        g.set_option(gpu.OPT_SMALL_RUN, small)
        for _ in range(3):
            g.run_bp_multi(lp, ev, 1.0, 0.5, 200, m)
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record()
        for _ in range(5):
            g.run_bp_multi(lp, ev, 1.0, 0.5, 200, m)
        e[1].record()
        torch.cuda.synchronize()
        times[small] = e[0].elapsed_time(e[1])
    assert times[1] <= 2 * times[0], times
