"""One-launch runs that keep the variables' totals instead of every slot's value (more than about
7,250 variables a block): hard evidence in the last variables, whose explicit sums are the last
entries of their array. Bitwise the multi-launch run (PGM_OPT_SMALL_RUN 0)."""
import numpy as np
import pytest

from paper_2202_04110_gb300 import workloads as W
from tests.test_gpu_small_run import _hard, _run

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


def _clamp_last(ev, n):
    """Infinite entries, both kinds and both states, in the last n variables and a few others."""
    ev = _hard(ev, 1e-4, 3, both=True)
    last = ev.reshape(-1, 2)[-n:]
    last[0::3, 0] = -np.inf
    last[1::3, 1] = -np.inf
    last[-1] = -np.inf
    return ev


@pytest.mark.parametrize("shape", [(1090, 1101), (1200, 1209)])
@pytest.mark.parametrize("T", [1.0, 0.0])
def test_one_graph(gpu, shape, T):
    p = W.ising_grid(*shape, seed=1)
    ev = _clamp_last(p.evidence, 700)
    _, want, _, _, fw = _run(gpu, p.graph, p.log_pot, ev, T, 0.5, 9, 0)
    _, got, _, _, fg = _run(gpu, p.graph, p.log_pot, ev, T, 0.5, 9, 1)
    assert np.array_equal(got, want, equal_nan=True) and fg == fw


def test_two_samples(gpu):
    """76 blocks a sample: the first sample's last sums lie before the second one's first."""
    import torch
    p = W.ising_grid(775, 777, seed=2)
    rng = np.random.default_rng(4)
    ev = np.stack([_clamp_last(rng.standard_normal(p.evidence.size).astype(np.float32), 900) for _ in range(2)])
    ev[1, :1800:4] = -np.inf
    g = gpu.Graph(p.graph)
    m = torch.zeros(2, p.graph.n_edge_states, device="cuda")
    g.run_bp_multi(torch.as_tensor(p.log_pot).cuda(), torch.as_tensor(ev).cuda(), 1.0, 0.5, 9, m)
    got = m.cpu().numpy()
    for s in range(2):
        _, want, _, _, _ = _run(gpu, p.graph, p.log_pot, ev[s], 1.0, 0.5, 9, 0)
        assert np.array_equal(got[s], want, equal_nan=True), s
