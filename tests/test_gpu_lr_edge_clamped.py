"""RBMs with a whole layer clamped (one state's evidence -inf), the ordinary conditional inference, in
edge-order log-ratios: the edge-state iteration's results, and about the unclamped run's time."""
import numpy as np
import pytest

from paper_2202_04110_gb300 import workloads as W
from tests.test_gpu_lr_edge import _close

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


def _clamp(p, n_vis, layer, keep=0):
    e = p.evidence.reshape(-1, 2).copy()
    idx = np.arange(n_vis) if layer == "visible" else np.arange(n_vis, e.shape[0])
    idx = idx[keep:]
    e[idx, np.random.default_rng(1).integers(0, 2, idx.size)] = -np.inf
    p.evidence = e.ravel()
    return p


@pytest.mark.parametrize("shape", [(67, 71), (70, 1), (100, 150), (3, 1025), (784, 500)])
@pytest.mark.parametrize("layer", ["visible", "hidden"])
@pytest.mark.parametrize("T", [1.0, 0.0])
def test_clamped_layer(gpu, shape, layer, T):
    p = _clamp(W.rbm(*shape, seed=shape[1]), shape[0], layer)
    _close(gpu, p, T, 0.5, 12)
    m0 = -np.abs(np.random.default_rng(3).standard_normal((p.graph.n_edges, 2))).astype(np.float32)
    m0[5::97, 0] = -np.inf  # infinite messages at clamped variables: the explicit sums
    p = _clamp(W.rbm(*shape, seed=2), shape[0], layer, keep=1)
    _close(gpu, p, T, 0.3, 7, m0=m0.ravel())


@pytest.mark.parametrize("shape,layer", [((784, 500), "visible"), ((2000, 128), "hidden")])
def test_cost(gpu, shape, layer):
    """With explicit sums for every clamped variable: 2.0 and 2.2 times the unclamped run."""
    import torch
    times = []
    for p in (W.rbm(*shape, seed=1), _clamp(W.rbm(*shape, seed=1), shape[0], layer)):
        g = gpu.Graph(p.graph)
        lp, ev, m = torch.as_tensor(p.log_pot).cuda(), torch.as_tensor(p.evidence).cuda(), g.new_msgs()
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        for r in range(6):
            if r == 3:
                e[0].record()
            g.run_bp(lp, ev, 1.0, 0.5, 100, m.zero_())
        e[1].record()
        torch.cuda.synchronize()
        times.append(e[0].elapsed_time(e[1]))
    assert times[1] <= 1.5 * times[0], times
