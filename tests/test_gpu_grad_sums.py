"""The sums of the one-launch gradient over a variable's factors are float-float: on a star whose leaves
0 and 2 send the centre adjoints of 10^5 that cancel exactly, what leaves 1 and 3 send is left. An
FP32 sum in slot order loses it (half an ulp of 10^5 is 0.004, the rest about 0.1). Tolerance: the
rest itself is a product of a few sigmas of some ulp each; 64 ulp = 7.6e-6 of it."""
import numpy as np
import pytest

import oracle
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


@pytest.mark.parametrize("n_iters,entries", [(1, (0,)), (2, (4,))])
def test_cancelling_adjoints(gpu, n_iters, entries):
    """Variable 0 the centre, 1 .. 4 the leaves; after one iteration the centre's evidence gradient is the
    sum of all four, after two leaf 4's holds the sum of the other three."""
    import torch
    pairs = np.array([[0, 1], [0, 2], [0, 3], [0, 4]], np.int32)
    graph = W.FactorGraph(np.full(5, 2, np.int32), [W.EnumGroup(W.PAIR2_CFG.copy(), pairs, False)], [])
    J = np.array([0.7, 0.4, 0.7, 0.5], np.float32)
    lp = np.stack([J, -J, -J, J], 1).ravel()
    ev = np.array([[0.1, -0.2], [0.3, 0.0], [0.2, 0.5], [0.3, 0.0], [-0.4, 0.1]], np.float32).ravel()
    cot = np.zeros((5, 2), np.float32)
    cot[1], cot[3] = (-3e5, 3e5), (3e5, -3e5)
    cot[2] = (-0.2, 0.3)
    args = [torch.as_tensor(a).cuda() for a in (lp, ev, cot.ravel())]
    g = gpu.Graph(graph)
    _, d_ev = g.grad(args[0], args[1], 1.0, 0.5, n_iters, 4, args[2])
    got = d_ev.cpu().numpy().reshape(5, 2)
    want = np.asarray(oracle.grad(graph, lp, ev, 1.0, 0.5, n_iters, cot.ravel())[1]).reshape(5, 2)
    for v in entries:
        assert 1e-3 < abs(want[v, 1]) < 1.0  # (what is left of the sum)
        assert np.max(np.abs(got[v] - want[v])) <= 64 * 2.0 ** -23 * abs(want[v, 1]), (got[v], want[v])
