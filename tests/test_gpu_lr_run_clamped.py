"""One-launch runs with many clamped variables, some of whose messages are infinite or huge (the explicit
sums) and most finite (the infinity itself): bitwise the multi-launch run, from each form."""
import numpy as np
import pytest

from paper_2202_04110_gb300 import workloads as W
from tests.test_gpu_lr_run import _same

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


@pytest.mark.parametrize("shape", [(10, 10), (20, 20), (40, 41), (97, 101), (317, 241), (700, 700), (1090, 1101)])
@pytest.mark.parametrize("T", [1.0, 0.0])
def test_clamped(gpu, shape, T):
    p = W.ising_grid(*shape, seed=shape[0])
    rng = np.random.default_rng(1)
    e = p.evidence.reshape(-1, 2).copy()
    idx = np.flatnonzero(rng.random(e.shape[0]) < 0.3)
    e[idx, rng.integers(0, 2, idx.size)] = -np.inf
    e[idx[::11]] *= np.float32(3e37)  # the finite entry near overflow
    p.evidence = e.ravel()
    _same(gpu, p, T, 0.5, 9)
    m0 = -np.abs(rng.standard_normal((p.graph.n_edges, 2))).astype(np.float32)
    m0[rng.random(len(m0)) < 0.02, 0] = -np.inf
    m0[rng.random(len(m0)) < 0.02] *= np.float32(1e37)
    _same(gpu, p, T, 0.3, 5, m0.ravel())
