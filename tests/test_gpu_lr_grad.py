"""pgm_grad as one launch (binary graphs with a table per factor): within 1e-4 of the largest
entry of the oracle's adjoint (the criterion of the launches it replaces), on one block, a cluster
and the grid; the same bits on every call; hard evidence; and the recorded launches' bits
where the kernel hands the call back (tables with -inf entries, contradictory evidence)."""
import numpy as np
import pytest

import oracle
from paper_2202_04110_gb300 import workloads as W
from tests.test_gpu_small_run import _hard
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


def _grad(gpu, p, T, damping, n_iters, cot, small=1, repeat=2):
    import torch
    g = gpu.Graph(p.graph)
    g.set_option(gpu.OPT_SMALL_RUN, small)
    args = [torch.as_tensor(np.asarray(a, np.float32)).cuda() for a in (p.log_pot, p.evidence)]
    c = torch.as_tensor(cot).cuda()
    outs = [[t.cpu().numpy() for t in g.grad(*args, T, damping, n_iters, 7, c)] for _ in range(repeat)]
    for a, b in outs[1:]:
        assert np.array_equal(a, outs[0][0], equal_nan=True) and np.array_equal(b, outs[0][1], equal_nan=True)
    assert not g.flags(clear=True) & 8
    return outs[0]


def _close(got, want, tol=1e-4):
    for a, b in zip(got, want):
        assert np.all(np.isfinite(a))
        assert np.max(np.abs(a - b)) <= tol * max(1.0, np.max(np.abs(b)))


@pytest.mark.parametrize("shape", [(1, 2), (3, 4), (22, 22), (23, 23), (26, 27), (64, 64), (5, 400), (90, 100), (95, 96),
                                   (120, 130)])
def test_against_the_oracle(gpu, shape):
    p = W.ising_grid(*shape, seed=shape[0] + shape[1])
    cot = np.random.default_rng(1).standard_normal(p.evidence.size).astype(np.float32)
    for T, damping, n in ((1.0, 0.5, 12), (0.6, 0.0, 5)):
        want = oracle.grad(p.graph, p.log_pot, p.evidence, T, damping, n, cot)
        _close(_grad(gpu, p, T, damping, n, cot), want[:2])


@pytest.mark.parametrize("p", [random_numbering(30, 33, 1), W.ising_grid(20, 20, 2), W.ising_grid(100, 100, 3)])
def test_hard_evidence_and_bail(gpu, p):
    cot = np.random.default_rng(2).standard_normal(p.evidence.size).astype(np.float32)
    soft = p.evidence
    p.evidence = _hard(soft, 0.05, 3)
    _close(_grad(gpu, p, 1.0, 0.5, 9, cot), _grad(gpu, p, 1.0, 0.5, 9, cot, small=0), 1e-5)
    p.evidence = soft
    pot = p.log_pot
    p.log_pot = pot.copy()
    p.log_pot[5] = -np.inf  # handed back to the launches
    a, b = _grad(gpu, p, 1.0, 0.5, 6, cot), _grad(gpu, p, 1.0, 0.5, 6, cot, small=0)
    assert np.array_equal(a[0], b[0], equal_nan=True) and np.array_equal(a[1], b[1], equal_nan=True)
    p.log_pot = pot
