"""One-launch runs above the small forms: a cooperative grid of blocks (one graph), and
several blocks per sample (pgm_run_bp_multi), held bitwise to the multi-launch run
(PGM_OPT_SMALL_RUN 0), whose results the other tests hold to the oracle."""
import numpy as np
import pytest

from paper_2202_04110_gb300 import workloads as W
from tests.test_gpu_small_run import _hard, _run
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


def _same(binding, p, T, damping, n_iters, m0=None):
    _, mm, _, _, fm = _run(binding, p.graph, p.log_pot, p.evidence, T, damping, n_iters, 0, m0)
    _, ms, _, _, fs = _run(binding, p.graph, p.log_pot, p.evidence, T, damping, n_iters, 1, m0)
    assert np.array_equal(ms, mm, equal_nan=True), f"max diff {np.nanmax(np.abs(ms - mm))}"
    assert fs == fm, (fs, fm)


@pytest.mark.parametrize("shape", [(129, 128), (317, 241), (3000, 17), (17, 3000), (1, 40001), (500, 500), (1000, 1000),
                                   (1200, 1209), (1210, 1210)])
def test_sizes(gpu, shape):
    """Records in shared memory up to about 400,000 variables, streamed above; 17 x 3000 splits
    most factors and 1210 x 1210 exceeds the SMs: both keep the launches."""
    p = W.ising_grid(*shape, seed=shape[0])
    for T, it in ((1.0, 21), (0.0, 10)):
        _same(gpu, p, T, 0.5, it)


@pytest.mark.parametrize("rows,cols", [(150, 150), (700, 700)])
@pytest.mark.parametrize("T", [1.0, 0.0])
def test_hard_inputs(gpu, rows, cols, T):
    """Clamped and contradictory evidence, tables with -inf entries, warm starts, damping 0."""
    p = W.ising_grid(rows, cols, seed=4)
    p.evidence = _hard(p.evidence, 0.02, 5, both=True)
    rng = np.random.default_rng(6)
    pot = p.log_pot.reshape(-1, 4).copy()
    hit = np.flatnonzero(rng.random(pot.shape[0]) < 0.01)
    pot[hit, rng.integers(0, 4, hit.size)] = -np.inf
    p.log_pot = pot.ravel()
    _same(gpu, p, T, 0.5, 12)
    _same(gpu, p, T, 0.0, 7)
    m0 = np.zeros(p.graph.n_edge_states, np.float32)
    m0[::2] = -np.abs(rng.standard_normal(m0.size // 2))
    _same(gpu, p, T, 0.3, 9, m0)


def test_random_numbering_keeps_its_results(gpu):
    """Nearly every factor joins two blocks (the multi-launch run where the workspace is short)."""
    _same(gpu, random_numbering(150, 150, 3), 1.0, 0.5, 15)


@pytest.mark.parametrize("rows,cols,S", [(10, 10, 200), (40, 41, 9), (90, 100, 5), (97, 101, 20), (256, 256, 23)])
@pytest.mark.parametrize("per_sample", [False, True])
def test_samples(gpu, rows, cols, S, per_sample):
    """One block per sample, several, and records in shared memory or streamed, in one or
    more launches: each sample bitwise the multi-launch run of it alone."""
    import torch
    p = W.ising_grid(rows, cols, seed=8)
    rng = np.random.default_rng(9)
    ev = rng.standard_normal((S, p.evidence.size)).astype(np.float32)
    ev[0] = _hard(ev[0], 0.05, 10)
    pots = np.stack([p.log_pot * (1 + 0.1 * s) for s in range(S)]).astype(np.float32) if per_sample else p.log_pot
    g = gpu.Graph(p.graph)
    lp, evt = torch.as_tensor(pots).cuda(), torch.as_tensor(ev).cuda()
    m = torch.zeros(S, p.graph.n_edge_states, device="cuda")
    g.run_bp_multi(lp, evt, 1.0, 0.5, 11, m)
    got = m.cpu().numpy()
    assert g.flags(clear=True) == 0
    for s in {0, 1, S // 2, S - 1}:
        _, want, _, _, _ = _run(gpu, p.graph, pots[s] if per_sample else pots, ev[s], 1.0, 0.5, 11, 0)
        assert np.array_equal(got[s], want), s
