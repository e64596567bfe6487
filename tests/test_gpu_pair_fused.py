"""The fused form of dense K-state pairwise groups (variable and factor pass in one kernel,
the default for members whose only group this is with at most 4 factors per variable): bitwise
the two-pass thread form (PGM_OPT_PAIR_FORM 1), which the other tests hold to the oracle."""
import numpy as np
import pytest

from paper_2202_04110_gb300 import workloads as W
from tests.test_gpu_pair_forms import _hard, _run_form

pytestmark = pytest.mark.gpu
FUSED = {4: 16, 8: 17, 16: 18}


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_04110_gb300 import build
    build.build()
    from paper_2202_04110_gb300 import binding
    return binding


def _chain(n, K, seed, shared=True, w=1.0):
    """A chain of n variables with one general (asymmetric) table, or one per factor."""
    rng = np.random.default_rng(seed)
    pairs = np.stack([np.arange(n - 1), np.arange(1, n)], 1).astype(np.int32)
    g = W.FactorGraph(np.full(n, K, np.int32), [W.EnumGroup(W.dense_pair_cfg(K, K), pairs, shared)], [])
    pot = rng.normal(0, w, K * K * (1 if shared else n - 1)).astype(np.float32)
    return W.Problem("chain", g, pot, rng.standard_normal(n * K).astype(np.float32), 1.0, 0.5, 10)


def _same(gpu, p, T, n_iters, damping=0.5, samples=0, ev=None, fused=True):
    K = int(p.graph.num_states[-1]) if not isinstance(p.graph, list) else None
    ev = p.evidence if ev is None else ev
    g0, a = _run_form(gpu, p.graph, p.log_pot, ev, T, n_iters, 0, damping, samples)
    g1, b = _run_form(gpu, p.graph, p.log_pot, ev, T, n_iters, 1, damping, samples)
    if K:
        assert (g0.launches()[-1][1] == FUSED[K]) == fused
    assert np.array_equal(a, b, equal_nan=True), np.nanmax(np.abs(a - b))
    assert g0.flags(clear=True) == g1.flags(clear=True)


@pytest.mark.parametrize("K", [4, 8, 16])
@pytest.mark.parametrize("T", [0.0, 0.7, 1.0])
def test_tile_edges(gpu, K, T):
    for n in (2, 63, 64, 65, 129, 5000):
        _same(gpu, _chain(n, K, n), T, 9)
    _same(gpu, W.potts_grid(37, K, 1), T, 12)
    _same(gpu, W.potts_grid(1 + 64, K, 1), T, 3, damping=0.0)
    _same(gpu, _chain(200, K, 5, shared=False), T, 7, fused=False)  # a table per factor: the two passes
    _same(gpu, _chain(200, K, 6, w=40.0), T, 7)             # range above 60 T: entry by entry
    _same(gpu, _hard(W.potts_grid(30, K, 2, w=9.0), 0.1, 3), T, 15)


@pytest.mark.parametrize("T", [0.0, 1.0])
def test_batch_and_samples(gpu, T):
    """Members of several state counts and sizes at any offset, a member alone and in the
    batch, and many samples at once."""
    ps = [W.potts_grid(s, K, s) for s, K in ((9, 4), (16, 8), (5, 16), (21, 16), (8, 2), (33, 4), (2, 8))]
    b = W.Problem("b", [p.graph for p in ps], np.concatenate([p.log_pot for p in ps]),
                  np.concatenate([p.evidence for p in ps]), T, 0.5, 8)
    _same(gpu, b, T, 8)
    g, m = _run_form(gpu, b.graph, b.log_pot, b.evidence, T, 8, 0)
    for i, p in enumerate(ps):
        if p.graph.num_states[0] == 2:
            continue
        mem = g.member(i)
        _, alone = _run_form(gpu, p.graph, p.log_pot, p.evidence, T, 8, 0)
        assert np.array_equal(m[mem["es_off"]:mem["es_off"] + mem["n_edge_states"]], alone)
    for K in (4, 16):
        p = W.potts_grid(13, K, 7)
        ev = np.random.default_rng(1).standard_normal((5, p.evidence.size)).astype(np.float32)
        _same(gpu, p, T, 6, samples=5, ev=ev)


def test_not_taken(gpu):
    """A variable with 5 factors, and two groups on one variable, keep the two passes."""
    K = 4
    star = np.stack([np.zeros(5), np.arange(1, 6)], 1).astype(np.int32)
    g = W.FactorGraph(np.full(6, K, np.int32), [W.EnumGroup(W.dense_pair_cfg(K, K), star, True)], [])
    rng = np.random.default_rng(0)
    p = W.Problem("star", g, rng.standard_normal(16).astype(np.float32), rng.standard_normal(24).astype(np.float32), 1.0, 0.5, 5)
    _same(gpu, p, 1.0, 5, fused=False)
    p = _chain(20, K, 3)
    g = p.graph
    g.enum_groups.append(W.EnumGroup(W.dense_pair_cfg(K, K), np.array([[0, 2]], np.int32), True))
    p.log_pot = np.concatenate([p.log_pot, rng.standard_normal(16).astype(np.float32)])
    _same(gpu, p, 1.0, 5, fused=False)
