"""Runs of binary graphs with high-degree variables in edge-order log-ratios, held to the
edge-state iteration (PGM_OPT_LOG_RATIO 0), whose results the other tests hold to the oracle.
Both are FP32 runs within ATOL + RTOL |b| of the FP64 result in the normalised log-beliefs (the
repository's criterion), so within twice that of each other; -inf entries and flags are equal."""
import numpy as np
import pytest

from paper_2202_04110_gb300 import workloads as W
from paper_2202_04110_gb300.workloads import EnumGroup, FactorGraph, LogicGroup
from tests._parity import ATOL, RTOL, assert_beliefs_close
from tests.test_gpu_small_run import _hard

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


def _run(binding, p, T, damping, n_iters, lr_min, m0=None, shift=0, cuda_graph=1):
    import torch
    g = binding.Graph(p.graph)
    g.set_option(binding.OPT_LOG_RATIO, lr_min)
    g.set_option(binding.OPT_CUDA_GRAPH, cuda_graph)
    lp = torch.as_tensor(np.asarray(p.log_pot, np.float32)).cuda()
    ev = torch.as_tensor(np.asarray(p.evidence, np.float32)).cuda()
    start = torch.zeros(p.graph.n_edge_states) if m0 is None else torch.as_tensor(m0)
    m = torch.zeros(p.graph.n_edge_states + shift, device="cuda")[shift:]  # shift: pointer alignment
    for _ in range(2):  # the second call replays the recorded run
        m.copy_(start)
        g.run_bp(lp, ev, T, damping, n_iters, m)
    mm = m.clone()
    return mm.cpu().numpy(), g.beliefs(ev, mm, True).cpu().numpy(), g.flags(clear=True)


def _close(binding, p, T, damping, n_iters, **kw):
    ms, bs, fs = _run(binding, p, T, damping, n_iters, 0, kw.get("m0"))
    me, be, fe = _run(binding, p, T, damping, n_iters, 1, **kw)
    assert fs == fe, (fs, fe)
    assert (np.isneginf(ms) == np.isneginf(me)).all() and (np.isnan(ms) == np.isnan(me)).all()
    assert (np.fmax.reduce(me.reshape(-1, 2), axis=1) == 0).all()  # max-normalised
    assert (np.isnan(bs) == np.isnan(be)).all()  # (contradictory hard constraints)
    fin = ~np.isnan(bs)
    assert_beliefs_close(be[fin], bs[fin], atol=2 * ATOL, rtol=2 * RTOL, what=p.name)


@pytest.mark.parametrize("shape", [(65, 1), (1, 65), (67, 71), (3, 1023), (3, 1024), (3, 1025), (2, 4096), (2, 4097),
                                   (100, 150), (784, 500)])
@pytest.mark.parametrize("T", [1.0, 0.4, 0.0])
def test_sizes(gpu, shape, T):
    """Odd numbers of factors, low-degree variables beside the high ones, one and several rounds
    of a block's edges, and one factor more than the form takes."""
    p = W.rbm(*shape, seed=shape[1])
    for it in (1, 2, 9):
        _close(gpu, p, T, 0.5, it)


@pytest.mark.parametrize("T", [1.0, 0.0])
@pytest.mark.parametrize("shift", [0, 2])
def test_hard_inputs(gpu, T, shift):
    """Clamped and contradictory variables, tables with -inf entries, warm starts with -inf and
    doubly -inf messages, damping 0, messages aligned to 16 and 8 bytes."""
    p = W.rbm(70, 81, seed=4)
    rng = np.random.default_rng(6)
    pot = p.log_pot.reshape(-1, 4).copy()
    hit = np.flatnonzero(rng.random(pot.shape[0]) < 0.002)
    pot[hit, rng.integers(0, 4, hit.size)] = -np.inf
    p.log_pot = pot.ravel()
    p.evidence = _hard(p.evidence, 0.05, 5)
    _close(gpu, p, T, 0.5, 6, shift=shift)
    _close(gpu, p, T, 0.0, 7, shift=shift, cuda_graph=0)
    m0 = np.zeros((p.graph.n_edges, 2), np.float32)
    m0[:, 0] = -np.abs(rng.standard_normal(len(m0)))
    m0[rng.random(len(m0)) < 0.003, 1] = -np.inf
    _close(gpu, p, T, 0.3, 5, m0=m0.ravel(), shift=shift)
    m0[7] = -np.inf
    _close(gpu, p, T, 0.3, 5, m0=m0.ravel(), shift=shift)
    p.evidence = _hard(p.evidence, 0.05, 5, both=True)
    _close(gpu, p, T, 0.5, 6, shift=shift)


def test_groups(gpu):
    """Several groups (a factor pair across two of them), shared and own tables, a hub over a chain."""
    rng = np.random.default_rng(2)
    n = 301
    cfg = W.rbm(1, 1, 0).graph.enum_groups[0].cfg
    hub = np.stack([np.zeros(n - 1), np.arange(1, n)], 1).astype(np.int32)
    chain = np.stack([np.arange(1, n - 1), np.arange(2, n)], 1).astype(np.int32)
    g = FactorGraph(np.full(n, 2, np.int32), [EnumGroup(cfg.copy(), chain[:151], False),
                                              EnumGroup(cfg.copy(), hub, True),
                                              EnumGroup(cfg.copy(), chain[151:], False)], [])
    p = W.Problem("hub over a chain", g, (0.3 * rng.standard_normal(g.n_potentials)).astype(np.float32),
                  rng.standard_normal(2 * n).astype(np.float32), 1.0, 0.5, 10)
    for T in (1.0, 0.0):
        _close(gpu, p, T, 0.5, 11)


def _logic(fans, kind, n_vars, hubs, seed, extra=0):
    """OR / AND factors of the given fan-ins over n_vars variables; the first `hubs` variables are
    parents of every factor in turn (variable 0 of `extra` more factors of fan-in 1)."""
    rng = np.random.default_rng(seed)
    fans = list(fans) + [1] * extra
    par, child = [], []
    for i, n in enumerate(fans):
        v = rng.choice(np.arange(hubs, n_vars), n + 1, replace=False)
        v[0] = 0 if n == 1 else i % hubs
        par.append(v[:n])
        child.append(v[n])
    off = np.concatenate([[0], np.cumsum(fans)]).astype(np.int32)
    return LogicGroup(kind, off, np.concatenate(par).astype(np.int32), np.array(child, np.int32))


@pytest.mark.parametrize("fans", [(1, 2), (1, 2, 3, 4), (5, 31, 32, 33, 64), (65, 127, 128), (129, 192), (193, 256), (257,)])
@pytest.mark.parametrize("kind", ["or", "and"])
@pytest.mark.parametrize("extra", [0, 4200])
def test_logic(gpu, fans, kind, extra):
    """Max-product over OR / AND factors at every kernel's edges of fan-in (257: the edge-state
    form), with hubs of 70 and of more than 4,096 factors; also clamped variables."""
    n = 400
    reps = 210 // len(fans) + 1
    k = W.OR if kind == "or" else W.AND
    g = FactorGraph(np.full(n, 2, np.int32), [],
                    [_logic(list(fans) * reps, k, n, 3, len(fans), extra), _logic([2] * 37, k, n, 1, 5)])
    rng = np.random.default_rng(fans[0])
    p = W.Problem(f"{kind} {fans}", g, np.zeros(0, np.float32), rng.standard_normal(2 * n).astype(np.float32), 0.0, 0.5, 6)
    for it in (1, 6):
        _close(gpu, p, 0.0, 0.5, it)
    _close(gpu, p, 0.0, 0.0, 4, cuda_graph=0, shift=2)
    p.evidence = _hard(p.evidence, 0.02, 7)
    _close(gpu, p, 0.0, 0.5, 5)
    m0 = np.zeros((g.n_edges, 2), np.float32)
    m0[:, 1] = -np.abs(rng.standard_normal(len(m0)))
    m0[rng.random(len(m0)) < 0.002, 0] = -np.inf
    _close(gpu, p, 0.0, 0.3, 3, m0=m0.ravel())


def test_deconvolution_images(gpu):
    """AND and OR launches of one graph, weights of degree above 4,096 in blocks of 1024."""
    for n_img in (1, 3, 50):
        _close(gpu, W.deconvolution(4, n_img=n_img, n_iters=10), 0.0, 0.5, 10)
