"""The max-product form of shared pairwise configuration lists that takes four factors per
warp (k_enum_pairs), held bitwise to the thread-per-factor form on groups that both take and
stepwise to the oracle on larger state counts, at its edges: fewer than four factors in the last
warp and block, different state counts of the two neighbours, hard evidence, high-degree
variables, samples, two groups."""
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


def _lists(n_fac, Ka, Kb, n_cfg, seed, hub=False):
    """n_fac factors between random variables of Ka and Kb states over one random list."""
    rng = np.random.default_rng(seed)
    na, nb = (1 if hub else n_fac // 2 + 1), n_fac // 2 + 1
    codes = np.sort(rng.choice(Ka * Kb, size=min(n_cfg, Ka * Kb), replace=False))
    cfg = np.stack([codes // Kb, codes % Kb], 1).astype(np.int32)
    pairs = np.stack([rng.integers(0, na, n_fac), na + rng.permutation(n_fac) % nb], 1).astype(np.int32)
    g = W.FactorGraph(np.concatenate([np.full(na, Ka), np.full(nb, Kb)]).astype(np.int32), [W.EnumGroup(cfg, pairs, True)], [])
    pot = rng.standard_normal(cfg.shape[0]).astype(np.float32)
    return g, pot, rng.standard_normal(na * Ka + nb * Kb).astype(np.float32)


def _run(gpu, g, pot, ev, n_iters, damping, block):
    import torch
    G = gpu.Graph(g)
    G.set_option(gpu.OPT_ENUM_BLOCK, block)
    m = G.new_msgs()
    G.run_bp(torch.as_tensor(pot).cuda(), torch.as_tensor(ev).cuda(), 0.0, damping, n_iters, m)
    return m.cpu().numpy(), G.flags(clear=True)


@pytest.mark.parametrize("n_fac,Ka,Kb,n_cfg", [(4864, 7, 7, 30), (4865, 5, 9, 40), (4867, 33, 31, 200), (5001, 3, 60, 90)])
@pytest.mark.parametrize("damping", [0.5, 0.0])
def test_equals_the_thread_form(gpu, n_fac, Ka, Kb, n_cfg, damping):
    """(a list of at most 256 configurations and a state sum of at most 64: both forms run)"""
    g, pot, ev = _lists(n_fac, Ka, Kb, n_cfg, n_fac)
    ev[::37] = -np.inf
    for it in (1, 6):
        a, fa = _run(gpu, g, pot, ev, it, damping, 1)
        b, fb = _run(gpu, g, pot, ev, it, damping, 0)
        assert np.array_equal(a, b, equal_nan=True), np.nanmax(np.abs(a - b))
        assert fa == fb


@pytest.mark.parametrize("n_fac,Ka,Kb,n_cfg,hub", [(4900, 49, 49, 361, False), (4866, 130, 126, 900, False), (5000, 17, 40, 300, True)])
def test_one_step_of_the_oracle(gpu, n_fac, Ka, Kb, n_cfg, hub):
    g, pot, ev = _lists(n_fac, Ka, Kb, n_cfg, 3, hub)
    import torch
    G = gpu.Graph(g)
    lp, evt, m = torch.as_tensor(pot).cuda(), torch.as_tensor(ev).cuda(), G.new_msgs()
    for done in (0, 3):
        G.run_bp(lp, evt, 0.0, 0.5, done, m)
        m0 = m.cpu().numpy().astype(np.float64)
        G.run_bp(lp, evt, 0.0, 0.5, 1, m)
        want, _ = oracle.run_bp(g, pot, ev, 0.0, 0.5, 1, msgs=m0)
        got = m.cpu().numpy()
        assert np.all(np.abs(got - want) <= 1e-4 + 1e-6 * np.abs(want))


def test_samples(gpu):
    """Many samples at once equal the single runs."""
    import torch
    g, pot, ev = _lists(4870, 20, 30, 150, 5)
    evs = np.random.default_rng(6).standard_normal((3, ev.size)).astype(np.float32)
    G = gpu.Graph(g)
    m = torch.zeros(3, g.n_edge_states, device="cuda")
    G.run_bp_multi(torch.as_tensor(pot).cuda(), torch.as_tensor(evs).cuda(), 0.0, 0.5, 4, m)
    for s in range(3):
        assert np.array_equal(m[s].cpu().numpy(), _run(gpu, g, pot, evs[s], 4, 0.5, 1)[0])
