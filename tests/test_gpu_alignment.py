"""Arrays that start at an odd multiple of 4 bytes where a call takes them: the same bits as from an
aligned copy. (Contiguous views of larger tensors, as autograd hands them over.)"""
import numpy as np
import pytest

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


def _shifted(a):
    import torch
    buf = torch.empty(a.size + 1, device="cuda")
    assert buf.data_ptr() % 8 == 0
    v = buf[1:].view(a.shape)
    v.copy_(torch.as_tensor(a))
    return v


# one block, a cluster, the grid; the launches (a table of -inf hands the call to them)
@pytest.mark.parametrize("shape,hard", [((9, 11), False), ((64, 64), False), ((120, 130), False), ((64, 64), True)])
def test_cotangent(gpu, shape, hard):
    import torch
    p = W.ising_grid(*shape, seed=3)
    if hard:
        p.log_pot[5] = -np.inf
    cot = np.random.default_rng(4).standard_normal(p.evidence.size).astype(np.float32)
    g = gpu.Graph(p.graph)
    lp, ev = torch.as_tensor(p.log_pot).cuda(), torch.as_tensor(p.evidence).cuda()
    want = g.grad(lp, ev, 1.0, 0.5, 8, 4, torch.as_tensor(cot).cuda())
    got = g.grad(lp, ev, 1.0, 0.5, 8, 4, _shifted(cot))
    for a, b in zip(got, want):
        assert torch.equal(a.nan_to_num(7.0), b.nan_to_num(7.0))


def test_backward_through_a_concatenation(gpu):
    """The cotangent of torch.cat([one value, beliefs]) is a view at an odd offset."""
    import torch
    p = W.ising_grid(30, 31, seed=5)
    g = gpu.Graph(p.graph)
    w = torch.as_tensor(np.random.default_rng(6).standard_normal(1 + p.evidence.size).astype(np.float32)).cuda()
    grads = []
    for cat in (False, True):
        lp = torch.as_tensor(p.log_pot).cuda().requires_grad_(True)
        ev = torch.as_tensor(p.evidence).cuda().requires_grad_(True)
        nb = gpu.lbp_beliefs(lp, ev, g, 1.0, 0.5, 8, 4)
        out = torch.cat([torch.zeros(1, device="cuda"), nb]) @ w if cat else nb @ w[1:].clone()
        grads.append(torch.autograd.grad(out, (lp, ev)))
    for a, b in zip(*grads):
        assert torch.equal(a, b)


@pytest.mark.parametrize("rows,cols,S", [(10, 10, 5), (20, 21, 9), (40, 41, 4), (90, 100, 3)])
@pytest.mark.parametrize("per_sample", [False, True])
def test_samples(gpu, rows, cols, S, per_sample):
    """Evidence, log-potentials and messages of many samples."""
    import torch
    p = W.ising_grid(rows, cols, seed=7)
    rng = np.random.default_rng(8)
    ev = rng.standard_normal((S, p.evidence.size)).astype(np.float32)
    lp = np.stack([p.log_pot * (1 + s) for s in range(S)]).astype(np.float32) if per_sample else p.log_pot
    m0 = -np.abs(rng.standard_normal((S, p.graph.n_edge_states))).astype(np.float32)
    g = gpu.Graph(p.graph)
    on = [torch.as_tensor(a).cuda() for a in (lp, ev, m0)]
    want = g.run_bp_multi(on[0], on[1], 1.0, 0.5, 9, on[2].clone())
    for which in ((1,), (0, 2), (0, 1, 2)):
        a = [_shifted(h) if i in which else torch.as_tensor(h).cuda() for i, h in enumerate((lp, ev, m0))]
        assert torch.equal(g.run_bp_multi(a[0], a[1], 1.0, 0.5, 9, a[2]), want), which
