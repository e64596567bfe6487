"""One-launch runs whose waits run out (PGM_OPT_WAIT_POLLS 0; with 1 a block looks once for another's
value, which may be there): the kernel ends, PGM_FLAG_TIMEOUT is raised, calls that return results to the host fail, the
gradient comes from the launches, and the next run of the graph with an ordinary limit is the
multi-launch run's bits. The flag also shows that a shape takes a form of several blocks at all."""
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


def _graph(gpu, shape):
    import torch
    p = W.ising_grid(*shape, seed=shape[0])
    return p, gpu.Graph(p.graph), torch.as_tensor(p.log_pot).cuda(), torch.as_tensor(p.evidence).cuda()


def _run(g, lp, ev, n=40):
    m = g.new_msgs()
    g.run_bp(lp, ev, 1.0, 0.5, n, m)
    return m


# a cluster; the grid with records in shared memory, streamed with every slot's value, with totals
CLUSTER, GRID = [(30, 30), (90, 99)], [(120, 130), (317, 241), (700, 700), (1100, 1101)]


@pytest.mark.parametrize("shape", CLUSTER + GRID)
def test_run(gpu, shape):
    import torch
    p, g, lp, ev = _graph(gpu, shape)
    g.set_option(gpu.OPT_SMALL_RUN, 0)
    want = _run(g, lp, ev)
    g.set_option(gpu.OPT_SMALL_RUN, 1)
    for polls in (0, 1, 0):
        g.set_option(gpu.OPT_WAIT_POLLS, polls)
        _run(g, lp, ev)
        assert g.flags(clear=True) & gpu.FLAG_TIMEOUT or polls == 1
        g.set_option(gpu.OPT_WAIT_POLLS, 1 << 22)
        assert torch.equal(_run(g, lp, ev), want)
        assert g.flags(clear=True) == 0


@pytest.mark.parametrize("shape", [(10, 10), (24, 24)])
def test_no_waits(gpu, shape):
    """One block waits for nobody (setting 1), a cluster does (setting 2)."""
    p, g, lp, ev = _graph(gpu, shape)
    g.set_option(gpu.OPT_WAIT_POLLS, 0)
    _run(g, lp, ev)
    f1 = g.flags(clear=True)
    g.set_option(gpu.OPT_SMALL_RUN, 2)
    _run(g, lp, ev)
    assert bool(f1 & gpu.FLAG_TIMEOUT) == (shape[0] > 10) and g.flags(clear=True) & gpu.FLAG_TIMEOUT


def test_samples(gpu):
    import torch
    p, g, lp, ev = _graph(gpu, (97, 101))
    evs = torch.stack([ev * (1 + 0.1 * s) for s in range(9)])

    def run():
        return g.run_bp_multi(lp, evs, 1.0, 0.5, 20, torch.zeros(9, g.info["n_edge_states"], device="cuda"))

    want = run()
    assert g.flags(clear=True) == 0
    g.set_option(gpu.OPT_WAIT_POLLS, 0)
    run()
    assert g.flags(clear=True) & gpu.FLAG_TIMEOUT
    g.set_option(gpu.OPT_WAIT_POLLS, 1 << 22)
    assert torch.equal(run(), want) and g.flags(clear=True) == 0


@pytest.mark.parametrize("shape", [(90, 99), (120, 130)])
def test_host_call_and_early_exit_fail(gpu, shape):
    p, g, lp, ev = _graph(gpu, shape)
    want = g.infer_host(p.log_pot, p.evidence, 1.0, 0.5, 40)[0].copy()
    g.set_option(gpu.OPT_WAIT_POLLS, 0)
    with pytest.raises(gpu.PgmError) as ei:
        g.infer_host(p.log_pot, p.evidence, 1.0, 0.5, 40)
    assert ei.value.status == -3 and "TIMEOUT" in str(ei.value)
    if shape in CLUSTER:  # early-exit runs take the cluster form only
        with pytest.raises(gpu.PgmError):
            g.run_bp_until(lp, ev, 1.0, 0.5, 40, 0.0, 20, g.new_msgs())
    g.set_option(gpu.OPT_WAIT_POLLS, 1 << 22)
    assert np.array_equal(g.infer_host(p.log_pot, p.evidence, 1.0, 0.5, 40)[0], want)
    assert g.run_bp_until(lp, ev, 1.0, 0.5, 40, 0.0, 20, g.new_msgs())[0] == 40


@pytest.mark.parametrize("shape", [(64, 64), (120, 130)])
def test_gradient_takes_the_launches(gpu, shape):
    import torch
    p, g, lp, ev = _graph(gpu, shape)
    cot = torch.as_tensor(np.random.default_rng(1).standard_normal(p.evidence.size).astype(np.float32)).cuda()
    one = g.grad(lp, ev, 1.0, 0.5, 30, 7, cot)
    g.set_option(gpu.OPT_WAIT_POLLS, 0)
    got = g.grad(lp, ev, 1.0, 0.5, 30, 7, cot)
    assert g.flags(clear=True) == 0
    g.set_option(gpu.OPT_SMALL_RUN, 0)
    want = g.grad(lp, ev, 1.0, 0.5, 30, 7, cot)
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    assert not torch.equal(one[0], want[0])  # (the one launch rounds differently: it did run)
