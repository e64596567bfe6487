"""A gradient whose one-launch history does not fit the device's free memory: the launches, and the
same call again neither asks for that memory nor waits for other streams; once there is room, the one
launch. (Takes most of the device's memory for a moment.)"""
import time

import numpy as np
import pytest

from paper_2202_04110_gb300 import workloads as W

pytestmark = pytest.mark.gpu

LEAVE = 200 << 20  # below the history of 600 iterations on 40,000 variables (385 MB), above the launches' 50 MB


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_04110_gb300 import build
    build.build()
    from paper_2202_04110_gb300 import binding
    return binding


def test_no_room_for_the_history(gpu):
    import torch
    p = W.ising_grid(200, 200, seed=1)
    lp, ev = torch.as_tensor(p.log_pot).cuda(), torch.as_tensor(p.evidence).cuda()
    cot = torch.as_tensor(np.random.default_rng(2).standard_normal(p.evidence.size).astype(np.float32)).cuda()

    def grad(g):
        return [t.clone() for t in g.grad(lp, ev, 1.0, 0.5, 600, 30, cot)]

    one = grad(gpu.Graph(p.graph))
    g = gpu.Graph(p.graph)
    g.set_option(gpu.OPT_SMALL_RUN, 0)
    launches = grad(g)
    assert not torch.equal(one[0], launches[0])
    g = gpu.Graph(p.graph)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    if free < 4 * LEAVE:
        pytest.skip("the device's memory is in use")
    fill = torch.empty(free - LEAVE, dtype=torch.uint8, device="cuda")
    try:
        for _ in range(2):
            assert all(torch.equal(a, b) for a, b in zip(grad(g), launches))
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            torch.cuda._sleep(2_000_000_000)  # about a second
        t0 = time.perf_counter()
        out = g.grad(lp, ev, 1.0, 0.5, 600, 30, cot)
        spent = time.perf_counter() - t0
        assert not side.query() and spent < 0.4, spent
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(out, launches))
    finally:
        del fill
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
    assert all(torch.equal(a, b) for a, b in zip(grad(g), one))


def test_history_limit(gpu):
    """512 MiB of kept values (16 bytes per variable, 152 blocks of 264, and iteration): the one launch up
    to there, whose bits differ from the launches', the launches above."""
    import torch
    p = W.ising_grid(200, 200, seed=1)
    lp, ev = torch.as_tensor(p.log_pot).cuda(), torch.as_tensor(p.evidence).cuda()
    cot = torch.as_tensor(np.random.default_rng(2).standard_normal(p.evidence.size).astype(np.float32)).cuda()
    at_most = (512 << 20) // (152 * 264 * 16)
    for n, same in ((at_most, False), (at_most + 1, True)):
        out = []
        for small in (1, 0):
            g = gpu.Graph(p.graph)
            g.set_option(gpu.OPT_SMALL_RUN, small)
            out.append(g.grad(lp, ev, 1.0, 0.5, n, 30, cot)[0])
        assert torch.equal(*out) == same, n
