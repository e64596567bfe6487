"""Runs take their log-potentials after the work that precedes them on the stream: a kernel of the
caller that lets its dependents start at once and writes the table much later must have written it
before the run's first launch reads it."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2202_04110_gb300 import workloads as W

pytestmark = pytest.mark.gpu

LATE_COPY = r"""
#include <cuda_runtime.h>
__global__ void late_copy(float *dst, const float *src, int n, int us) {
    asm volatile("griddepcontrol.launch_dependents;");
    for (int i = 0; i < us; ++i) __nanosleep(1000);
    for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}
extern "C" int run_late_copy(float *dst, const float *src, int n, int us, void *stream) {
    late_copy<<<1, 256, 0, static_cast<cudaStream_t>(stream)>>>(dst, src, n, us);
    return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2202_04110_gb300 import build
    build.build()
    from paper_2202_04110_gb300 import binding
    return binding


@pytest.fixture(scope="module")
def late_copy(tmp_path_factory):
    from paper_2202_04110_gb300 import build
    d = tmp_path_factory.mktemp("late_copy")
    (d / "late_copy.cu").write_text(LATE_COPY)
    so = str(d / "late_copy.so")
    subprocess.run([build.nvcc_path(), *build.ARCH, "-shared", "-Xcompiler", "-fPIC", "-o", so, str(d / "late_copy.cu")], check=True)
    return ctypes.CDLL(so).run_late_copy


S = 3


def _calls(gpu, g, lp, ev, p, n_iters):
    """The calls whose first launch may be the factor kernel, name -> (prepare, call): everything that
    touches the stream besides the call itself is in prepare."""
    import torch
    n = g.info["n_edge_states"]
    m, ms, evs, cot = torch.zeros(n, device="cuda"), torch.zeros(S, n, device="cuda"), ev.repeat(S, 1), torch.ones_like(ev)

    def direct(on):
        g.set_option(gpu.OPT_CUDA_GRAPH, on)
        m.zero_()

    return {"multi": (ms.zero_, lambda: g.run_bp_multi(lp, evs, p.T, 0.5, n_iters, ms)),
            "direct": (lambda: direct(0), lambda: g.run_bp(lp, ev, p.T, 0.5, n_iters, m)),
            "recorded": (lambda: direct(1), lambda: g.run_bp(lp, ev, p.T, 0.5, n_iters, m)),
            "batch": (m.zero_, lambda: g.run_bp_batch(lp, ev, [p.T], [0.5], [n_iters], m)),
            "gradient": (m.zero_, lambda: g.grad(lp, ev, 1.0, 0.5, n_iters, 2, cot)[0])}


@pytest.mark.parametrize("K", [4, 8, 16])
@pytest.mark.parametrize("T", [1.0, 0.0])
@pytest.mark.parametrize("n_iters", [1, 2])
def test_table_written_right_before_the_run(gpu, late_copy, K, T, n_iters):
    import torch
    p = W.potts_grid(24, K, seed=K, T=T)
    g = gpu.Graph(p.graph)
    ev = torch.as_tensor(p.evidence).cuda()
    new = torch.as_tensor(p.log_pot).cuda()
    stale = torch.as_tensor(np.random.default_rng(K).standard_normal(p.log_pot.size).astype(np.float32)).cuda()
    want = {}
    for name, (prepare, call) in _calls(gpu, g, new, ev, p, n_iters).items():
        prepare()
        want[name] = call().clone()
    lp = stale.clone()
    for name, (prepare, call) in _calls(gpu, g, lp, ev, p, n_iters).items():
        prepare()
        call()  # (everything allocated and recorded)
        prepare()
        lp.copy_(stale)
        torch.cuda.synchronize()
        stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
        assert late_copy(ctypes.c_void_p(lp.data_ptr()), ctypes.c_void_p(new.data_ptr()), lp.numel(), 300, stream) == 0
        got = call()
        torch.cuda.synchronize()
        assert torch.equal(got, want[name]), name
