"""Calls on a stream confined to a part of the device's SMs (a green context's), where a launch of one
block per SM of the device is refused: the forms without such a launch, bitwise as ever."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2202_04110_gb300 import workloads as W

pytestmark = pytest.mark.gpu

GREEN = r"""
#include <cuda.h>
extern "C" int green_stream(int device, int min_sms, void **stream, int *sms) {
    CUdevice dev;
    CUdevResource all, part;
    CUdevResourceDesc desc;
    CUgreenCtx ctx;
    unsigned n = 1;
    CUresult r = cuDeviceGet(&dev, device);
    if (r == CUDA_SUCCESS) r = cuDeviceGetDevResource(dev, &all, CU_DEV_RESOURCE_TYPE_SM);
    if (r == CUDA_SUCCESS) r = cuDevSmResourceSplitByCount(&part, &n, &all, nullptr, 0, (unsigned)min_sms);
    if (r == CUDA_SUCCESS) r = cuDevResourceGenerateDesc(&desc, &part, 1);
    if (r == CUDA_SUCCESS) r = cuGreenCtxCreate(&ctx, desc, dev, CU_GREEN_CTX_DEFAULT_STREAM);
    CUstream s = nullptr;
    if (r == CUDA_SUCCESS) r = cuGreenCtxStreamCreate(&s, ctx, CU_STREAM_NON_BLOCKING, 0);
    *stream = s;
    *sms = r == CUDA_SUCCESS ? (int)part.sm.smCount : 0;
    return (int)r;
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
def stream(gpu, tmp_path_factory):
    import torch
    from paper_2202_04110_gb300 import build
    torch.zeros(1, device="cuda")  # the device's primary context
    d = tmp_path_factory.mktemp("green")
    (d / "green.cu").write_text(GREEN)
    so = str(d / "green.so")
    subprocess.run([build.nvcc_path(), *build.ARCH, "-shared", "-Xcompiler", "-fPIC", "-o", so, str(d / "green.cu"), "-lcuda"], check=True)
    s, sms = ctypes.c_void_p(), ctypes.c_int()
    r = ctypes.CDLL(so).green_stream(torch.cuda.current_device(), 32, ctypes.byref(s), ctypes.byref(sms))
    if r != 0:
        pytest.skip(f"no green context here (CUresult {r})")
    assert 32 <= sms.value < torch.cuda.get_device_properties(0).multi_processor_count
    return torch.cuda.ExternalStream(s.value)


def _inputs(gpu, shape):
    import torch
    p = W.ising_grid(*shape, seed=shape[0])
    g = gpu.Graph(p.graph)
    g.set_option(gpu.OPT_WAIT_POLLS, 20000)  # (a launch that is not refused gives up soon)
    return p, g, torch.as_tensor(p.log_pot).cuda(), torch.as_tensor(p.evidence).cuda()


@pytest.mark.parametrize("shape", [(110, 120), (317, 241), (700, 700)])
def test_run(gpu, stream, shape):
    import torch
    p, g, lp, ev = _inputs(gpu, shape)
    want = g.run_bp(lp, ev, 1.0, 0.5, 30, g.new_msgs())
    assert g.flags(clear=True) == 0
    for _ in range(2):
        m = g.new_msgs()
        torch.cuda.synchronize()
        g.run_bp(lp, ev, 1.0, 0.5, 30, m, stream=stream)
        stream.synchronize()
        assert torch.equal(m, want) and g.flags(clear=True, stream=stream) == 0


def test_host_call(gpu, stream):
    p, g, lp, ev = _inputs(gpu, (317, 241))
    want = g.infer_host(p.log_pot, p.evidence, 1.0, 0.5, 30)[0].copy()
    assert np.array_equal(g.infer_host(p.log_pot, p.evidence, 1.0, 0.5, 30, stream=stream)[0], want)


@pytest.mark.parametrize("shape,S", [((97, 101), 9), ((317, 241), 2)])
def test_samples(gpu, stream, shape, S):
    import torch
    p, g, lp, ev = _inputs(gpu, shape)
    evs = torch.stack([ev * (1 + 0.1 * s) for s in range(S)])
    want = g.run_bp_multi(lp, evs, 1.0, 0.5, 20, torch.zeros(S, g.info["n_edge_states"], device="cuda"))
    m = torch.zeros_like(want)
    torch.cuda.synchronize()
    g.run_bp_multi(lp, evs, 1.0, 0.5, 20, m, stream=stream)
    stream.synchronize()
    assert torch.equal(m, want) and g.flags(clear=True, stream=stream) == 0


def test_gradient(gpu, stream):
    import torch
    p, g, lp, ev = _inputs(gpu, (120, 130))
    cot = torch.ones_like(ev)
    want = g.grad(lp, ev, 1.0, 0.5, 12, 4, cot)
    torch.cuda.synchronize()
    got = g.grad(lp, ev, 1.0, 0.5, 12, 4, cot, stream=stream)
    stream.synchronize()
    for a, b in zip(got, want):
        assert torch.max(torch.abs(a - b)) <= 1e-4 * max(1.0, float(torch.max(torch.abs(b))))
