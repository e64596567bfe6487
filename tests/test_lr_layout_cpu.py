"""The one-launch runs' own sizing functions (csrc/lr_layout.h), compiled for the host: the layouts that
the kernels walk fit what is asked for, what is asked for fits a block at every size the forms are
taken at, every item has a thread, and samples share a launch within the device."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2202_04110_gb300 import workloads as W
from tests.test_lr_run_cpu import random_numbering

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2202_04110_gb300", "csrc")
ALONE, CLUSTER, GRID = 0, 1, 2
SMS, SMEM, SMALL_V, SMALL_F, BLOCK_V, CLUSTER_V = 152, 232448 - 256, 1024, 2048, 700, 9000

WRAP = r"""
#include "lr_layout.h"
using namespace pgm;
extern "C" {
long constants(int i) {
    const long c[] = {kPlanSms, kPlanSmem, kLrSmallMaxV, kLrSmallMaxF, kLrBlockAutoV, kLrClusterAutoV};
    return c[i];
}
long c_run_smem(int x, int res, int lam, int Vc, int f, int h) { return (long)run_smem(x, res, lam, Vc, f, h); }
long c_grad_smem(int x, int Vc, int f, int h) { return (long)grad_smem(x, Vc, f, h); }
long c_lam_max(long slots) { return (long)lam_floats_max(slots); }
int c_run_threads(int Vc, int items) { return run_threads(Vc, items); }
int c_grid_blocks(int V, int n_sm, int smem) { return lr_grid_blocks(V, n_sm, smem); }
void c_push(int V, int E, long *o) {
    const PushShape p = push_shape(V, E);
    o[0] = p.edges, o[1] = p.threads, o[2] = p.two, o[3] = (long)p.smem;
}
void c_multi(int V, int S, int local, long *o) {
    const LrMultiPlan p = lr_multi_plan(V, S, local, kPlanSms, kPlanSmem, true);
    o[0] = p.S, o[1] = p.nb, o[2] = p.Vc, o[3] = p.f_cap, o[4] = p.h_cap, o[5] = p.res, o[6] = (long)p.sample_bytes;
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("lr_layout")
    (d / "wrap.cpp").write_text(WRAP)
    so = str(d / "wrap.so")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", so, str(d / "wrap.cpp")], check=True)
    lib = ctypes.CDLL(so)
    for f in ("constants", "c_run_smem", "c_grad_smem", "c_lam_max"):
        getattr(lib, f).restype = ctypes.c_long
    return lib


def _out(f, n, *args):
    o = (ctypes.c_long * n)()
    f(*args, o)
    return list(o)


def _walk(parts):
    """Offsets of (element bytes, count) arrays laid one after the other: each at a multiple of its
    element; the end."""
    at = 0
    for size, n in parts:
        assert at % size == 0, parts
        at += size * n
    return at


def _run_parts(x, res, lam, Vc, f, h):
    """k_lr_run's shared memory in its order: records, lam or totals, evidence, inbox, d, addresses."""
    return (([(16, f), (16, h)] if res else []) + [(4, 4 * Vc) if lam else (8, Vc)] + ([(8, Vc)] if res else [])
            + ([(8, 2 * h)] if x == CLUSTER else []) + [(4, 4 * Vc)] + ([(4, h)] if res else []))


def _grad_parts(x, Vc, f, h):
    """k_lr_grad's: records, their gradients, evidence, inbox, lam, d, the evidence's gradient, addresses."""
    return ([(16, f), (16, h), (16, f), (16, h), (8, Vc)] + ([(8, 2 * h)] if x == CLUSTER else [])
            + [(4, 4 * Vc), (4, 4 * Vc), (4, Vc), (4, h)])


def test_constants(lib):
    assert [lib.constants(i) for i in range(6)] == [SMS, SMEM, SMALL_V, SMALL_F, BLOCK_V, CLUSTER_V]


@pytest.mark.parametrize("Vc", [1, 2, 57, 256, 1023, 1024, 1705, 7255, 9674])
def test_layouts_fit_what_is_asked_for(lib, Vc):
    for f, h in ((0, 0), (2 * Vc, 4 * Vc), (2 * Vc - 1, 1), (1, 4 * Vc - 3)):
        for x, res, lam in ((ALONE, 1, 1), (ALONE, 0, 1), (ALONE, 0, 0), (CLUSTER, 1, 1), (GRID, 1, 1), (GRID, 0, 1), (GRID, 0, 0)):
            need = _walk(_run_parts(x, res, lam, Vc, f, h))
            assert need <= lib.c_run_smem(x, res, lam, Vc, f, h) <= need + 16
        for x in (ALONE, CLUSTER, GRID):
            need = _walk(_grad_parts(x, Vc, f, 0 if x == ALONE else h))
            assert need <= lib.c_grad_smem(x, Vc, f, 0 if x == ALONE else h) <= need + 16


@pytest.mark.parametrize("C", [8, 16])
def test_cluster_worst_case_fits(lib, C):
    for V in (1, 2, 701, 1025, 4096, 8999, C * SMALL_V - 1, C * SMALL_V):
        Vc = -(-V // C)
        if V > C * SMALL_V:
            continue
        assert lib.c_run_smem(CLUSTER, 1, 1, Vc, 2 * Vc, 4 * Vc) <= SMEM and 4 * Vc <= 1 << 16
        for graph in (W.ising_grid(1, V, 0).graph, random_numbering(1, V, 2).graph) if V > 1 else ():
            blk = graph.enum_groups[0].vars.astype(np.int64) // Vc
            whole = blk[:, 0] == blk[:, 1]
            assert np.bincount(blk[whole, 0], minlength=C).max() <= 2 * Vc
            assert np.bincount(blk[~whole].ravel(), minlength=C).max() <= 4 * Vc


@pytest.mark.parametrize("V", [701, 1000, 9001, 38912, 76397, 250000, 1000000, 1102760, 1102761, 1200090, 1450800, 1470448, 1480000])
def test_grid_blocks(lib, V):
    nb = lib.c_grid_blocks(V, SMS, SMEM)
    if V > 1470448:  # 9,674 variables a block at 24 bytes
        assert nb == 0
        return
    Vc = -(-V // nb)
    assert 2 <= nb <= SMS and nb * Vc >= V and 4 * Vc <= 1 << 16  # (slots are 16 bits)
    assert lib.c_run_smem(GRID, 0, 0, Vc, 0, 0) <= SMEM
    # explicit sums: a last block's of fewer variables end inside the scratch
    last = V - (nb - 1) * Vc
    assert 4 * (nb - 1) * Vc + 3 * Vc + max(last, 1) <= lib.c_lam_max(ctypes.c_long(4 * V))
    assert (lib.c_run_smem(GRID, 0, 1, Vc, 0, 0) <= SMEM) == (V <= 1102760)  # lam per slot: 7,255 a block
    for f in (1, Vc, 2 * Vc):
        t = lib.c_run_threads(Vc, f)
        assert t % 32 == 0 and t == min(1024, max(32, -(-max(Vc, f) // 32) * 32))


@pytest.mark.parametrize("V,E", [(1, 2), (2, 2), (100, 360), (200, 600), (200, 602), (400, 1024), (484, 1026), (700, 2048),
                                 (700, 2050), (1024, 4096), (1024, 2)])
def test_one_block(lib, V, E):
    edges, threads, two, smem = _out(lib.c_push, 4, V, E)
    assert threads <= 1024 and threads % 32 == 0 and V <= threads  # (a thread per variable where two)
    owned = [t + j * threads for j in range(edges) for t in range(threads) if t + j * threads < E]
    assert sorted(owned) == list(range(E))
    need = _walk([(4, 4 * V), (4, 4 * V)] + ([(8, V)] if two else []))
    assert need <= smem <= 48 * 1024 and (edges == 1 or two)


@pytest.mark.parametrize("V,S,local", [(100, 32, 1), (1536, 7, 1), (1537, 3, 1), (5000, 16, 1), (5000, 16, 0), (9000, 40, 1),
                                       (65536, 32, 1), (65536, 5, 1), (250000, 7, 1), (602175, 2, 1), (1000000, 3, 1),
                                       (1480000, 2, 1), (20000, 3, 0), (100, 100000, 1),
                                       (2025, 2, 0), (3000, 2, 0), (3001, 2, 0), (3600, 20, 0), (3600, 21, 0), (9409, 32, 0),
                                       (9409, 138, 0), (9409, 139, 0)])
def test_samples_per_launch(lib, V, S, local):
    Sc, nb, Vc, f, h, res, sample = _out(lib.c_multi, 7, V, S, local)
    if Sc == 0:  # (the numbering is not local and one block a sample does not pay; or no room)
        assert V > 9674 * SMS if local else V > 9674 or (V > 3000 and S < (V / 800) ** 2)
        return
    assert local or V <= 3000 or S >= (V / 800) ** 2
    assert 1 <= Sc <= S and nb * Vc >= V and (nb - 1) * Vc < V and 4 * Vc <= 1 << 16
    assert nb == 1 or Sc * nb <= SMS
    assert f == 2 * Vc and h == (4 * Vc if nb > 1 else 0)
    x = GRID if nb > 1 else ALONE
    assert bool(res) == (lib.c_run_smem(x, 1, 1, Vc, f, h) <= SMEM)
    assert res or lib.c_run_smem(x, 0, 0, Vc, 0, 0) <= SMEM
    # launch_lr_multi_run's layout: records, split records, two inboxes, addresses, explicit sums, directory
    parts = ([] if res else [(16, Sc * nb * f), (16, Sc * nb * h)]) + [(8, 2 * Sc * nb * h)] + ([] if res else [(4, Sc * nb * h)])
    assert _walk(parts + [(4, 4 * nb * Vc * Sc), (4, 4 * V * Sc)]) <= Sc * sample
