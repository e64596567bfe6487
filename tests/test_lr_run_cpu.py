"""Index arithmetic of the one-launch runs of binary pairwise graphs, checked on the host.

The kernels of lr_run.cu split a graph's variables into blocks of Vc, list each block's
whole factors (both variables in the block) and split ones (one item per block they join),
and exchange one value per split item through an inbox word of the other block. This restates the partition,
the item counts, the inbox addressing and the workspace layout, and checks over grids,
chains and random numberings that every message is computed exactly once, every inbox word
has exactly one writer, and every index stays inside its array.
"""
import numpy as np
import pytest

from paper_2202_04110_gb300 import workloads as W

N_SM, SMEM, MIN_V = 152, 232448 - 256, 256  # a GB300: SMs, shared memory per block; kLrGridMinV
CLUSTER_V, CLUSTER = 1024, 16


def slots(graph):
    """tab4 [V, 4] incoming edges (ascending, -1 padded) and each edge's (variable, slot index)."""
    e_var = graph.enum_groups[0].vars.reshape(-1).astype(np.int64)
    order = np.argsort(e_var, kind="stable")
    start = np.searchsorted(e_var[order], np.arange(graph.n_vars))
    k = np.empty(e_var.size, np.int64)
    k[order] = np.arange(e_var.size) - start[e_var[order]]
    assert k.max() < 4
    return e_var, k


def grid_plan(V, n_sm=N_SM):
    Vc = max(-(-V // n_sm), MIN_V)
    nb = -(-V // Vc)
    if nb < 2 or 24 * Vc + 16 > SMEM or Vc >= 1 << 14:
        return 0, 0
    return nb, -(-V // nb)


def items(graph, nb, Vc):
    """Per block the whole factors and the split items (edge ids)."""
    e_var, _ = slots(graph)
    mul = ((1 << 40) + Vc - 1) // Vc
    blk = np.array([(int(v) * mul) >> 40 for v in e_var]) if e_var.size < 5000 else (e_var * mul) >> 40
    assert np.array_equal(blk, e_var // Vc) and blk.max() < nb
    a, b = blk[0::2], blk[1::2]
    whole = a == b
    return blk, whole


def smem(res, Vc, f, h, cluster=False):
    return 24 * Vc + (8 * Vc + 16 * f + 20 * h if res else 0) + (16 * h if cluster else 0) + 16


def random_numbering(rows, cols, seed):
    p = W.ising_grid(rows, cols, seed)
    perm = np.random.default_rng(seed).permutation(rows * cols).astype(np.int32)
    p.graph.enum_groups[0].vars[:] = perm[p.graph.enum_groups[0].vars]
    return p


GRAPHS = {
    "129x128": lambda: W.ising_grid(129, 128, 0), "317x241": lambda: W.ising_grid(317, 241, 0),
    "17x3000": lambda: W.ising_grid(17, 3000, 0), "3000x17": lambda: W.ising_grid(3000, 17, 0),
    "1x40001": lambda: W.ising_grid(1, 40001, 0), "500x500": lambda: W.ising_grid(500, 500, 0),
    "random 150x150": lambda: random_numbering(150, 150, 1), "1000x1000": lambda: W.ising_grid(1000, 1000, 0),
    "1200x1209": lambda: W.ising_grid(1200, 1209, 0),
}


@pytest.mark.parametrize("name", list(GRAPHS))
def test_grid_items_and_workspace(name):
    graph = GRAPHS[name]().graph
    V, E = graph.n_vars, graph.n_edges
    F = E // 2
    nb, Vc = grid_plan(V)
    assert 2 <= nb <= N_SM and (nb - 1) * Vc < V + Vc  # (a last block may own nothing)
    e_var, k = slots(graph)
    blk, whole = items(graph, nb, Vc)
    nF = np.bincount(blk[0::2][whole], minlength=nb)
    split = np.repeat(~whole, 2)
    nH = np.bincount(blk[split], minlength=nb)
    assert nF.sum() + nH.sum() // 2 == F
    off = np.concatenate([[0], np.cumsum(nH)])
    # a split edge's item: any order within its block; its value comes from the other edge
    item = np.empty(E, np.int64)
    for b in range(nb):
        mine = np.flatnonzero(split & (blk == b))
        item[mine] = off[b] + np.arange(mine.size)
    e = np.flatnonzero(split)
    dst = item[e ^ 1]
    assert np.array_equal(np.sort(dst), np.arange(e.size))  # one writer per word
    n_split = e.size
    # packed slots: local variable in 14 bits, slot index in 2
    assert (e_var - blk * Vc).max() < min(Vc, 1 << 14) and k.max() < 4
    res = smem(True, Vc, nF.max(), nH.max()) <= SMEM
    if res:  # inboxes (8 bytes) in m_tmp [16 F] and prm [12 F]
        fits = 2 * n_split <= 3 * F
        if fits:
            assert 8 * n_split <= 16 * F and 8 * n_split <= 12 * F
    else:    # records in m_tmp [16 F] and prm [12 F], inboxes in b [8 V]
        fits = 20 * n_split <= 12 * F and 16 * n_split <= 8 * V
        assert 16 * int(nF.sum()) <= 16 * F and smem(False, Vc, 0, 0) <= SMEM
    assert fits or "random" in name or name == "17x3000"


@pytest.mark.parametrize("V", [701, 1025, 4096, 16384])
def test_cluster_items_fit_their_worst_case(V):
    Vc = -(-V // CLUSTER)
    assert Vc <= CLUSTER_V
    f, h = 2 * Vc, 4 * Vc  # 4 slots per variable: a whole factor takes two, a split item one
    assert smem(True, Vc, f, h, cluster=True) <= SMEM
    for graph in (W.ising_grid(1, V, 0).graph, random_numbering(1, V, 2).graph):
        blk, whole = items(graph, CLUSTER, Vc)
        assert np.bincount(blk[0::2][whole], minlength=CLUSTER).max(initial=0) <= f
        assert np.bincount(blk[np.repeat(~whole, 2)], minlength=CLUSTER).max(initial=0) <= h


@pytest.mark.parametrize("V,S", [(100, 32), (1537, 3), (5000, 16), (9000, 40), (65536, 32), (65536, 5), (250000, 7),
                                 (1000000, 3)])
def test_samples_per_launch(V, S):
    v_max = min((1 << 14) - 1, (SMEM - 16) // 24)
    nb_min = -(-V // v_max)
    nb, Sc = 1, S
    if V > 1536:
        chunks = -(-S // (N_SM // nb_min))
        Sc = -(-S // chunks)
        nb = min(N_SM // Sc, -(-V // MIN_V))
    Vc = -(-V // nb)
    nb = -(-V // Vc)
    assert 1 <= Sc <= S and (nb == 1 or Sc * nb <= N_SM) and Vc <= v_max
    f, h = 2 * Vc, 4 * Vc if nb > 1 else 0
    if smem(True, Vc, f, h) > SMEM:
        assert smem(False, Vc, 0, 0) <= SMEM
