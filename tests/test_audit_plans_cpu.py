"""Checked mode's range checks of the plans that launches index by: the one-launch run's items by block
and the fused K-state form's block records. On the host (pgm_audit_desc): valid plans pass, a corrupted
entry is found at its position, the extreme values inside its range are accepted."""
import pytest

from paper_2202_04110_gb300 import workloads as W

GRID_OFF, FUSE = 13, 14


@pytest.fixture(scope="module")
def lib():
    from paper_2202_04110_gb300 import build
    build.build()
    from paper_2202_04110_gb300 import binding
    return binding


@pytest.mark.parametrize("shape,blocks", [((27, 26), 3), ((120, 130), 61), ((317, 241), 152)])
def test_items_of_a_one_launch_run(lib, shape, blocks):
    fg = W.ising_grid(*shape, seed=0).graph
    F = fg.n_edges // 2
    assert lib.audit_desc(fg) == (-1, -1)
    last = 2 * blocks + 1  # (whole, split) per block, then the totals
    for pos in (0, 1, last):
        for bad in (-1, 2 * F + 1):
            assert lib.audit_desc(fg, GRID_OFF, pos, bad) == (GRID_OFF, pos)
        assert lib.audit_desc(fg, GRID_OFF, pos, F) == (-1, -1)
    with pytest.raises(lib.PgmError):
        lib.audit_desc(fg, GRID_OFF, last + 1, 0)


def test_graphs_without_such_plans(lib):
    for fg in (W.ising_grid(10, 10, 0).graph, W.rbm(70, 80, 2).graph):
        for arr in (GRID_OFF, FUSE):
            with pytest.raises(lib.PgmError):
                lib.audit_desc(fg, arr, 0, 0)


@pytest.mark.parametrize("K,side", [(4, 30), (8, 41), (16, 30), (16, 300)])
def test_fused_blocks(lib, K, side):
    fg = W.potts_grid(side, K, 0).graph
    per = (128 if side < 300 else 256) * 4 // K  # one round of a block's teams
    n = -(-side * side // per)
    tail = side * side - (n - 1) * per
    assert lib.audit_desc(fg) == (-1, -1)
    assert lib.audit_desc(fg, FUSE, 0, -1) == (FUSE, 0)
    assert lib.audit_desc(fg, FUSE, n - 1, side * side - tail + 1) == (FUSE, n - 1)
    assert lib.audit_desc(fg, FUSE, n - 1, side * side - tail) == (-1, -1)
    with pytest.raises(lib.PgmError):
        lib.audit_desc(fg, FUSE, n, 0)
