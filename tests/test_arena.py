"""The context's device arena (on a fake device): the pools that it may give back
make way for any other buffer, whether the budget or the device is short, and
are themselves refused rather than anything else given up for them."""
import pytest

from paper_2406_04795_gb300 import mf

MB = 1 << 20
TABLES, EDGES, POOLS = 2, 3, 18  # MF_SLOT_BATCHROOTS = 18


@pytest.mark.parametrize("budget,device", [(100, 1000), (1000, 100), (100, 100)])
def test_pools_make_way(budget, device):
    got = mf.mf_diag_arena(budget * MB, device * MB,
                           [(TABLES, 40 * MB), (POOLS, 30 * MB), (EDGES, 50 * MB), (POOLS, 30 * MB),
                            (TABLES, 50 * MB)])
    assert [g[0] // MB for g in got] == [40, 30, 50, 0, 50]
    assert [g[1] // MB for g in got] == [40, 70, 90, 90, 100]


def test_refused_without_pools():
    got = mf.mf_diag_arena(1000 * MB, 100 * MB, [(TABLES, 60 * MB), (EDGES, 60 * MB), (EDGES, 40 * MB)])
    assert [g[0] // MB for g in got] == [60, 0, 40]


def test_what_a_slot_holds_is_kept():
    got = mf.mf_diag_arena(100 * MB, 100 * MB, [(TABLES, 60 * MB), (TABLES, 10 * MB), (POOLS, 40 * MB),
                                                (POOLS, 20 * MB)])
    assert [g[0] // MB for g in got] == [60, 60, 40, 40] and got[-1][1] == 100 * MB
