"""The search's passes pick the edges per warp from the size of each step; the
traced set, the end values and the cells must not depend on it.  A batch cap
splits every level into steps of that many edges, so caps around the group
sizes (4, 32) and around one block of warps reach each of them, with and
without a ragged last group."""
import pytest
import torch

from paper_2406_04795_gb300 import workloads as W

pytestmark = pytest.mark.gpu

EDGES = ("edge_y", "edge_mask", "edge_f")
CELLS = ("cell_y", "cell_perm", "cell_off", "cell_idx")  # written when cells are asked for
COUNTS = ("n_edges", "n_cells", "n_vertices", "n_boundary", "levels")


@pytest.fixture(scope="module")
def ctx():
    from paper_2406_04795_gb300.api import Context
    c = Context(0, 16 << 30)
    yield c
    c.close()


@pytest.mark.parametrize("d,lam,seed", [(2, 0.03, 2), (3, 0.12, 2), (5, 0.42, 4), (6, 0.7, 5),
                                        (8, 1.1, 7)])
def test_traced_set_is_the_same_for_every_step_size(ctx, d, lam, seed):
    w = W.random_small(d, 14, seed, lam, gamma=1.5, n_seeds=4, box=1.3)

    def run(cap):
        return ctx.trace(w.sv, w.alpha, w.gamma, w.b, w.lam, w.offset, w.lo, w.hi, w.seeds,
                         roots=False, cells=d <= 6, batch_cap=cap, max_edges=1 << 18, max_cells=1 << 21,
                         sort=True)

    full = run(1 << 24)
    assert full["n_edges"] > 20
    for cap in (3, 5, 33, 255, 1000):
        r = run(cap)
        assert [r[k] for k in COUNTS] == [full[k] for k in COUNTS]
        for k in EDGES + (CELLS if d <= 6 else ()):
            assert torch.equal(r[k], full[k]), (cap, k)
