"""The search's step protocol (host simulation over the kernels' own functions):
whatever the order in which the blocks of an edges pass start and finish, those
without work last among them, every edge is expanded exactly once, in the levels
of the breadth-first search and in steps of at most the cap; and a search whose
kernels the device refuses ends with an error, noticed or not."""
import numpy as np
import pytest

from paper_2406_04795_gb300 import mf


def _appends(rng, sizes):
    """The edges that each edge appends, so that the levels have these sizes
    (edges are numbered as they are appended)."""
    out = []
    for n, following in zip(sizes, list(sizes[1:]) + [0]):
        out.append(rng.multinomial(following, np.full(n, 1.0 / n)))
    return np.concatenate(out)


@pytest.mark.parametrize("d,grid,cap", [(3, 24, 1 << 24), (3, 24, 700), (4, 16, 1 << 24),
                                        (6, 40, 1 << 24), (2, 8, 900), (5, 1, 64)])
def test_every_edge_is_expanded_once_in_any_block_order(d, grid, cap):
    for seed in range(8):
        rng = np.random.default_rng(100 * d + seed)
        # levels from a single edge to several rounds of every warp, neighbours
        # of different sizes: the blocks with work change from step to step
        sizes = np.exp(rng.uniform(0.0, np.log(500.0 * grid), size=24)).astype(np.int64)
        appends = _appends(rng, sizes)
        got, levels, steps = mf.mf_diag_search(d, grid, cap, appends, int(sizes[0]), seed)
        assert (got == 1).all()
        assert levels == sizes.size
        assert steps == sum(-(-int(s) // cap) for s in sizes)


def test_no_seed_edges():
    got, levels, steps = mf.mf_diag_search(3, 8, 100, np.ones(10, np.int32), 0, 1)
    assert not got.any() and (levels, steps) == (0, 0)


@pytest.mark.parametrize("refused", [0, 1, 2, 5, 10])
@pytest.mark.parametrize("status", [mf.MF_OK, mf.MF_ERR_CUDA])
def test_refused_launches_end_the_search(refused, status):
    appends = _appends(np.random.default_rng(3), np.array([5, 40, 300, 700, 200, 90, 30, 7, 5, 3, 2, 1, 1]))
    with pytest.raises(mf.MfError) as e:
        mf.mf_diag_search(3, 8, 1 << 24, appends, 5, 1, refused=refused, status=status)
    assert e.value.code == mf.MF_ERR_CUDA
