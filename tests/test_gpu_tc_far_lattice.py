"""The tensor-core evaluation on a lattice whose coordinates are large (an offset
of many lattice steps, up to the key packing's limits): the tile bases stay among
the tiles' vertices, so that only vertices near the manifold are rechecked, and
the traced set is the FP64 path's."""
import numpy as np
import pytest
import torch

from paper_2406_04795_gb300 import mf
from paper_2406_04795_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps", [0, 60_000_000, 70_000_000, 120_000_000, -500_000_000])
def test_recheck_does_not_depend_on_the_offset(steps):
    from paper_2406_04795_gb300.api import Context
    ctx = Context(0, 8 << 30)
    w = W.random_small(3, 14, 2, 0.06, gamma=1.5, n_seeds=4, box=1.3)
    # y + (steps, -steps, 0): the coordinate sum, and with it L y's common part,
    # stays, so the lattice is the same one up to rounding
    off = np.array(w.offset) - w.lam * np.array([steps, -steps, 0.0])

    def run(precision):
        return ctx.trace(w.sv, w.alpha, w.gamma, w.b, w.lam, off, w.lo, w.hi, w.seeds,
                         precision=precision, cells=False, max_edges=1 << 18, sort=True)

    a, b = run(mf.MF_FP64), run(mf.MF_MIXED_BF16)
    assert a["n_edges"] > 5000 and b["n_vertices"] == a["n_vertices"]
    for k in ("edge_y", "edge_mask"):
        assert torch.equal(a[k], b[k]), k
    # a band of 1e-3 about the manifold, against half a lattice step (|f| ~ 0.02)
    # on both sides of it: far below half of the vertices
    assert b["n_recheck"] < 0.5 * b["n_vertices"]
    ctx.close()
