"""Cell enumeration in every dimension (its lanes per edge depend on it): the
star of one lattice vertex, counted exactly, and a d = 6 trace against the
oracle."""
import math

import numpy as np
import pytest

from paper_2406_04795_gb300 import workloads as W
from tests import _parity as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2406_04795_gb300.api import Context
    c = Context(0, 16 << 30)
    yield c
    c.close()


@pytest.mark.parametrize("d", [2, 3, 4, 5, 6, 7, 8])
def test_star_of_one_vertex(ctx, d):
    lam = 0.2
    w = W.sphere_workload(d, r=0.3 * lam, gamma=1.0 / (lam * lam), lam=lam)
    w.sv = W.lattice_offset(d, lam)[None, :].copy()  # vertex y = 0
    w.seeds = w.sv + 0.3 * lam * np.eye(d)[0]
    g = P.gpu_trace(ctx, w, max_edges=1 << 16, max_cells=1 << 19)
    assert g["n_edges"] == 2 * (2 ** d - 1)  # the vertex's edges
    assert g["n_cells"] == math.factorial(d + 1)  # its n-simplices
    cells = np.concatenate([g["cell_y"], g["cell_perm"].astype(np.int64)], 1)
    assert len(np.unique(cells, axis=0)) == len(cells)


def test_cells_d6_against_oracle(ctx):
    w = W.random_small(6, 12, 5, 1.2, gamma=1.5, n_seeds=3, box=1.1)
    g = P.gpu_trace(ctx, w, roots=False, max_cells=1 << 20)
    o = P.oracle_trace(w, roots=False)
    rep = P.compare_traces(w, g, o, check_t=False)
    assert rep["n_diff"] == 0 and rep["n_cells"] > 100
