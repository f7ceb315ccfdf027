"""Sorted cells in both key forms: (vertex key, rank of pi) in one 64-bit word,
and two sorts where the two do not fit (d = 8 on a fine lattice).  The zero set
is a small sphere around one lattice vertex: every edge and every n-simplex at
the vertex crosses."""
import math

import numpy as np
import pytest

from paper_2406_04795_gb300 import mf
from paper_2406_04795_gb300 import workloads as W
from tests import _parity as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2406_04795_gb300.api import Context
    c = Context(0, 16 << 30)
    yield c
    c.close()


@pytest.mark.parametrize("d,lam", [(2, 0.01), (3, 0.1), (5, 0.3), (6, 0.05), (7, 0.2), (8, 0.11)])
def test_star_of_one_vertex_sorted(ctx, d, lam):
    w = W.sphere_workload(d, r=0.3 * lam, gamma=1.0 / (lam * lam), lam=lam)
    w.sv = W.lattice_offset(d, lam)[None, :].copy()  # vertex y = 0
    w.seeds = w.sv + 0.3 * lam * np.eye(d)[0]
    g = P.gpu_trace(ctx, w, sort=True, max_edges=1 << 16, max_cells=1 << 19)
    assert g["n_edges"] == 2 * (2 ** d - 1)  # the vertex's edges
    assert g["n_cells"] == math.factorial(d + 1)  # its n-simplices
    assert np.all(np.diff(g["cell_off"]) == d)  # each has d edges at the vertex
    dom = mf.mf_domain()
    for i in range(d):
        dom.lo[i], dom.hi[i], dom.offset[i] = w.lo[i], w.hi[i], w.offset[i]
    keys, ok = mf.mf_vertex_keys(d, w.lam, dom, g["cell_y"])
    assert ok.all()
    code = np.zeros(len(keys), np.uint64)
    for k in range(d):
        code = code * np.uint64(8) + g["cell_perm"][:, k].astype(np.uint64)
    up = keys[1:] > keys[:-1]
    same = keys[1:] == keys[:-1]
    assert np.all(up | (same & (code[1:] > code[:-1])))
    ek, _ = mf.mf_vertex_keys(d, w.lam, dom, g["edge_y"])
    ek = ek.astype(object) * (1 << d) + g["edge_mask"].astype(object)
    assert all(ek[i] < ek[i + 1] for i in range(len(ek) - 1))
    # each row holds the edges whose two vertices are in the cell, once each
    rows = g["cell_idx"].reshape(-1, d)
    assert np.all(np.sort(rows, 1)[:, 1:] != np.sort(rows, 1)[:, :-1])
