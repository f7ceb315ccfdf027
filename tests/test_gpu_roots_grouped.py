"""The root solve grouped by base vertex: lists around its lanes-per-edge limits
(64 and 192 vectors), around the longest list it takes (512: edges beyond go to
the per-edge kernel), and a single vector, against the FP64 oracle; and a
subset of the edges in several precisions against the same trace."""
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


def _many_vectors(d, n_sv, lam, seed):
    """n_sv vectors all within reach of every vertex (gamma small), f changing
    sign across the box; the zero set is smooth on the lattice's scale."""
    w = W.random_small(d, 12, seed, lam, gamma=1.5, n_seeds=4, box=1.2)
    rng = np.random.default_rng(seed)
    extra = n_sv - 12
    if extra > 0:
        sv = rng.uniform(-1.2, 1.2, size=(extra, d))
        al = 1e-3 * rng.normal(size=extra)
        w.sv, w.alpha = np.concatenate([w.sv, sv]), np.concatenate([w.alpha, al])
    return w


@pytest.mark.parametrize("d,lam,n_sv", [(3, 0.25, 64), (3, 0.25, 65), (2, 0.06, 192),
                                        (4, 0.4, 193), (3, 0.25, 512), (3, 0.25, 513),
                                        (5, 0.5, 200), (7, 0.9, 70)])
@pytest.mark.parametrize("precision", [mf.MF_FP64, mf.MF_MIXED_FP32])
def test_list_lengths_against_oracle(ctx, d, lam, n_sv, precision):
    w = _many_vectors(d, n_sv, lam, 5 + d)
    g = P.gpu_trace(ctx, w, precision, cells=False)
    o = P.oracle_trace(w, cells=False)
    rep = P.compare_traces(w, g, o, f_tol=1e-12 if precision == mf.MF_FP64 else 1e-3,
                           t_tol=1e-9 if precision == mf.MF_FP64 else 1e-6, check_cells=False)
    assert rep["n_diff"] == 0 and rep["n_edges"] > 50


def test_one_vector(ctx):
    w = W.sphere_workload(3, r=0.9, gamma=1.0, lam=0.2)
    g = P.gpu_trace(ctx, w, cells=False)
    o = P.oracle_trace(w, cells=False)
    assert P.compare_traces(w, g, o, check_cells=False)["n_diff"] == 0


def test_more_edges_than_one_chunk_of_vertices(ctx):
    """Every edge of a trace of some 1e5 edges is solved once: t in (0, 1), and
    f changes sign across t +- 1e-7."""
    w = W.config_d5(lam=0.25)
    r = ctx.trace(w.sv, w.alpha, w.gamma, w.b, w.lam, w.offset, w.lo, w.hi, w.seeds, cells=False)
    t = r["edge_t"].cpu().numpy()
    assert t.min() >= 0.0 and t.max() <= 1.0 and r["n_edges"] > 50000
    f = ctx.eval(w.sv, w.alpha, w.gamma, w.b, r["points"]).cpu().numpy()
    # |f| at the root is below |f'| dt + the evaluation's 1e-12: |f'| per unit
    # of t is at most a few times the end values' difference on this lattice
    ef = r["edge_f"].cpu().numpy()
    assert np.all(np.abs(f) <= 1e-8 * np.abs(ef[:, 1] - ef[:, 0]) + 1e-11)
