"""The root solve grouped by base vertex in its other modes: the mixed path's
accuracy (BF16) and a mixed path with exact roots at every list length where the
instantiation or the kernel changes, the run-time dimension, and a trace of more
edges than one chunk of the solve's pools."""
import numpy as np
import pytest

from paper_2406_04795_gb300 import mf
from paper_2406_04795_gb300 import workloads as W
from tests import _parity as P
from tests.test_gpu_roots_grouped import _many_vectors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2406_04795_gb300.api import Context
    c = Context(0, 64 << 30)
    yield c
    c.close()


def _order(y, mask):
    y, mask = np.asarray(y), np.asarray(mask)
    return np.lexsort(np.concatenate([y, mask[:, None]], 1).T)


# t: the paths' stated accuracies, 1e-6 of the mixed ones and 1e-9 with exact
# roots, and the oracle's own 1e-9 below the first
@pytest.mark.parametrize("n_sv", [64, 65, 128, 129, 192, 193, 256, 257, 320, 321, 512, 513])
@pytest.mark.parametrize("precision,exact,t_tol", [(mf.MF_MIXED_BF16, False, 1e-6),
                                                   (mf.MF_MIXED_FP32, True, 1e-9)])
def test_mixed_list_lengths_against_oracle(ctx, n_sv, precision, exact, t_tol):
    w = _many_vectors(3, n_sv, 0.1, 8)
    o = P.oracle_trace(w, cells=False)
    r = ctx.trace(w.sv, w.alpha, w.gamma, w.b, w.lam, w.offset, w.lo, w.hi, w.seeds,
                  precision=precision, cells=False, exact_roots=exact, max_edges=1 << 16)
    y, m, t = (r[k].cpu().numpy() for k in ("edge_y", "edge_mask", "edge_t"))
    a, b = _order(y, m), _order(o["edge_y"], o["edge_mask"])
    assert r["n_edges"] > 50 and np.array_equal(y[a], o["edge_y"][b])
    assert np.array_equal(m[a], o["edge_mask"][b])
    one = o["edge_multiroot"][b] == 0
    assert np.abs(t[a] - o["edge_t"][b])[one].max() <= t_tol


def test_run_time_dimension(ctx):
    w = _many_vectors(8, 70, 1.1, 13)
    g = P.gpu_trace(ctx, w, mf.MF_FP64, cells=False)
    o = P.oracle_trace(w, cells=False)
    rep = P.compare_traces(w, g, o, f_tol=1e-12, t_tol=1e-9, check_cells=False)
    assert rep["n_diff"] == 0 and rep["n_edges"] > 50


def test_more_edges_than_the_pools_hold(ctx):
    """f at every point is within what an error of 1e-9 in t leaves: |f'| per
    unit of t is at most a few times the end values' difference here."""
    w = W.config_d5(lam=0.095)
    r = ctx.trace(w.sv, w.alpha, w.gamma, w.b, w.lam, w.offset, w.lo, w.hi, w.seeds, cells=False,
                  max_edges=1 << 23)
    assert r["n_edges"] > 1 << 22
    t = r["edge_t"]
    assert float(t.min()) >= 0.0 and float(t.max()) <= 1.0
    f = ctx.eval(w.sv, w.alpha, w.gamma, w.b, r["points"])
    ef = r["edge_f"]
    assert bool((f.abs() <= 1e-8 * (ef[:, 1] - ef[:, 0]).abs() + 1e-11).all())
