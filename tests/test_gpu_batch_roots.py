"""Roots of batched traces on both sides of the size from which a slot takes the
single trace's root solve, in one batch and in several precisions, against the
traces one by one; and that solve's pools beside the context's other work: a
subdivision in progress, and a budget that does not hold them too."""
import numpy as np
import pytest
import torch

from paper_2406_04795_gb300 import mf
from paper_2406_04795_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CAP = dict(max_edges=1 << 18)


def _key(r, w):
    return np.lexsort(np.concatenate([r["edge_y"].cpu().numpy(),
                                      r["edge_mask"].cpu().numpy()[:, None]], 1).T)


def _roots(r, w):
    return r["edge_t"].cpu().numpy()[_key(r, w)]


def _trace(ctx, w, p):
    return ctx.trace(w.sv, w.alpha, w.gamma, w.b, w.lam, w.offset, w.lo, w.hi, w.seeds, precision=p,
                     cells=False, **CAP)


def _workloads():
    # a few hundred to some 1e5 edges
    return [W.random_small(d, 40, 3 + i, lam, gamma=1.5, n_seeds=4, box=1.2)
            for i, (d, lam) in enumerate([(3, 0.3), (3, 0.04), (4, 0.25), (5, 0.6), (4, 0.5)])]


@pytest.mark.parametrize("precision", [mf.MF_FP64, mf.MF_MIXED_FP32, mf.MF_MIXED_BF16])
def test_batch_against_single_traces(precision):
    from paper_2406_04795_gb300.api import Context
    ctx = Context(0, 24 << 30)
    ws = _workloads()
    rs = ctx.trace_batch(ws, [precision] * len(ws), cells=False, capacities=[CAP] * len(ws))
    # both solve to 1e-9 (FP64) or 1e-6 (mixed) of the root
    tol = 2e-9 if precision == mf.MF_FP64 else 2e-6
    n = []
    for w, r in zip(ws, rs):
        one = _trace(ctx, w, precision)
        assert r["n_edges"] == one["n_edges"]
        a, b = _roots(r, w), _roots(one, w)
        assert np.all((a > 0) & (a < 1)) and np.abs(a - b).max() <= tol
        n.append(r["n_edges"])
    assert min(n) < 8192 < max(n)
    ctx.close()


def test_pools_are_given_back():
    """A trace that fits the budget beside the batch, but not beside the pools
    too, still runs and still has its roots."""
    from paper_2406_04795_gb300.api import Context
    ws = _workloads()
    a = Context(0, 24 << 30)
    ref = _roots(_trace(a, ws[1], mf.MF_FP64), ws[1])
    t_bytes = mf.mf_ctx_bytes(a.h)
    a.close()
    a = Context(0, 24 << 30)
    a.trace_batch(ws[1:3], [mf.MF_FP64] * 2, cells=False, capacities=[CAP] * 2)
    b_bytes = mf.mf_ctx_bytes(a.h)
    a.close()
    c = Context(0, t_bytes + b_bytes - (1 << 20))
    c.trace_batch(ws[1:3], [mf.MF_FP64] * 2, cells=False, capacities=[CAP] * 2)
    got = _roots(_trace(c, ws[1], mf.MF_FP64), ws[1])
    assert np.abs(got - ref).max() <= 2e-9
    assert mf.mf_ctx_bytes(c.h) <= t_bytes + b_bytes - (1 << 20)
    c.close()


def test_batch_beside_a_subdivision():
    """Batches that grow their pools between a subdivision's calls leave it as
    it was."""
    from paper_2406_04795_gb300.api import Context
    w = W.random_small(3, 40, 4, 0.1, gamma=1.5, n_seeds=4, box=1.2)
    ws = _workloads()
    ctx = Context(0, 24 << 30)
    kw = dict(cells_per_batch=200, max_edges=1 << 16)
    a = ctx.subdiv(w, 2, **kw)
    ctx.close()
    ctx = Context(0, 24 << 30)
    calls = []

    def batch(_):
        if len(calls) < 3:
            ctx.trace_batch(ws[len(calls):len(calls) + 2], [mf.MF_FP64] * 2, cells=False,
                            capacities=[CAP] * 2)
        calls.append(1)

    b = ctx.subdiv(w, 2, each_batch=batch, **kw)
    ctx.close()
    assert len(calls) >= 3
    # an edge of a face that two batches share is in both: compare each edge once
    ea, eb = [dict(zip(map(tuple, torch.cat([r["edge_y"], r["edge_mask"][:, None].int()], 1).tolist()),
                       r["edge_t"].tolist())) for r in (a, b)]
    assert ea.keys() == eb.keys() and len(ea) > 1000
    assert max(abs(ea[k] - eb[k]) for k in ea) <= 2e-9
