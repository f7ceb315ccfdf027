"""The proof server takes its root pools at creation: serving allocates nothing,
whatever the sizes of the traces that finish, on a budget with room for the
pools and on one without; the roots are the single trace's."""
import numpy as np
import pytest

from paper_2406_04795_gb300 import mf
from paper_2406_04795_gb300 import workloads as W
from tests.test_gpu_batch_roots import _roots, _trace

pytestmark = pytest.mark.gpu

CAP = dict(max_edges=1 << 18)


@pytest.mark.parametrize("budget", [24 << 30, (4 << 30) + (1 << 20)])
def test_serving_allocates_nothing(budget):
    from paper_2406_04795_gb300.api import Context
    # edges: a few hundred, some 1e4, some 1e5
    ws = [W.random_small(3, 40, 3, lam, gamma=1.5, n_seeds=4, box=1.2) for lam in (0.3, 0.08, 0.04)]
    ctx = Context(0, budget)
    server = ctx.server(max_slots=4, hbm_bytes=4 << 30)
    held = mf.mf_ctx_bytes(ctx.h)
    assert held <= budget and (held > (4 << 30)) == (budget > (5 << 30))
    got = []
    for w in ws:
        rid = server.submit(w, precision=mf.MF_FP64, cells=False, **CAP)
        while rid not in server.done():
            server.step()
        got.append(server.fetch(rid))
        assert mf.mf_ctx_bytes(ctx.h) == held
    server.close()
    ctx.close()
    n = [r["n_edges"] for r in got]
    assert n[0] < 8192 < n[1] < n[2]
    ref = Context(0, 8 << 30)
    for w, r in zip(ws, got):
        assert np.abs(_roots(r, w) - _roots(_trace(ref, w, mf.MF_FP64), w)).max() <= 2e-9
    ref.close()
