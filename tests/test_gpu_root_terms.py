"""The profile's count of the root solve's FP32 terms: one per listed vector and
evaluation that an edge needs, the last evaluation included.  With a single
vector it is the number of evaluations: a step and the last one for each edge at
least, and no more than the solve's 12 steps, the last one and as many again for
an edge that is solved a second time."""
import pytest

from paper_2406_04795_gb300 import mf
from paper_2406_04795_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,lam", [(2, 0.01), (3, 0.05), (4, 0.1)])
def test_fp32_terms_of_one_vector(d, lam):
    from paper_2406_04795_gb300.api import Context
    ctx = Context(0, 8 << 30)
    w = W.sphere_workload(d, r=0.9, gamma=1.0, lam=lam)
    mf.mf_ctx_set_profiling(ctx.h, True)
    r = ctx.trace(w.sv, w.alpha, w.gamma, w.b, w.lam, w.offset, w.lo, w.hi, w.seeds, cells=False,
                  max_edges=1 << 20)
    n, terms = r["n_edges"], mf.mf_ctx_get_stats(ctx.h)["roots"]["terms_weak"]
    mf.mf_ctx_set_profiling(ctx.h, False)
    ctx.close()
    assert n > 500 and 2 * n <= terms <= 26 * n
