"""Every launch variant that the autotuner times reaches a launch: three search
chunks, eighteen variants of the edge-by-edge root solve, whatever solve the
trace itself takes, and the precision's evaluation variants."""
import pytest

from paper_2406_04795_gb300 import mf
from paper_2406_04795_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,n", [(mf.MF_FP64, 24), (mf.MF_MIXED_BF16, 23),
                                         (mf.MF_MIXED_FP32, 21)])
def test_candidates_reach_a_launch(precision, n):
    from paper_2406_04795_gb300.api import Context
    ctx = Context(0, 16 << 30)
    t = ctx.autotune(W.config_d5(lam=0.3), precision=precision)
    assert t["n_candidates"] == n and t["ms_roots"] > 0
    ctx.close()
