"""A trace beside other work on the GPU, which holds back blocks of the search's
kernels: the same edges, cells, end values and levels as alone."""
import pytest
import torch

from paper_2406_04795_gb300 import mf
from paper_2406_04795_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FIELDS = ("edge_y", "edge_mask", "edge_f", "cell_y", "cell_perm", "cell_off", "cell_idx")
COUNTS = ("n_edges", "n_cells", "n_vertices", "n_boundary", "levels")


@pytest.mark.parametrize("d,lam,repeats", [(3, 0.05, 12), (4, 0.2, 12), (5, 0.42, 6)])
def test_same_traced_set_beside_matmuls_on_another_stream(d, lam, repeats):
    from paper_2406_04795_gb300.api import Context
    ctx = Context(0, 16 << 30)
    w = W.random_small(d, 14, 2, lam, gamma=1.5, n_seeds=4, box=1.3)

    def run():
        return ctx.trace(w.sv, w.alpha, w.gamma, w.b, w.lam, w.offset, w.lo, w.hi, w.seeds,
                         precision=mf.MF_FP64, roots=False, max_edges=1 << 18, max_cells=1 << 21,
                         sort=True)

    alone = run()
    assert alone["n_edges"] > 1000
    side = torch.cuda.Stream()
    a = torch.randn((2048, 2048), device="cuda", dtype=torch.bfloat16)
    out = torch.empty_like(a)
    torch.cuda.synchronize()
    for _ in range(repeats):
        with torch.cuda.stream(side):
            for _ in range(300):
                torch.mm(a, a, out=out)
        r = run()
        assert [r[k] for k in COUNTS] == [alone[k] for k in COUNTS]
        for k in FIELDS:
            assert torch.equal(r[k], alone[k]), k
    torch.cuda.synchronize()
    ctx.close()
