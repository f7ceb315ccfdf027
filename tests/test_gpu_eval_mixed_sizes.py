"""The FP32 mixed evaluator at the edges of its tiles: support vectors around
one tile of 256, several tiles, more tiles than a block has warps, and point
counts around the 32 of a block, for every dimension, against FP64 numpy."""
import numpy as np
import pytest

from paper_2406_04795_gb300 import mf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2406_04795_gb300.api import Context
    c = Context(0, 8 << 30)
    yield c
    c.close()


@pytest.mark.parametrize("d,n_sv,n", [(2, 1, 1), (3, 255, 31), (4, 256, 32), (5, 257, 33),
                                      (6, 2048, 65), (7, 2049, 640), (8, 2305, 1000)])
@pytest.mark.parametrize("precision", [mf.MF_FP64, mf.MF_MIXED_FP32])
def test_eval_sizes(ctx, d, n_sv, n, precision):
    rng = np.random.default_rng(100 * d + n)
    gamma, b = 1.5, 0.2
    sv = rng.uniform(-2, 2, size=(n_sv, d))
    alpha = rng.normal(size=n_sv)
    q = rng.uniform(-2, 2, size=(n, d))
    r2 = ((q[:, None, :] - sv[None]) ** 2).sum(-1)
    t = np.abs(alpha) * np.exp(-gamma * r2)
    f = np.exp(-gamma * r2) @ alpha + b
    got = ctx.eval(sv, alpha, gamma, b, q, precision=precision, band=1e-9).cpu().numpy()
    if precision == mf.MF_FP64:
        tol = 1e-12 * np.ones(n)
    else:
        # per term: 2 gamma eta sqrt(d) r with eta = 2.01 u (2 + 2), (d + 4) u
        # gamma r^2 and 2^-20, u = 2^-24; and the blocked sums' (256 + tiles) u
        u = 2.0 ** -24
        rel = (2 * gamma * 2.01 * u * 4 * np.sqrt(d * r2) + (d + 4) * u * gamma * r2 + 2.0 ** -20 +
               (256 + n_sv / 256 + 4) * u)
        tol = 1.1 * (t * rel).sum(1) + 1e-12
    assert np.all(np.abs(got - f) <= tol)


def test_eval_model_sizes_around_the_ranking_limit(ctx):
    """The vectors' order on the GPU up to 32768 of them, on the host beyond:
    f is the same function either way."""
    rng = np.random.default_rng(7)
    d, gamma, b = 3, 30.0, 0.1
    q = rng.uniform(-3, 3, size=(200, d))
    for n_sv in (32767, 32768, 32769):
        sv = rng.uniform(-3, 3, size=(n_sv, d))
        alpha = rng.normal(size=n_sv)
        f = np.exp(-gamma * ((q[:, None, :] - sv[None]) ** 2).sum(-1)) @ alpha + b
        got = ctx.eval(sv, alpha, gamma, b, q).cpu().numpy()
        assert np.max(np.abs(got - f)) <= 1e-11
