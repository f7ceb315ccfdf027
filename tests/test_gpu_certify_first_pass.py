"""The first certification pass with the most elements it takes (8 capsules and
64 spheres: element indices past 63), with one obstacle of each type alone,
and with obstacles large enough to hold elements deep inside, against the FP64
oracle."""
import math

import numpy as np
import pytest

import oracle
from tests.test_gpu_certify_ext import _compare, _robot, _rot

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2406_04795_gb300.api import Context
    c = Context(0, 4 << 30)
    yield c
    c.close()


def _obstacle(rng, typ, reach, size):
    R = _rot(rng) if typ != 1 else np.eye(3)
    c = rng.uniform(-0.5 * reach, 0.5 * reach, 3)
    dims = [size * rng.uniform(0.5, 1.0, 3), [0.5 * size, 0, 0], [0.4 * size, 1.2 * size, 0]][typ]
    return np.concatenate([R.reshape(-1), c]), dims


@pytest.mark.parametrize("types,size,links,caps,spheres", [
    ([0], 0.4, 3, True, 0), ([1], 0.4, 3, True, 2), ([2], 0.4, 4, True, 1), ([0, 1, 2], 1.5, 5, True, 3),
    ([0, 1, 2, 0, 1, 2], 0.5, 8, True, 8), ([2, 0], 1.5, 8, False, 8), ([], 0.4, 3, True, 1)])
def test_first_pass_against_oracle(ctx, types, size, links, caps, spheres):
    rng = np.random.default_rng(17 * links + len(types))
    dh, radius, sph = _robot(rng, links, spheres_per_link=max(spheres, 1), radius=0.05)
    reach = float(dh[:, 2].sum())
    obs = [_obstacle(rng, t, reach, size) for t in types]
    ty = np.array(types, np.int32)
    pose = np.array([o[0] for o in obs]).reshape(-1, 12)
    dims = np.array([o[1] for o in obs], np.float64).reshape(-1, 3)
    pts = rng.uniform(-math.pi, math.pi, size=(777, links))
    kw = dict(spheres=sph if spheres else None)
    g = ctx.certify_ex(dh, radius if caps else None, ty, pose, dims, pts, **kw)
    o = oracle.certify_ex(dh, radius if caps else None, ty, pose, dims, pts, **kw)
    if types:
        _compare(g, o)
    else:
        assert np.array_equal(g["verdict"].cpu().numpy(), o["verdict"])
        assert np.array_equal(np.isinf(g["margin"].cpu().numpy()), np.isinf(o["margin"]))
