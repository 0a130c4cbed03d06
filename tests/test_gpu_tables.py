"""Cell geometry without tables: angular coordinates that split more often than their
(sin, cos) tables reach, and rotation coordinates with more cells than a rotation table
holds, evaluate the basis directly; with tables is the ordinary case of every other test."""
import math

import numpy as np
import pytest

import oracle
from paper_2107_11810_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2107_11810_gb300 import build
    build.build()


def deep_plane():
    p = inputs.plane3d(n=40, inlier_frac=0.4, eps=0.2, sigma=0.001, seed=51)
    p.eps = np.array([math.pi / 2 ** 17 * 1.01, 0.4, 0.2])     # theta splits 17 times
    return p


def deep_yaw():
    p = inputs.pose3dof(n=60, inlier_frac=0.3, eps_xy=3.0, eps_yaw_deg=1.0, seed=52)
    p.eps = np.array([2 * math.pi / 2 ** 18 * 1.01, 3.0, 3.0])  # yaw splits 18 times
    return p


def deep_rotation():
    p = inputs.radial5dof(n=40, inlier_frac=0.5, prior_deg=1.0, levels=8, seed=53)      # 2^24 rotation cells
    p.eps = np.concatenate([p.eps[:3], [2.5, 2.5]])
    return p


@pytest.mark.parametrize("make", [deep_plane, deep_yaw, deep_rotation])
@pytest.mark.parametrize("precision", [0, 1])
def test_geometry_without_tables_equals_the_oracle(make, precision):
    from paper_2107_11810_gb300 import vote as v
    p = make()
    o = oracle.solve(p.family, p.eps, p.bounds, p.params)
    s = v.Solver(p.family, p.eps, p.bounds, precision=precision)
    r = s.solve(torch.from_numpy(np.ascontiguousarray(p.params)).cuda())
    assert r["depth"] == o["depth"]
    assert np.array_equal(r["best_leaf"], o["best_leaf"])
    assert np.array_equal(v.mask_words_to_numpy(r["mask"]), o["mask"])
