"""The replay screens surfaces in one jump from the root before it takes the steps: the
same counts and reach masks as the oracle's steps, at every level of the best leaf's path
(where surfaces pass) and of cells beside it (where they just fail), around the sizes at
which a block's share ends."""
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


MAKE = {
    "line2d": lambda: inputs.line2d(n=2500, inlier_frac=0.5, eps=0.02, seed=51),
    "plane3d": lambda: inputs.plane3d(n=2500, inlier_frac=0.5, eps=0.05, sigma=0.005, seed=52),
    "pose3dof": lambda: inputs.pose3dof(n=2500, inlier_frac=0.5, eps_xy=1.0, eps_yaw_deg=2.0, seed=53),
    "rays3d": lambda: inputs.rays3d(n=2500, inlier_frac=0.5, seed=54),
    "pointset2d": lambda: inputs.pointset2d(m=50, eps=0.05, seed=55),
    "affine4d": lambda: inputs.affine4d(n=2500, inlier_frac=0.5, eps=0.1, noise=0.01, seed=56),
    "pose6dof": lambda: inputs.pose6dof(n=1500, inlier_frac=0.5, prior_deg=5.0, levels=4, seed=57),
    "radial5dof": lambda: inputs.radial5dof(n=1500, inlier_frac=0.5, prior_deg=5.0, levels=4, seed=58),
}


@pytest.mark.parametrize("name", sorted(MAKE))
def test_replay_equals_oracle_along_the_best_path(name):
    from paper_2107_11810_gb300 import vote as v
    p = MAKE[name]()
    s = v.Solver(p.family, p.eps, p.bounds)
    L, Lj = s.levels()
    best = s.solve(torch.from_numpy(np.ascontiguousarray(p.params)).cuda())["best_leaf"]
    rng = np.random.default_rng(4)
    for n in (1, 1023, 1024, 1025, p.params.shape[1]):
        prm = np.ascontiguousarray(p.params[:, :n])
        t = torch.from_numpy(prm).cuda()
        for level in range(0 if n > 1025 else L, L + 1):
            at = [int(best[j]) >> max(0, int(Lj[j]) - level) for j in range(p.d)]
            beside = [min(max(x + int(rng.integers(-1, 2)), 0), 2 ** min(level, int(Lj[j])) - 1) for j, x in enumerate(at)]
            for coords in (at, beside):
                ub, lb, reach = s.cell_counts(t, level, coords, want_reach=True)
                oub, olb, oreach = oracle.cell_counts(p.family, p.eps, p.bounds, prm, level, coords, want_reach=True)
                assert (ub, lb) == (oub, olb)
                assert np.array_equal(v.mask_words_to_numpy(reach), oreach)


# residuals at x of the dependent coordinates, the parameter row each moves one to one with
# (of its opposite sign), and the essential parameters' part of the radius per half-width
RESIDUAL = {
    "line2d": lambda q, x: ([x[1] - (q[1] - q[0] * x[0])], [1], [np.abs(q[0])]),
    "rays3d": lambda q, x: ([x[1] - (q[0] * x[0] + q[1]), x[2] - (q[2] * x[0] + q[3])], [1, 3],
                            [np.abs(q[0]), np.abs(q[2])]),
    "pose3dof": lambda q, x: ([x[1] - (q[0] - (q[2] * np.cos(x[0]) - q[3] * np.sin(x[0]))),
                               x[2] - (q[1] - (q[2] * np.sin(x[0]) + q[3] * np.cos(x[0])))], [0, 1],
                              [np.hypot(q[2], q[3])] * 2),
}


def surfaces_beyond_reach(name, p, leaf, n, rng):
    """Surfaces whose residual at the leaf's centre exceeds its whole radius (canonization
    error included) by 2 to 6 snap steps in the first dependent coordinate."""
    from paper_2107_11810_gb300 import vote as v
    k = v.level_constants(p.family, p.eps, p.bounds)
    lo, hi = np.asarray(p.bounds, dtype=float).reshape(-1, 2).T
    h = (hi - lo) * 2.0 ** -(k["Lj"] + 1.0)
    x = lo + (2 * np.asarray(leaf) + 1) * h
    q = p.params[:, rng.integers(0, p.params.shape[1], n)]
    r, rows, lam = RESIDUAL[name](q, x)
    nd = len(rows)
    R = p.eps[-nd] + h[-nd] + lam[0] * h[0] + k["A"][-1][0]
    for j in range(nd):
        want = (R + k["s_f"][0] * rng.uniform(2.0, 6.0, n)) * rng.choice([-1.0, 1.0], n) if j == 0 else 0.0
        q[rows[j]] += r[j] - want
    return np.ascontiguousarray(q)


@pytest.mark.parametrize("name", sorted(RESIDUAL))
def test_replay_keeps_surfaces_that_pass_by_the_canonization_error(name):
    """The snaps on the way move a residual by up to the accumulated canonization error, so
    some surfaces just beyond a leaf's radius pass every step, and count."""
    from paper_2107_11810_gb300 import vote as v
    p = MAKE[name]()
    s = v.Solver(p.family, p.eps, p.bounds)
    leaf = s.solve(torch.from_numpy(np.ascontiguousarray(p.params)).cuda())["best_leaf"]
    prm = surfaces_beyond_reach(name, p, leaf, 400_000, np.random.default_rng(9))
    L, _ = s.levels()
    oub, olb, oreach = oracle.cell_counts(p.family, p.eps, p.bounds, prm, L, leaf, want_reach=True)
    assert oub > 0                               # some do pass
    ub, lb, reach = s.cell_counts(torch.from_numpy(prm).cuda(), L, leaf, want_reach=True)
    assert (ub, lb) == (oub, olb)
    assert np.array_equal(v.mask_words_to_numpy(reach), oreach)
