"""The search order (dives along the cells with the largest bounds, level stores that are
appended to) never changes a result: small steps make every dive select, gather and
append, in both record formats and with grouping's multiplicities."""
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


PROBLEMS = {
    "line2d": lambda: inputs.line2d(n=3000, inlier_frac=0.2, eps=0.01, seed=31),
    "plane3d": lambda: inputs.plane3d(n=2011, inlier_frac=0.1, eps=0.05, sigma=0.002, seed=32),
    "pose3dof": lambda: inputs.pose3dof(n=1500, inlier_frac=0.2, eps_xy=1.0, eps_yaw_deg=2.0, seed=33),
    "pointset2d": lambda: inputs.pointset2d(m=45, eps=0.05, seed=34),
    "pose6dof": lambda: inputs.pose6dof(n=400, inlier_frac=0.2, prior_deg=5.0, levels=4, seed=35),
}


@pytest.mark.parametrize("name", sorted(PROBLEMS))
@pytest.mark.parametrize("chunk", [500, 4096])
@pytest.mark.parametrize("precision,group", [(1, 0), (1, 1), (0, 0)])
def test_dives_and_appended_levels_do_not_change_results(name, chunk, precision, group):
    from paper_2107_11810_gb300 import vote as v
    p = PROBLEMS[name]()
    o = oracle.solve(p.family, p.eps, p.bounds, p.params)
    t = torch.from_numpy(np.ascontiguousarray(p.params)).cuda()
    tests = set()
    for dive in (0, 2, 2):
        s = v.Solver(p.family, p.eps, p.bounds, precision=precision, chunk_records=chunk)
        s.set_option(v.VOTE_OPT_DIVE, dive)
        s.set_option(v.VOTE_OPT_GROUP, group)
        r = s.solve(t)
        assert r["depth"] == o["depth"]
        assert np.array_equal(r["best_leaf"], o["best_leaf"])
        assert np.array_equal(v.mask_words_to_numpy(r["mask"]), o["mask"])
        if dive:
            tests.add(s.stats()["tests"])
    assert len(tests) == 1                       # the order is a function of the input alone
