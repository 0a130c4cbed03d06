"""The count pass leaves a cell once none of its children can reach the pruning threshold:
same results and counters as without (a trace lists every child, so it tests them all), for
cells that one warp counts and cells that many share, and with steps that split a level."""
import numpy as np
import pytest

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
    "line2d": lambda: inputs.line2d(n=200_003, inlier_frac=0.05, eps=0.002, seed=61),
    "plane3d_few": lambda: inputs.plane3d(n=3001, inlier_frac=0.1, eps=0.01, sigma=0.002, seed=62),
    "plane3d_many": lambda: inputs.plane3d(n=150_001, inlier_frac=0.03, eps=0.05, sigma=0.005, seed=63),
    "pose3dof": lambda: inputs.pose3dof(n=120_007, inlier_frac=0.01, eps_xy=0.5, eps_yaw_deg=1.0, seed=64),
    "rays3d": lambda: inputs.rays3d(n=50_001, inlier_frac=0.02, eps=0.002, seed=65),
    "affine4d": lambda: inputs.affine4d(n=4001, inlier_frac=0.05, eps=0.03, noise=0.005, seed=66),
    "pointset2d": lambda: inputs.pointset2d(m=150, eps=0.02, seed=67),
    "pose6dof": lambda: inputs.pose6dof(n=2001, inlier_frac=0.05, prior_deg=5.0, levels=6, seed=68),
    "radial5dof": lambda: inputs.radial5dof(n=2001, inlier_frac=0.05, prior_deg=5.0, levels=6, seed=69),
}


@pytest.mark.parametrize("name", sorted(PROBLEMS))
@pytest.mark.parametrize("chunk", [None, 100_000])
def test_leaving_cells_early_changes_nothing(name, chunk):
    from paper_2107_11810_gb300 import vote as v
    p = PROBLEMS[name]()
    t = torch.from_numpy(np.ascontiguousarray(p.params)).cuda()
    got = []
    for trace in (0, 1):
        s = v.Solver(p.family, p.eps, p.bounds)
        if chunk:
            s.set_option(v.VOTE_OPT_CHUNK_RECORDS, chunk)
        s.set_option(v.VOTE_OPT_TRACE_CAP, trace)
        for _ in range(2):                       # first pass and repeated
            r = s.solve(t)
            got.append((r["depth"], tuple(r["best_leaf"]), v.mask_words_to_numpy(r["mask"]).tobytes()))
    assert got[0] == got[1] == got[2] == got[3]
    assert got[0][0] > 0
