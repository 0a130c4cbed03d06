"""Levels expanded one after the other without the host in between (small levels, from the
root): same results and same counters whatever the context had allocated before, whether
the levels fit, outgrow the room kept for them or run out of cells, and the same results as
the step-by-step path (taken while kernels are timed)."""
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


# sizes: one surface, a tile and its neighbours, and (last of each) levels beyond the
# 131,072 record slots that a level is first given
PROBLEMS = [("line2d", n) for n in (1, 31, 32, 33, 500, 20000)] + [("pose3dof", n) for n in (64, 9000)] + \
           [("pose6dof", n) for n in (7, 300)]


def make(name, n):
    if name == "line2d":
        return inputs.line2d(n=n, inlier_frac=0.2, eps=0.02, seed=41)
    if name == "pose3dof":
        return inputs.pose3dof(n=n, inlier_frac=0.2, eps_xy=1.0, eps_yaw_deg=2.0, seed=42)
    return inputs.pose6dof(n=n, inlier_frac=0.2, prior_deg=5.0, levels=4, seed=43)


@pytest.mark.parametrize("precision", [1, 0])
@pytest.mark.parametrize("name,n", PROBLEMS)
def test_chain_equals_oracle_and_stepwise(name, n, precision):
    from paper_2107_11810_gb300 import vote as v
    p = make(name, n)
    o = oracle.solve(p.family, p.eps, p.bounds, p.params)
    t = torch.from_numpy(np.ascontiguousarray(p.params)).cuda()
    s = v.Solver(p.family, p.eps, p.bounds, precision=precision)
    counters = []
    for timing in (0, 0, 1, 0):                  # first pass, repeated, stepwise, chain again
        s.set_option(v.VOTE_OPT_KERNEL_TIMING, timing)
        r = s.solve(t)
        assert r["depth"] == o["depth"]
        assert np.array_equal(r["best_leaf"], o["best_leaf"])
        assert np.array_equal(r["best_point"], o["best_point"])
        assert np.array_equal(v.mask_words_to_numpy(r["mask"]), o["mask"])
        if not timing:
            q = s.stats()
            counters.append([q[k] for k in ("tests", "cells", "chunks", "launches", "rechecks", "records")])
    assert counters[0] == counters[1] == counters[2]


def test_chain_with_the_depth_as_lower_bound():
    from paper_2107_11810_gb300 import vote as v
    p = make("line2d", 500)
    o = oracle.solve(p.family, p.eps, p.bounds, p.params)
    s = v.Solver(p.family, p.eps, p.bounds)
    s.set_option(v.VOTE_OPT_INITIAL_LB, o["depth"])          # only the winning path survives
    r = s.solve(torch.from_numpy(np.ascontiguousarray(p.params)).cuda())
    assert r["depth"] == o["depth"]
    assert np.array_equal(v.mask_words_to_numpy(r["mask"]), o["mask"])
