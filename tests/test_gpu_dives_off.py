"""Without dives (VOTE_OPT_DIVE 0) the search goes depth first: the leaves below its first
steps are what raises the pruning bound.  Opened level by level it finds no leaf until every
level above is expanded: point sets then tested 7.0 times the pairs of the search with dives
and held 2.7e8 record slots of one level, against 2.1 times and 5.4e7 depth first in steps of
2^23 records.  The bounds below lie between the two."""
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


@pytest.mark.parametrize("chunk", [None, 1 << 23])
def test_without_dives_leaves_are_reached_early(chunk):
    from paper_2107_11810_gb300 import vote as v
    p = inputs.pointset2d(m=150, eps=0.02, seed=9)
    t = torch.from_numpy(np.ascontiguousarray(p.params)).cuda()
    got, stats = [], []
    for dive in (2, 0):
        s = v.Solver(p.family, p.eps, p.bounds, chunk_records=chunk)
        s.set_option(v.VOTE_OPT_DIVE, dive)
        r = s.solve(t)
        got.append((r["depth"], tuple(r["best_leaf"]), v.mask_words_to_numpy(r["mask"]).tobytes()))
        stats.append(s.stats())
    assert got[0] == got[1]
    assert stats[1]["tests"] <= 4 * stats[0]["tests"]
    assert stats[1]["peak_records"] <= 180_000_000
