"""Counters of work done: pairs decided (stats), pairs evaluated (without those of cells that
the count pass left), and the bytes of the count and emit passes, which follow the second.
With steps of 2^22 records a warp owns cells of up to 16 tiles and shares larger ones, with the
default steps cells of up to 64; steps of 100,000 records give a warp two tiles, of which it
can hardly leave any."""
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
    "plane3d_few": lambda: inputs.plane3d(n=20_011, inlier_frac=0.05, eps=0.02, seed=6),
    "plane3d_many": lambda: inputs.plane3d(n=150_001, inlier_frac=0.03, eps=0.05, sigma=0.005, seed=63),
    "affine4d": lambda: inputs.affine4d(n=5003, inlier_frac=0.05, eps=0.03, seed=10),
    "radial5dof": lambda: inputs.radial5dof(n=2003, prior_deg=5.0, levels=6, seed=12),
}


@pytest.mark.parametrize("name", sorted(PROBLEMS))
@pytest.mark.parametrize("chunk", [None, 1 << 22, 100_000])
def test_evaluated_pairs(name, chunk):
    from paper_2107_11810_gb300 import vote as v
    if name in ("affine4d", "plane3d_few") and chunk == 100_000:
        pytest.skip("hundreds of thousands of steps")
    p = PROBLEMS[name]()
    t = torch.from_numpy(np.ascontiguousarray(p.params)).cuda()
    s = v.Solver(p.family, p.eps, p.bounds, chunk_records=chunk)
    s.solve(t)
    assert s.evaluated_tests() == -1                         # not counted
    s.set_option(v.VOTE_OPT_KERNEL_TIMING, 1)
    keep = []
    for _ in range(2):
        s.solve(t)
        st = s.stats()
        keep.append([st[k] for k in ("tests", "records", "cells", "leaves", "chunks")])
        assert 0 < s.evaluated_tests() <= st["tests"]
        assert chunk == 100_000 or s.evaluated_tests() < st["tests"]      # cells were left
    assert keep[0] == keep[1]
    if chunk is None:
        s.set_option(v.VOTE_OPT_TRACE_CAP, 1)                # every child is listed: none is left
        s.solve(t)
        assert s.evaluated_tests() == s.stats()["tests"]


def test_batch_and_empty_problems():
    from paper_2107_11810_gb300 import vote as v
    p = inputs.radial5dof(n=2003, prior_deg=5.0, levels=6, seed=12)
    s = v.Solver(p.family, p.eps, p.bounds)
    s.set_option(v.VOTE_OPT_KERNEL_TIMING, 1)
    flat, offs = v.pack_batch([p.params, p.params[:, :0], p.params])
    s.solve_batched((torch.from_numpy(flat).cuda(), offs))
    assert 0 < s.evaluated_tests() < s.stats()["tests"]
    s.solve(torch.empty((5, 0), dtype=torch.float64, device="cuda"))
    assert s.evaluated_tests() == 0


def test_bytes_follow_the_work_done():
    from paper_2107_11810_gb300 import vote as v
    p = PROBLEMS["plane3d_few"]()
    t = torch.from_numpy(np.ascontiguousarray(p.params)).cuda()
    s = v.Solver(p.family, p.eps, p.bounds)
    s.set_option(v.VOTE_OPT_KERNEL_TIMING, 1)
    s.solve(t)
    L, Lj = s.levels()
    slots = s.level_stats()["records"].astype(float)
    ns = np.array([2.0 ** np.sum(Lj > l) for l in range(L)])
    words = np.where(np.arange(L) == 0, 4, 2)                # 16-bit fields from level 1 on
    every = slots * 4 * words + slots / 32 * 4 * ns          # records and ballots of every tile
    count, emit = s.kernel_times()["test_count"][2], s.kernel_times()["test_emit"][2]
    assert 0 < count < every.sum()
    # the share left is that of the pairs, up to the cells' last tiles
    share = s.evaluated_tests() / s.stats()["tests"]
    assert abs(count / every.sum() - share) < 0.1
    # child records written once (dives copy theirs, so at least those expanded below the root
    # and not copied); of the records read only tiles of cells with surviving children
    written = (slots[1:] * 8).sum()
    assert 0 < emit < every[:-1].sum() + written
