"""Where device memory is short a solve gives back what it holds and is repeated depth first in
small steps, and a batch goes on with fewer workers: the results are the same.  Free memory is
bounded by a tensor that takes the rest.  The 6DoF search below holds 39 GB when it can and
needs 6 GB; eight affine searches at a time hold 10 GB each and need 3.5 GB."""
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


def take_all_but(free_bytes):
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    return torch.empty(max(free - free_bytes, 1), dtype=torch.uint8, device="cuda")


def result(v, r):
    return r["depth"], tuple(r["best_leaf"]), tuple(r["best_point"]), v.mask_words_to_numpy(r["mask"]).tobytes()


def test_solve_repeats_with_less_memory():
    from paper_2107_11810_gb300 import vote as v
    p = inputs.pose6dof()
    t = torch.from_numpy(np.ascontiguousarray(p.params)).cuda()
    s = v.Solver(p.family, p.eps, p.bounds)
    want = result(v, s.solve(t))
    s.close()
    rest = take_all_but(16 << 30)
    s = v.Solver(p.family, p.eps, p.bounds)
    for _ in range(2):                           # the context stays usable
        assert result(v, s.solve(t)) == want
    pinned = torch.from_numpy(p.params).pin_memory()
    h = s.solve_host(pinned)
    assert (h["depth"], tuple(h["best_leaf"])) == want[:2]
    del rest
    torch.cuda.empty_cache()
    assert result(v, s.solve(t)) == want


def test_batch_goes_on_with_fewer_workers():
    from paper_2107_11810_gb300 import vote as v
    probs = [inputs.affine4d(seed=2107 + i) for i in range(10)]
    p0 = probs[0]
    assert all(np.array_equal(p.bounds, p0.bounds) for p in probs)
    s = v.Solver(p0.family, p0.eps, p0.bounds)
    want = [result(v, s.solve(torch.from_numpy(np.ascontiguousarray(p.params)).cuda())) for p in probs]
    s.close()
    flat, offs = v.pack_batch([p.params for p in probs])
    flat = torch.from_numpy(flat).cuda()
    rest = take_all_but(16 << 30)
    s = v.Solver(p0.family, p0.eps, p0.bounds)
    s.set_option(v.VOTE_OPT_BATCH_WORKERS, 8)
    r = s.solve_batched((flat, offs))
    masks = v.mask_words_to_numpy(r["masks"])
    for b, p in enumerate(probs):
        w = r["word_offsets"][b]
        assert (r["depths"][b], tuple(r["best_leaves"][b]), tuple(r["best_points"][b]),
                masks[w:w + (p.n + 31) // 32].tobytes()) == want[b]
    assert np.all(r["latency_ms"] > 0)
    del rest
