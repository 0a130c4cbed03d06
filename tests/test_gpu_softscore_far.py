"""Soft score: surfaces that contribute exactly 0 are left out by an FP32 test; what it
must not leave out (residuals just inside, values outside FP32's range, NaN and infinite
inputs or gradients) goes through the FP64 evaluation as before."""
import math

import numpy as np
import pytest

from paper_2107_11810_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = 0.25


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2107_11810_gb300 import build
    build.build()


def line_score(xy, mask=None, upstream=1.0):
    """Score and gradients of lines b = y - x m at (m, b) = (0.5, 1)."""
    from paper_2107_11810_gb300 import vote
    from paper_2107_11810_gb300.softscore import SoftScore
    s = vote.Solver(inputs.LINE2D, [0.01, 0.01], [-1.0, 1.0, -1.0, 2.0])
    q = torch.tensor(np.ascontiguousarray(xy), dtype=torch.float64, device="cuda", requires_grad=True)
    p = torch.tensor([0.5, 1.0], dtype=torch.float64, device="cuda", requires_grad=True)
    out = SoftScore.apply(p, q, s, mask, [TOL])
    out.backward(torch.tensor(upstream, dtype=torch.float64, device="cuda"))
    return float(out.detach()), p.grad.cpu().numpy(), q.grad.cpu().numpy()


def at(u, x):
    """The line through x whose residual is u tolerances."""
    return np.stack([x, 1.0 + 0.5 * x - TOL * u])


@pytest.mark.parametrize("n", [1, 31, 32, 33, 1000, 40001])
@pytest.mark.parametrize("share", [0.0, 0.03, 0.5, 1.0])
def test_near_surfaces_among_far_ones(n, share):
    # every warp queues a different number of surfaces; n covers partial words and warps
    rng = np.random.default_rng(n)
    x = rng.uniform(-3.0, 3.0, n)
    near = rng.uniform(0.0, 1.0, n) < share
    u = np.where(near, rng.uniform(-3.0, 3.0, n), rng.choice([-1.0, 1.0], n) * rng.uniform(39.0, 1e6, n))
    S, gp, gq = line_score(at(u, x))
    r = 1.0 - (at(u, x)[1] - 0.5 * x)
    k = np.exp(-0.5 * (r / TOL) ** 2)
    dr = -k * r / TOL ** 2
    # sums of at most n terms below max|term| in any order: n 2^-53 relative to sum|.|
    eps = n * 2.0 ** -52 + 1e-13
    assert abs(S - k.sum()) <= eps * k.sum()
    for got, want in zip(gp, [dr * x, dr]):
        assert abs(got - want.sum()) <= eps * np.abs(want).sum()
    assert np.all(gq[:, ~near] == 0.0)
    assert np.allclose(gq, np.stack([dr * 0.5, -dr]), rtol=1e-12, atol=0.0)


def test_smallest_contributions_are_kept():
    u = np.array([38.0, 38.5, 38.59, 38.7])          # exp: 3e-314, 1e-322, 5e-324, 0
    S, _, _ = line_score(at(u[:1], np.zeros(1)))
    assert S == pytest.approx(math.exp(-0.5 * 38.0 ** 2), rel=1e-6)
    for v in u[1:3]:
        assert line_score(at(np.array([v]), np.zeros(1)))[0] > 0.0
    assert line_score(at(u[3:] + 0.2, np.zeros(1)))[0] == 0.0


@pytest.mark.parametrize("value", [math.nan, math.inf, 1e200, 1e-310, 4e38])
@pytest.mark.parametrize("masked", [False, True])
def test_values_outside_fp32_take_the_fp64_path(value, masked):
    x = np.linspace(-1.0, 1.0, 70)
    xy = at(np.full(70, 0.5), x)
    xy[1, 37] = value
    words = np.full(3, -1, np.int32)
    words[1] = ~(1 << 5)                              # surface 37 has weight 0
    mask = torch.from_numpy(words).cuda() if masked else None
    S, gp, gq = line_score(xy, mask)
    r = 1.0 - (xy[1] - 0.5 * x)
    w = np.ones(70)
    if masked:
        w[37] = 0.0
    with np.errstate(all="ignore"):
        k = w * np.exp(-0.5 * (r / TOL) ** 2)
        want = k.sum()
    assert (math.isnan(S) and math.isnan(want)) or S == pytest.approx(want, rel=1e-12)


def test_infinite_upstream_gradient_is_not_hidden_by_far_surfaces():
    _, gp, gq = line_score(at(np.array([100.0, 0.5]), np.array([0.1, 0.2])), upstream=math.inf)
    assert np.isnan(gp).all() and np.isnan(gq[:, 0]).all()
