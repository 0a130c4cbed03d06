"""The work that a user of this framework has it do, as cases for timing.

A case names a generator of ``paper_2107_11810_gb300.inputs``, its sizes and the call:

* ``solve``      one complete search on device buffers: lift, canonization, proximity
                 test, pruning and splitting down to the leaves, inlier mask;
* ``solve_host`` the same on pinned host buffers, copies inside the call;
* ``batch``      independent searches in one call (``vote_solve_batched``);
* ``softscore``  the soft inlier score with its gradients by the point and by every
                 surface parameter (forward and backward of the refinement).

The sizes are those of the benchmark workloads where one pass of them takes less
than two seconds; the plane workload is split into its two halves (its point count at
a coarser eps, its eps at fewer points), and the pose workloads use the +-5 deg prior.
"""
import math

import numpy as np
import torch

from paper_2107_11810_gb300 import inputs, softscore, vote

# children per cell and rough FP32 operations of one (child, surface) test, input rows
FAMILY = {"line2d": (4, 7, 2), "plane3d": (8, 10, 3), "pose3dof": (8, 14, 4), "rays3d": (8, 10, 4),
          "pointset2d": (16, 10, 4), "affine4d": (16, 10, 4), "pose6dof": (64, 30, 5), "radial5dof": (32, 17, 5)}
ARGS = ("n", "m", "eps", "eps_xy", "eps_yaw_deg", "inlier_frac", "noise", "sigma", "prior_deg", "levels")


def listed():
    return [
        # a handful of edge points from one image patch: launches and round trips count
        {"name": "line2d_n500", "call": "solve", "make": "line2d", "n": 500, "inlier_frac": 0.2, "eps": 0.01},
        # line fitting in one image (the smallest benchmark workload)
        {"name": "line2d_n10k", "call": "solve", "make": "line2d", "n": 10_000, "inlier_frac": 0.1, "eps": 0.01},
        # intersection of rays, a bundle of viewing rays (Sec. 4.3)
        {"name": "rays3d_n100k", "call": "solve", "make": "rays3d", "n": 100_000, "inlier_frac": 0.02, "eps": 0.002},
        # large-scale localisation with known gravity: one query with a million matches
        {"name": "pose3dof_n1m", "call": "solve", "make": "pose3dof", "n": 1_000_000, "inlier_frac": 0.01,
         "eps_xy": 0.25, "eps_yaw_deg": 0.5},
        # a server's batch of queries of very different, ragged sizes
        {"name": "pose3dof_batch24", "call": "batch", "make": "pose3dof", "num": 24, "n_lo": 1000,
         "n_hi": 100_000, "sizes": 3},
        # plane fitting at the benchmark's eps: deep search, few surfaces in a cell
        {"name": "plane3d_n10k_fine", "call": "solve", "make": "plane3d", "n": 10_000, "inlier_frac": 0.05,
         "eps": 0.005},
        # plane fitting with the benchmark's point count: many surfaces in every cell
        {"name": "plane3d_n1m_coarse", "call": "solve", "make": "plane3d", "n": 1_000_000, "inlier_frac": 0.02,
         "eps": 0.03},
        # calibrated camera with a rotation prior (an IMU): 64 children per cell
        {"name": "pose6dof_n5000", "call": "solve", "make": "pose6dof", "n": 5000, "inlier_frac": 0.05,
         "prior_deg": 5.0, "levels": 7},
        # radial camera with unknown focal length: 32 children per cell
        {"name": "radial5dof_n5000", "call": "solve", "make": "radial5dof", "n": 5000, "inlier_frac": 0.05,
         "prior_deg": 5.0, "levels": 7},
        # alignment of two point sets without correspondences (every pair is a surface)
        {"name": "pointset2d_m300", "call": "solve", "make": "pointset2d", "m": 300, "eps": 0.01},
        # hyperplanes in 4-space
        {"name": "affine4d_n10k", "call": "solve", "make": "affine4d", "n": 10_000, "inlier_frac": 0.05,
         "eps": 0.02},
        # gradient step of the refinement over all matches of the large query
        {"name": "softscore_pose3dof_n1m", "call": "softscore", "make": "pose3dof", "n": 1_000_000,
         "inlier_frac": 0.01, "eps_xy": 0.25, "eps_yaw_deg": 0.5},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges.  The cost of a search grows with n eps^-k, so
    the finest eps go with fewer surfaces."""
    call = rng.choice(["solve", "solve", "solve", "solve", "solve", "solve_host", "batch", "softscore"])
    if call == "batch":
        return {"call": call, "make": "pose3dof", "num": rng.randint(2, 32), "n_lo": _log(rng, 300, 3000),
                "n_hi": _log(rng, 10_000, 100_000), "sizes": rng.randint(0, 1000)}
    make = rng.choice(sorted(set(FAMILY) - {"radial5dof"} if call == "softscore" else FAMILY))
    case = {"call": call, "make": make}
    if make == "line2d":
        case.update(n=_log(rng, 100, 100_000), eps=round(math.exp(rng.uniform(math.log(0.005), math.log(0.03))), 5))
    elif make == "rays3d":
        case.update(n=_log(rng, 500, 300_000), eps=round(math.exp(rng.uniform(math.log(0.002), math.log(0.02))), 5))
    elif make == "pose3dof":
        case.update(n=_log(rng, 500, 1_000_000), eps_xy=rng.choice([0.25, 0.4, 0.5, 1.0]),
                    eps_yaw_deg=rng.choice([0.5, 0.7, 1.0, 2.0]))
    elif make == "plane3d":
        n = _log(rng, 300, 500_000)
        e0 = max(0.005, 0.005 * math.sqrt(n / 25_000.0))
        case.update(n=n, eps=round(math.exp(rng.uniform(math.log(e0), math.log(0.06))), 5))
    elif make == "pointset2d":
        case.update(m=_log(rng, 8, 350), eps=round(math.exp(rng.uniform(math.log(0.01), math.log(0.05))), 5))
    elif make == "affine4d":
        case.update(n=_log(rng, 200, 20_000), eps=round(math.exp(rng.uniform(math.log(0.03), math.log(0.1))), 5))
    else:
        case.update(n=_log(rng, 200, 8000), prior_deg=rng.choice([2.5, 4.0, 5.0]), levels=rng.choice([5, 6, 7]))
    if make != "pointset2d":
        case["inlier_frac"] = round(rng.uniform(0.02, 0.2), 3)
    return case


def _batch_sizes(case):
    """Surfaces and inlier ratio of every problem of a batch, n log-uniform as in the benchmark's batch."""
    rng = np.random.default_rng(case["sizes"])
    n = np.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), case["num"]))
    return [(int(round(x)), f) for x, f in zip(n, rng.uniform(0.005, 0.05, case["num"]))]


def _problem(case, seed):
    """The case's synthetic scene (host arrays)."""
    return getattr(inputs, case["make"])(seed=seed, **{k: case[k] for k in ARGS if k in case})


def prepare(case, seed):
    state = {"call": case["call"]}
    if case["call"] == "batch":
        rng = np.random.default_rng(seed)
        probs = [inputs.pose3dof(n=n, inlier_frac=f, rng=rng) for n, f in _batch_sizes(case)]
        p = probs[0]
        flat, offsets = vote.pack_batch([q.params for q in probs])
        state["blocks"] = (torch.from_numpy(flat).cuda(), offsets)
    else:
        p = _problem(case, seed)
        host = torch.from_numpy(p.params)
        state["surfaces"] = host.pin_memory() if case["call"] == "solve_host" else host.cuda()
    state["solver"] = vote.Solver(p.family, p.eps, p.bounds, stream=torch.cuda.current_stream())
    if case["call"] == "softscore":
        # the refinement starts at the voted leaf's centre, here a quarter of eps off the
        # planted solution; every surface has weight 1
        state["point"] = torch.from_numpy(p.truth + 0.25 * p.eps).cuda().requires_grad_(True)
        state["surfaces"].requires_grad_(True)
    return state


def run(state):
    call, s = state["call"], state["solver"]
    if call == "solve":
        return s.solve(state["surfaces"])
    if call == "solve_host":
        return s.solve_host(state["surfaces"])
    if call == "batch":
        r = s.solve_batched(state["blocks"])
        return {k: r[k] for k in ("best_points", "best_leaves", "depths", "masks")}
    point, surfaces = state["point"], state["surfaces"]
    score = softscore.soft_score(point, surfaces, s)
    grad_point, grad_surfaces = torch.autograd.grad(score, (point, surfaces))
    return {"score": score.detach(), "grad_point": grad_point, "grad_surfaces": grad_surfaces}


def work(case):
    """Inputs read once and results written once; operations: every surface lifted and
    tested once against the children of the root, which no search can leave out (how
    many cells below it have to be opened depends on the data)."""
    children, ops, rows = FAMILY[case["make"]]
    if case["call"] == "batch":
        n = sum(size for size, _ in _batch_sizes(case))
    else:
        n = case["m"] ** 2 if "m" in case else case["n"]
    if case["call"] == "softscore":
        return {"bytes": 2 * 8 * rows * n, "flops": 2 * 40 * n}
    return {"bytes": 8 * rows * n + n // 8, "flops": children * ops * n}


def exact(case, seed):
    """The soft score and its gradients by torch's autograd in 64 bits from the surface
    equations in their global form.  The searches return integers (depth, leaf, mask) and
    the leaf's centre."""
    if case["call"] != "softscore":
        return None
    p = _problem(case, seed)
    q = torch.from_numpy(p.params).cuda().requires_grad_(True)
    x = torch.from_numpy(p.truth + 0.25 * p.eps).cuda().requires_grad_(True)
    make = case["make"]
    if make == "line2d":
        r = [x[1] - (q[1] - q[0] * x[0])]
    elif make == "plane3d":
        r = [x[2] - (q[0] * (torch.sin(x[0]) * torch.cos(x[1])) + q[1] * (torch.sin(x[0]) * torch.sin(x[1]))
                     + q[2] * torch.cos(x[0]))]
    elif make == "pose3dof":
        c, s = torch.cos(x[0]), torch.sin(x[0])
        r = [x[1] - (q[0] - (q[2] * c - q[3] * s)), x[2] - (q[1] - (q[2] * s + q[3] * c))]
    elif make == "rays3d":
        r = [x[1] - (q[0] * x[0] + q[1]), x[2] - (q[2] * x[0] + q[3])]
    elif make == "affine4d":
        r = [x[3] - (q[3] - (x[0] * q[0] + x[1] * q[1] + x[2] * q[2]))]
    elif make == "pointset2d":
        n2, ex, ey = q[0] * q[0] + q[1] * q[1], q[2] - x[0], q[3] - x[1]
        r = [x[2] - (q[0] * ex + q[1] * ey) / n2, x[3] - (q[1] * ex - q[0] * ey) / n2]
    else:                                              # pose6dof: X = R(phi) w + (x, y, z)
        zero = torch.zeros((), dtype=torch.float64, device="cuda")
        K = torch.stack([torch.stack([zero, -x[2], x[1]]), torch.stack([x[2], zero, -x[0]]),
                         torch.stack([-x[1], x[0], zero])])
        X = torch.linalg.matrix_exp(K) @ q[:3]
        r = [x[4] - (q[3] * (X[2] + x[3]) - X[0]), x[5] - (q[4] * (X[2] + x[3]) - X[1])]
    tol = p.eps[len(p.eps) - len(r):]
    u2 = sum((ri / float(t)) ** 2 for ri, t in zip(r, tol))
    score = torch.exp(-0.5 * u2).sum()
    grad_point, grad_surfaces = torch.autograd.grad(score, (x, q))
    return {"score": score.detach(), "grad_point": grad_point, "grad_surfaces": grad_surfaces}
