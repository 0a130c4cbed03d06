"""The lift rounds a surface's fields to whole steps and refuses values of 2^30 steps and more.
On the CPU: the kernel's own function, compiled for the host with overflow trapping, over values
on both sides of the limit and beyond the integer range, where the conversion saturates.  On
the GPU: the same limit through the solver."""
import os
import re
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_2107_11810_gb300", "csrc", "gv_kernels.cu")
LIMIT = 2.0 ** 30
INSIDE = [0.0, 0.49, -0.5, 1.5, 12345.0, LIMIT - 1.0, -(LIMIT - 1.0), LIMIT - 0.75, 5e-324]
OUTSIDE = [LIMIT, -LIMIT, LIMIT - 0.5, 2.0 ** 31 - 1.0, 2.0 ** 31, -2.0 ** 31, 2.0 ** 31 + 1.0, -2.0 ** 31 - 1.0,
           2.0 ** 32, 2.0 ** 52, -2.0 ** 62, 1e300, -1e300, float("inf"), float("-inf"), float("nan")]

HOST = """
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#define __device__
#define __forceinline__ inline
static double dmul(double a, double b) { return a * b; }
static int __double2hiint(double x) { int64_t b; std::memcpy(&b, &x, 8); return (int)(b >> 32); }
static int __double2int_rn(double x) {                      // saturates, NaN gives the smallest
    const double r = std::nearbyint(x);
    if (r >= 2147483647.0) return 2147483647;
    return r > -2147483648.0 ? (int)r : -2147483647 - 1;
}
FUNCTION
int main(int argc, char **argv) {
    for (int i = 1; i < argc; ++i) {
        bool bad = false;
        const int q = lift_q(std::strtod(argv[i], nullptr), 1.0, bad);
        std::printf("%d %d\\n", q, (int)bad);
    }
}
"""


def test_lift_refuses_out_of_range_fields_without_overflow(tmp_path):
    text = open(SRC).read()
    f = re.search(r"^__device__ __forceinline__ int lift_q\(.*?^}$", text, re.S | re.M).group(0)
    src, exe = tmp_path / "lift.cpp", tmp_path / "lift"
    src.write_text(HOST.replace("FUNCTION", f))
    subprocess.run(["g++", "-std=c++17", "-O2", "-fsanitize=signed-integer-overflow",
                    "-fsanitize-undefined-trap-on-error", str(src), "-o", str(exe)], check=True)
    values = INSIDE + OUTSIDE
    out = subprocess.run([str(exe)] + [repr(v) for v in values], capture_output=True, text=True)
    assert out.returncode == 0                               # no signed overflow
    got = [tuple(map(int, line.split())) for line in out.stdout.splitlines()]
    want = [(int(np.rint(v)), 0) for v in INSIDE] + [(0, 1)] * len(OUTSIDE)
    assert got == want


@pytest.mark.gpu
@pytest.mark.parametrize("steps", [LIMIT - 1.0, LIMIT, 2.0 ** 31 - 1.0, 2.0 ** 31, 2.0 ** 32 + 4096.0, 1e280])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_solver_refuses_out_of_range_surfaces(steps, sign):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2107_11810_gb300 import build, inputs, vote
    build.build()
    p = inputs.line2d(n=40, inlier_frac=0.5, eps=0.02, seed=81)
    s_f = vote.level_constants(p.family, p.eps, p.bounds)["s_f"][0]
    c = 0.5 * (p.bounds[2] + p.bounds[3])                    # the line's residual at the domain's centre: y - c
    params = p.params.copy()
    params[:, 7] = 0.0, sign * steps * s_f + c
    s = vote.Solver(p.family, p.eps, p.bounds)
    t = torch.from_numpy(np.ascontiguousarray(params)).cuda()
    if steps < LIMIT:
        assert s.solve(t)["depth"] > 0
    else:
        with pytest.raises(vote.VoteError) as e:
            s.solve(t)
        assert e.value.code == 1                             # VOTE_EINVAL
