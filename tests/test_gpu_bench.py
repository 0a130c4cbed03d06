"""bench.py times the call that a user makes: its warm-up, timed and end-to-end solves run with
kernel timing off (which takes small searches off their usual path); the kernel classes come
from a solve of their own."""
import json
import os
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_timed_solves_take_the_usual_path(monkeypatch, capsys):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2107_11810_gb300 import build, vote
    build.build()
    monkeypatch.syspath_prepend(ROOT)
    import bench
    calls, timing = [], [0]

    def set_option(self, key, value, f=vote.Solver.set_option):
        if key == vote.VOTE_OPT_KERNEL_TIMING:
            timing[0] = int(value)
        return f(self, key, value)

    def logged(name, f):
        def call(self, *a, **kw):
            calls.append((name, timing[0]))
            return f(self, *a, **kw)
        return call

    monkeypatch.setattr(vote.Solver, "set_option", set_option)
    monkeypatch.setattr(vote.Solver, "solve", logged("solve", vote.Solver.solve))
    monkeypatch.setattr(vote.Solver, "solve_host", logged("host", vote.Solver.solve_host))
    monkeypatch.setattr(sys, "argv", ["bench.py", "--workload", "line2d_n1e4", "--steps", "4", "--warmup", "3",
                                      "--no-cpu", "--no-fp64", "--no-group-stats"])
    bench.main()
    assert calls == [("solve", 0)] * 7 + [("solve", 1), ("solve", 1), ("host", 0)]
    line = json.loads(capsys.readouterr().out.strip().splitlines()[-1])
    assert line["steps"] == 4 and line["gpu_launches"] > 0 and line["kernel_ms"]["test_count"] > 0
    assert 0 < line["tests_per_s"] <= line["pairs_decided_per_s"]
    assert line["e2e"]["h2d_bytes_per_step"] == 2 * 8 * 10_000
