"""The bench's roofline entries name the kernel that ran and count what it moves."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402
from paper_1808_02558_gb300 import binding  # noqa: E402


def test_solve_roofline_follows_the_kernel():
    args = (191806, 64000, [60, 60], [4, 4], [1.0, 1.0], "pile40p")
    r = bench.solve_roofline(binding, binding.QP_SOLVER_RESIDENT, *args)
    k = bench.solve_roofline(binding, binding.QP_SOLVER_GLOBAL, *args)
    assert "k_cg_resident" in r["kernel"] and "k_pcg" in k["kernel"]
    assert r["bound"] == "latency" and k["bound"] == "hbm" and k["traffic"] is None
    # the resident kernel's iterations move nothing through HBM, the global kernel's all
    more = bench.solve_roofline(binding, binding.QP_SOLVER_RESIDENT, 191806, 64000, [90, 90], *args[3:])
    assert more["achieved"] == r["achieved"] < k["achieved"]
    assert r["us_per_iteration"] == pytest.approx(1000 / 60)


def test_qtt_schedule():
    full = lambda d, r: [min(r, 4 ** min(k, d - k)) for k in range(d + 1)]
    assert bench.qtt_schedule(full(20, 10)) == [5, 5, 5, 5]
    assert bench.qtt_schedule(full(12, 1)) == [5, 4, 3]
    assert bench.qtt_schedule(full(6, 2)) == [2, 2, 2]
    for d in range(1, 21):
        for r in (1, 4, 9, 10, 11, 12, 13, 16, 17, 24):
            plan = bench.qtt_schedule(full(d, r))
            assert sum(plan) == d and min(plan) >= 1 and max(plan) <= 5
