"""Right-hand sides that leave the resident solver nothing to do, or nothing that it can do:
identity rows alone, a tolerance met by zero, a breakdown."""
import math

import numpy as np
import pytest
import torch

from gpu_common import Problem, dev, to_np
from oracle import qp
from paper_1808_02558_gb300 import binding
from synth import lattice_scene

pytestmark = pytest.mark.gpu


def problem(slots):
    pb = Problem(None, lattice_scene(5, 1), slots)
    pb.keep = pb.state(*qp.initial_point(pb.Nc, pb.scene.mu))
    return pb, pb.keep[2]


def opts(pb, mixed, tol):
    return pb.ctx.solve_opts(tol=tol, mixed=mixed, inner_tol=1e-3 if mixed else 0.0)


@pytest.mark.parametrize("mixed", [0, 1])
@pytest.mark.parametrize("small", [0.0, 1e-13])
def test_identity_rows_alone(mixed, small):
    """S has identity rows for a contact's fourth slot: they are solved by their right-hand
    side, and the others at most to the tolerance."""
    pb, st = problem(4)
    rng = np.random.default_rng(2)
    rhs = np.zeros(pb.P)
    rhs[3:4 * pb.Nc:4] = rng.standard_normal(pb.Nc)
    rhs[0:4 * pb.Nc:4] = small
    dx = torch.full((pb.P,), float("nan"), dtype=torch.float64, device="cuda")
    stats = pb.ctx.newton_solve(st, dev(rhs), dx, opts(pb, mixed, 1e-10), allow=())
    assert stats.status == binding.QP_OK
    assert stats.rel_res <= 2e-13  # small sqrt(Nc) over the norm of Nc normal values
    got = to_np(dx)
    assert (got[3:4 * pb.Nc:4] == rhs[3:4 * pb.Nc:4]).all()
    got[3:4 * pb.Nc:4] = 0.0
    assert not got.any()


@pytest.mark.parametrize("mixed", [0, 1])
def test_tolerance_met_by_zero(mixed):
    pb, st = problem(3)
    rhs = dev(pb.pad(np.random.default_rng(1).standard_normal(3 * pb.Nc)))
    dx = torch.full_like(rhs, float("nan"))
    stats = pb.ctx.newton_solve(st, rhs, dx, opts(pb, mixed, 1.0), allow=())
    assert stats.status == binding.QP_OK and stats.iters == 0 and stats.rel_res == 1.0 and not to_np(dx).any()


@pytest.mark.parametrize("mixed", [0, 1])
def test_breakdown_reports_its_residual(mixed):
    """A breakdown before any progress is no residual of 0."""
    pb, st = problem(3)
    rhs = dev(pb.pad(np.random.default_rng(1).standard_normal(3 * pb.Nc)))
    rhs[4] = float("nan")
    dx = torch.empty_like(rhs)
    stats = pb.ctx.newton_solve(st, rhs, dx, opts(pb, mixed, 1e-10))
    assert stats.status == binding.QP_BREAKDOWN and math.isnan(stats.rel_res)
