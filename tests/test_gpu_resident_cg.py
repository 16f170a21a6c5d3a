"""The Jacobi-CG whose system stays on the SMs, at the sizes where its forms change:
one block, the FP64 form with a row a lane and the one with a contact a thread, one
and two contacts a thread in FP32; three and four slots, floor and walls; against the
residual of the oracle's Schur matrix."""
import numpy as np
import pytest
import torch

from gpu_common import Problem, dev, to_np
from oracle import qp
from paper_1808_02558_gb300 import binding
from synth import box_scene, column_scene, lattice_scene

pytestmark = pytest.mark.gpu


def centred(Nc, mu, seed):
    """An iterate inside the cones (a PDIP iterate's shape, without running one)."""
    rng = np.random.default_rng(seed)
    g = np.zeros((Nc, 3))
    g[:, 0] = 0.5 + rng.random(Nc)
    ang, rad = 2 * np.pi * rng.random(Nc), 0.8 * mu * g[:, 0] * np.sqrt(rng.random(Nc))
    g[:, 1], g[:, 2] = rad * np.cos(ang), rad * np.sin(ang)
    g = g.reshape(-1)
    return g, -(0.5 + rng.random(2 * Nc)) / qp.constraints(g, mu)


SCENES = [
    ("one block", lattice_scene(2, 1), 3),
    ("floor only", column_scene(7, 1, 2), 3),
    ("four slots", lattice_scene(5, 3, polydisperse=True), 4),
    ("32 contacts a block", lattice_scene(9, 4), 3),
    ("walls", box_scene(5, n=14, layers=14), 3),
    ("64 contacts a block", lattice_scene(15, 6), 3),
    ("78 contacts a block", lattice_scene(16, 7), 3),
    ("379 contacts a block", lattice_scene(27, 8), 3),
    ("575 contacts a block", lattice_scene(31, 9), 4),
]


@pytest.mark.parametrize("what,scene,slots", SCENES, ids=[s[0] for s in SCENES])
@pytest.mark.parametrize("mixed", [0, 1])
def test_residual_against_oracle(what, scene, slots, mixed):
    pb = Problem(None, scene, slots)
    g, lam = centred(pb.Nc, scene.mu, 11)
    gd, ld, st = pb.state(g, lam)
    b = np.random.default_rng(5).standard_normal(3 * pb.Nc)
    rhs = dev(pb.pad(b))
    dx = torch.full_like(rhs, float("nan"))
    tol = 1e-11
    for again in range(2):  # a second solve reuses the plan and the exchange slots
        opts = pb.ctx.solve_opts(tol=tol, maxit=50000, mixed=mixed, inner_tol=1e-3 if mixed else 0.0, max_outer=60)
        stats = pb.ctx.newton_solve(st, rhs, dx, opts, allow=())
        assert stats.status == binding.QP_OK and stats.rel_res <= tol
    S = qp.schur_matrix(pb.N, g, lam, scene.mu)
    x = pb.unpad(to_np(dx))
    # the kernel's own FP64 residual is at most tol; the oracle's differs by the rounding
    # of one product, eps || |S| |x| || a few times over
    noise = 64 * np.finfo(float).eps * np.linalg.norm(abs(S) @ np.abs(x))
    assert np.linalg.norm(b - S @ x) <= tol * np.linalg.norm(b) + noise
    full = to_np(dx)
    idx = (slots * np.arange(pb.Nc)[:, None] + np.arange(3)[None, :]).reshape(-1)
    rest = np.ones(full.size, bool)
    rest[idx] = False
    assert not full[rest].any()


def test_iteration_cap_and_zero_rhs():
    pb = Problem(None, lattice_scene(6, 1))
    g, lam = centred(pb.Nc, 0.5, 3)
    gd, ld, st = pb.state(g, lam)
    rhs = dev(pb.pad(np.random.default_rng(1).standard_normal(3 * pb.Nc)))
    dx = torch.empty_like(rhs)
    for mixed in (0, 1):
        stats = pb.ctx.newton_solve(st, rhs, dx, pb.ctx.solve_opts(tol=1e-10, maxit=7, mixed=mixed, inner_tol=1e-3 if mixed else 0.0))
        assert stats.status == binding.QP_NOT_CONVERGED and stats.iters == 7 and stats.rel_res > 1e-10
        stats = pb.ctx.newton_solve(st, torch.zeros_like(rhs), dx, pb.ctx.solve_opts(tol=1e-10, mixed=mixed), allow=())
        assert stats.status == binding.QP_OK and stats.iters == 0 and not to_np(dx).any()
        bad = rhs.clone()
        bad[0] = float("nan")
        stats = pb.ctx.newton_solve(st, bad, dx, pb.ctx.solve_opts(tol=1e-10, mixed=mixed))
        assert stats.status == binding.QP_BREAKDOWN
        # and the context still solves
        stats = pb.ctx.newton_solve(st, rhs, dx, pb.ctx.solve_opts(tol=1e-10, mixed=mixed, inner_tol=1e-3 if mixed else 0.0), allow=())
        assert stats.status == binding.QP_OK
