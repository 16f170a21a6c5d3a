"""Which kernel runs a Jacobi-CG solve, at the edges of the resident solver's room, and that
the kernel behind it solves what it refuses: against the residual of the oracle's Schur
matrix."""
import numpy as np
import pytest
import torch

from gpu_common import dev, to_np
from oracle import contacts as oc, qp
from paper_1808_02558_gb300 import binding, workload
from synth import Scene, box_scene, lattice_scene

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


def studded_ball():
    """Three concentric balls of radius 60, a hair apart, studded with 6700 small ones: every
    block of contacts touches all three, more shared bodies' runs than a block has room for."""
    n = 6700
    i = np.arange(n) + 0.5
    z, a = 1 - 2 * i / n, np.pi * (1 + 5 ** 0.5) * i
    at = 60.5 * np.stack([np.sqrt(1 - z * z) * np.cos(a), np.sqrt(1 - z * z) * np.sin(a), z], 1)
    pos = np.concatenate([at, 0.02 * np.eye(3)])
    vel = 0.1 * np.random.default_rng(3).standard_normal(pos.shape)
    return Scene(name="studded", pos=pos, vel=vel, omega=np.zeros_like(vel),
                 radius=np.concatenate([np.full(n, 0.5), np.full(3, 60.0)]), floor_z=-100.0, delta=0.1)


def solve(scene, mixed, tol, again=1):
    """Solve a centred iterate's system for a random right-hand side, check the residual
    (S = D^T M^-1 D + H in factors), and return what newton_solver_used says."""
    ctx = binding.Context()
    _, con = workload.assemble(ctx, scene)
    o = oc.detect(scene)
    assert o.Nc == con.Nc
    g, lam = centred(o.Nc, scene.mu, 11)
    D, m, H = qp.jacobian(scene, o), qp.inv_mass_diag(scene), qp.blockdiag(qp.schur_blocks(g, lam, scene.mu))
    b = np.random.default_rng(5).standard_normal(3 * o.Nc)
    gd, ld, rhs = (dev(v) for v in (qp.to_padded(g, o.Nc, 3, con.P), lam, qp.to_padded(b, o.Nc, 3, con.P)))
    st = ctx.state(gd, ld)
    opts = ctx.solve_opts(tol=tol, maxit=50000, mixed=mixed, inner_tol=1e-3 if mixed else 0.0, max_outer=60)
    for _ in range(again):
        dx = torch.full_like(rhs, float("nan"))
        stats = ctx.newton_solve(st, rhs, dx, opts, allow=())
        assert stats.status == binding.QP_OK and stats.rel_res <= tol
        x = qp.from_padded(to_np(dx), o.Nc, 3)
        # the oracle's residual differs by the rounding of one product, eps || |S| |x| || a
        # few times over
        size = abs(D).T @ (m * (abs(D) @ np.abs(x))) + abs(H) @ np.abs(x)
        res = np.linalg.norm(b - (D.T @ (m * (D @ x)) + H @ x))
        assert res <= tol * np.linalg.norm(b) + 64 * np.finfo(float).eps * np.linalg.norm(size)
    return ctx.solver_used(), con.Nc


def test_none_before_the_first_solve():
    assert binding.Context().solver_used() == (binding.QP_SOLVER_NONE, 0)


@pytest.mark.parametrize("mixed", [0, 1])
@pytest.mark.parametrize("n", [2, 9, 16, 27])
def test_piles_are_resident(n, mixed):
    assert solve(lattice_scene(n, 4), mixed, 1e-11)[0] == (binding.QP_SOLVER_RESIDENT, 1)


def test_edges_of_the_room_by_size():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    scene = lattice_scene(32, 9)  # 96 256 contacts: two a thread, and no FP64 form
    used, Nc = solve(scene, 1, 1e-10)
    assert 512 * sms < Nc <= 1280 * sms and used == (binding.QP_SOLVER_RESIDENT, 1)
    assert solve(scene, 0, 1e-10)[0] == (binding.QP_SOLVER_GLOBAL, 0)


def test_mixed_beyond_the_room():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    used, Nc = solve(lattice_scene(41, 2, polydisperse=True), 1, 1e-10)
    assert Nc > 1280 * sms and used == (binding.QP_SOLVER_GLOBAL, 0)


@pytest.mark.parametrize("mixed", [0, 1])
def test_refused_by_the_plan(mixed):
    (used, launches), _ = solve(studded_ball(), mixed, 1e-10, again=2)
    assert used == binding.QP_SOLVER_GLOBAL and launches >= 1


@pytest.mark.parametrize("mixed", [0, 1])
def test_a_refusal_is_remembered(mixed):
    scene = studded_ball()
    assert solve(scene, mixed, 1e-8, again=1)[0] == solve(scene, mixed, 1e-8, again=4)[0]


def test_sparse_contact_sets_are_resident():
    """A walled box of 55^3 falling spheres has about one body a contact, more than the usual
    room of a block holds: the second shape takes it, and the next solve goes there at once."""
    used, Nc = solve(box_scene(5, n=55, layers=55), 1, 1e-10, again=3)
    assert used == (binding.QP_SOLVER_RESIDENT, 4)
