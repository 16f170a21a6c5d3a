"""Newton solves of a PDIP run's late iterates, where the attainable accuracy is near the
tolerance: a solve that cannot reach its tolerance ends near the attainable accuracy and
returns the best solution that it formed, in FP64 and in mixed precision."""
import numpy as np
import pytest
import torch

from gpu_common import Problem, dev, to_np
from oracle import pdip, qp
from paper_1808_02558_gb300 import binding
from synth import lattice_scene

pytestmark = pytest.mark.gpu

KEEP = (18, 24, 27, 30)


@pytest.fixture(scope="module")
def pile():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pb = Problem(None, lattice_scene(8, 1, polydisperse=True))
    g, lam = qp.initial_point(pb.Nc, pb.scene.mu)
    pb.iter = {}
    for k in range(max(KEEP) + 1):
        if k in KEEP:
            pb.iter[k] = (g.copy(), lam.copy())
        g, lam, _ = pdip.pdip_step(pb.N, pb.r, pb.scene.mu, g, lam)
    return pb


def solve(pb, k, **opts):
    """Statistics of a solve of iterate k's Newton system, the oracle's residual of its
    result, and by how much the two may differ: a row's product sums some twenty terms,
    each rounded a few times, so 8 eps || |S| |x| || bounds it."""
    g, lam = pb.iter[k]
    gd, ld, st = pb.state(g, lam)
    t = pdip.NU * 2 * pb.Nc / float(-(qp.constraints(g, pb.scene.mu) @ lam))
    b = qp.newton_rhs(pb.N, pb.r, g, lam, t, pb.scene.mu)
    rhs = dev(pb.pad(b))
    dx = torch.full_like(rhs, float("nan"))
    stats = pb.ctx.newton_solve(st, rhs, dx, pb.ctx.solve_opts(**opts))
    S = qp.schur_matrix(pb.N, g, lam, pb.scene.mu)
    x, nb = pb.unpad(to_np(dx)), np.linalg.norm(b)
    return stats, np.linalg.norm(b - S @ x) / nb, 8 * np.finfo(float).eps * np.linalg.norm(abs(S) @ np.abs(x)) / nb


# 1e-12 is at the attainable accuracy from iterate 24 on (a restarted FP64 CG in NumPy
# stops between 7e-13 and 1e-11 there) and 1e-15 is out of reach for all of them; 1e-10
# leaves a factor of ten for the order of the sums
@pytest.mark.parametrize("k", KEEP)
@pytest.mark.parametrize("tol", [1e-12, 1e-15])
def test_fp64_near_the_attainable_accuracy(pile, k, tol):
    stats, res, noise = solve(pile, k, tol=tol, maxit=20000)
    assert stats.status == (binding.QP_OK if stats.rel_res <= tol else binding.QP_NOT_CONVERGED)
    assert stats.rel_res <= 1e-10
    assert abs(res - stats.rel_res) <= noise


@pytest.mark.parametrize("k", KEEP)
def test_fp64_converges_above_it(pile, k):
    stats, res, noise = solve(pile, k, tol=1e-10, maxit=20000)
    assert stats.status == binding.QP_OK and stats.rel_res <= 1e-10 and res <= 1e-10 + noise


# FP32 reaches its own end in these systems; started afresh from the true residual it needs
# about 2000 iterations at iterate 27 (NumPy, FP32), with the direction kept more than 20 000
@pytest.mark.parametrize("k", [18, 24, 27])
def test_mixed(pile, k):
    stats, res, noise = solve(pile, k, tol=1e-8, maxit=20000, mixed=1, inner_tol=1e-3, max_outer=80)
    assert stats.status == binding.QP_OK and stats.rel_res <= 1e-8
    assert abs(res - stats.rel_res) <= noise


def test_mixed_out_of_reach(pile):
    stats, res, noise = solve(pile, 30, tol=1e-15, maxit=6000, mixed=1, inner_tol=1e-3, max_outer=8)
    assert stats.status == binding.QP_NOT_CONVERGED and stats.rel_res < 1.0
    assert abs(res - stats.rel_res) <= noise
