"""Solves of two sizes from two host threads, a context each: what a launch needs is set
per launch or the same for all, so neither can spoil the other's."""
import threading
import time

import numpy as np
import pytest
import torch

from gpu_common import to_np
from paper_1808_02558_gb300 import binding, workload
from synth import lattice_scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mixed,sides", [(1, (12, 27)), (0, (17, 27)), (1, (31, 36))])
def test_two_threads_of_different_sizes(mixed, sides):
    """The two systems run in the same kernel with different shared memory."""
    def system(n):
        ctx = binding.Context()
        _, con = workload.assemble(ctx, lattice_scene(n, 1))
        gamma = torch.zeros(con.P, dtype=torch.float64, device="cuda")
        lam = torch.zeros(2 * con.Nc, dtype=torch.float64, device="cuda")
        st = ctx.state(gamma, lam)
        ctx.pdip_init(st, 1.0)
        rhs = torch.empty_like(gamma)
        ctx.newton_rhs(st, rhs)
        return ctx, st, rhs, torch.empty_like(rhs), (gamma, lam)

    systems = [system(n) for n in sides]
    opts = [s[0].solve_opts(tol=1e-14, maxit=3, mixed=mixed, inner_tol=1e-3 if mixed else 0.0) for s in systems]
    alone = []
    for (ctx, st, rhs, dx, _), o in zip(systems, opts):
        ctx.newton_solve(st, rhs, dx, o)
        assert ctx.solver_used()[0] == binding.QP_SOLVER_RESIDENT
        alone.append(to_np(dx))
    errors = []

    def work(k):
        ctx, st, rhs, dx, _ = systems[k]
        try:
            pause = np.random.default_rng(k).random(3000) * 2e-4
            for p in pause:  # (on one stream: without pauses each would wait for the other's kernel in turn)
                time.sleep(p)
                s = ctx.newton_solve(st, rhs, dx, opts[k])
                assert s.iters == 3
            assert (to_np(dx) == alone[k]).all()
        except Exception as e:  # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
