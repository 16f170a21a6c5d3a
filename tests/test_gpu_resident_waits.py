"""Failure detection without a GPU fault: the resident solver's waits are bounded.  A block
that leaves makes the others' waits run out; they record QP_TIMEOUT and return, and the
context's next solve clears the exchange slots and is as any other."""
import numpy as np
import pytest
import torch

from gpu_common import to_np
from paper_1808_02558_gb300 import binding, workload
from synth import lattice_scene

pytestmark = pytest.mark.gpu

POLLS = 20000  # about 10 ms


@pytest.mark.parametrize("mixed,n", [(0, 8), (0, 17), (1, 12), (1, 31)])
def test_waits_run_out_and_the_context_survives(mixed, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = binding.Context()
    _, con = workload.assemble(c, lattice_scene(n, 1))
    gamma = torch.zeros(con.P, dtype=torch.float64, device="cuda")
    lam = torch.zeros(2 * con.Nc, dtype=torch.float64, device="cuda")
    st = c.state(gamma, lam)
    c.pdip_init(st, 1.0)
    rhs = torch.empty_like(gamma)
    c.newton_rhs(st, rhs)
    opts = c.solve_opts(tol=1e-10, mixed=mixed, inner_tol=1e-3 if mixed else 0.0)

    def solve():
        dx = torch.full_like(rhs, float("nan"))
        stats = c.newton_solve(st, rhs, dx, opts, allow=())
        assert stats.status == binding.QP_OK and c.solver_used()[0] == binding.QP_SOLVER_RESIDENT
        return to_np(dx)

    want, scrap = solve(), torch.empty_like(rhs)
    assert c.selftest_resident(rhs, scrap, mixed, POLLS, -1) == binding.QP_OK
    for at in (0, 1):
        for block in (0, 3):
            assert c.selftest_resident(rhs, scrap, mixed, POLLS, block, at) == binding.QP_TIMEOUT
        assert np.array_equal(solve(), want)
    for bad in ((0, 1, 0), ((1 << 22) + 1, 1, 0), (POLLS, 100000, 0), (POLLS, 1, 2)):
        with pytest.raises(binding.QPError):
            c.selftest_resident(rhs, scrap, mixed, *bad)
    assert np.array_equal(solve(), want)
    c.close()


def test_needs_a_resident_contact_set():
    c = binding.Context()
    with pytest.raises(binding.QPError):  # no contacts yet
        c.selftest_resident(torch.zeros(4, dtype=torch.float64, device="cuda"),
                            torch.zeros(4, dtype=torch.float64, device="cuda"), 0, POLLS, -1)
