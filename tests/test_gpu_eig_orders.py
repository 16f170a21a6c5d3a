"""Compression's one-block eigensolver at rank caps whose Gram orders 4 r lie around the
line where the FP32 start begins (order 16) and where shared memory ends (64), against
the oracle's TT-SVD of the dense matrix.

Both cut the same spectra at the same places, so the approximation errors agree to the
rounding of the eigenvalues (1e-15 of the largest, twelve levels); where a cap cuts
between two eigenvalues their relative gap is above 1e-6 and the cut directions are exact
to 1e-9, which changes the error in second order: 1e-6 of the norm is asked for."""
import numpy as np
import pytest
import torch

from gpu_common import dev
from oracle import contacts as oc, qp, tt
from paper_1808_02558_gb300 import binding, workload
from synth import lattice_scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def scene():
    s = lattice_scene(4, 4, polydisperse=True)
    con = oc.detect(s)
    _, N, _ = qp.qp_data(s, con)
    g, lam = qp.initial_point(con.Nc, s.mu)
    _, P = qp.padded_size(con.Nc, 3)
    return s, con, g, lam, qp.padded_matrix(qp.schur_matrix(N, g, lam, s.mu), con.Nc, 3, P).toarray(), P


@pytest.mark.parametrize("eps,rmax", [(1e-2, r) for r in (3, 4, 5, 6, 9, 10, 15, 16, 17)] + [(1e-4, 16), (0.0, 5), (0.9, 16)])
def test_compress_orders(scene, eps, rmax):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    s, con, g, lam, S, P = scene
    ctx = binding.Context()
    workload.assemble(ctx, s, 3)
    X = ctx.qtt_compress(ctx.state(dev(qp.to_padded(g, con.Nc, 3, P)), dev(lam)), eps, rmax)
    want = tt.qtt_compress_dense(S, eps, rmax, reverse=True)
    got = tt.qtt_matrix(X.cores())
    assert X.ranks() == tt.tt_ranks(want)
    nrm = np.linalg.norm(S)
    assert abs(np.linalg.norm(got - S) - np.linalg.norm(tt.qtt_matrix(want) - S)) <= 1e-6 * nrm
    ctx.close()
