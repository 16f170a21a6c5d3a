"""Compression's Gram and projection kernels at rank caps on both sides of the lines
between them (a thread a parent at rank 1, tiles by sets of children to 16, scattered rows
above) and at odd ranks, at sizes whose sets and blocks hold few parents.

The approximation error and the ranks must be those of the oracle's TT-SVD of the dense
matrix; eigenvalues carry 1e-15 of the largest, so the errors agree to 1e-6 of the norm
with orders of magnitude to spare."""
import numpy as np
import pytest
import torch

from gpu_common import dev
from oracle import contacts as oc, qp, tt
from paper_1808_02558_gb300 import binding, workload
from synth import lattice_scene

pytestmark = pytest.mark.gpu
_dense = {}


def dense(n, slots):
    if (n, slots) not in _dense:
        s = lattice_scene(n, 5, polydisperse=True)
        con = oc.detect(s)
        _, N, _ = qp.qp_data(s, con)
        g, lam = qp.initial_point(con.Nc, s.mu)
        _, P = qp.padded_size(con.Nc, slots)
        S = qp.padded_matrix(qp.schur_matrix(N, g, lam, s.mu), con.Nc, slots, P).toarray()
        _dense[n, slots] = s, qp.to_padded(g, con.Nc, slots, P), lam, S
    return _dense[n, slots]


@pytest.mark.parametrize("n,slots", [(2, 3), (3, 4), (5, 3)])
@pytest.mark.parametrize("rmax", [1, 2, 5, 6, 7, 10, 11, 12, 16, 17])
def test_rank_caps(n, slots, rmax):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    s, g, lam, S = dense(n, slots)
    ctx = binding.Context()
    workload.assemble(ctx, s, slots)
    X = ctx.qtt_compress(ctx.state(dev(g), dev(lam)), 1e-3, rmax)
    want = tt.qtt_compress_dense(S, 1e-3, rmax, reverse=True)
    got = tt.qtt_matrix(X.cores())
    assert X.ranks() == tt.tt_ranks(want)
    assert abs(np.linalg.norm(got - S) - np.linalg.norm(tt.qtt_matrix(want) - S)) <= 1e-6 * np.linalg.norm(S)
    ctx.close()
