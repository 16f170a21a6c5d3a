"""The learned warm start's passes over contact rows at the sizes where their
tiles end: one contact, fewer than one 32-row stage, just past it, odd counts over
several blocks; forward, loss and every block of the gradient against the oracle."""
import numpy as np
import pytest
import torch

from gpu_common import Problem, assert_close, relerr, to_np
from oracle import mpnn
from paper_1808_02558_gb300 import learned
from synth import lattice_scene
from test_gpu_mpnn import SCALE, bf16_round

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,poly", [(1, False), (2, False), (2, True), (3, False), (5, False), (7, True)])
def test_rows_against_oracle(n, poly):
    pb = Problem(None, lattice_scene(n, 3 + n, polydisperse=poly))
    params = learned.init_params(n)
    theta = bf16_round(to_np(params))
    x = mpnn.features(pb.scene, pb.oc, pb.r, np.array(SCALE))
    out = torch.empty(3 * pb.Nc, dtype=torch.float32, device="cuda")
    pb.ctx.mpnn_forward(params, SCALE, out)
    want, _ = mpnn.forward(theta, x, pb.oc.a, pb.oc.b, pb.scene.M)
    # the bounds of the larger cases: FP32 layers of width 64 against FP64
    assert_close(to_np(out), want.reshape(-1), 1e-4, floor_rel=1e-2, what=f"forward, {pb.Nc} contacts")
    y = np.random.default_rng(n).standard_normal((pb.Nc, 3))
    g = torch.full_like(params, float("nan"))
    loss = pb.ctx.mpnn_grad(params, SCALE, torch.tensor(y.reshape(-1), dtype=torch.float32, device="cuda"), g)
    L, gw = mpnn.grad(theta, x, pb.oc.a, pb.oc.b, pb.scene.M, y.astype(np.float32).astype(np.float64))
    assert abs(loss - L) <= 1e-5 * L
    assert relerr(to_np(g).astype(np.float64), gw) <= 1e-4
    k = 0
    for s in mpnn.SHAPES:
        m = int(np.prod(s))
        assert_close(to_np(g)[k:k + m], gw[k:k + m], 1e-3, floor_rel=1e-2, what=f"gradient block {s}, {pb.Nc} contacts")
        k += m
