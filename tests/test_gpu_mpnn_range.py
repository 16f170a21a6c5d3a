"""Weight gradients at the ends of FP32's range: infinite partial sums stay infinite, and
partial sums whose running total leaves the range, but not their sum, add up."""
import numpy as np
import pytest
import torch

from gpu_common import Problem, to_np
from oracle import mpnn
from paper_1808_02558_gb300 import learned
from synth import lattice_scene
from test_gpu_mpnn import SCALE, bf16_round

pytestmark = pytest.mark.gpu

ROWS = 64  # contacts of a partial sum up to 64 rows an SM's four blocks
OFF_BO = sum(int(np.prod(s)) for s in mpnn.SHAPES[:-1])
OFF_WO = OFF_BO - 3 * 64
OFF_B3 = OFF_WO - 64


def test_infinite_residuals():
    """A residual past FP32's range makes the output layer's sums of its component infinite."""
    pb = Problem(None, lattice_scene(5, 2))
    params = learned.init_params(3)
    y = np.zeros((pb.Nc, 3), np.float32)
    c = pb.Nc // 2
    y[c, 1] = -3e38  # 2 (o - y) overflows
    g = torch.empty_like(params)
    pb.ctx.mpnn_grad(params, SCALE, torch.tensor(y.reshape(-1), device="cuda"), g)
    got = to_np(g)
    x = mpnn.features(pb.scene, pb.oc, pb.r, np.array(SCALE))
    h = mpnn.forward(bf16_round(to_np(params)), x, pb.oc.a, pb.oc.b, pb.scene.M)[1][-1][2][c]
    gb, gW = got[OFF_BO:], got[OFF_WO:OFF_BO].reshape(3, 64)
    assert gb[1] == np.inf and np.isfinite(gb[[0, 2]]).all()
    sure = np.abs(h) > 1e-3  # (an activation at 0 may fall to either side)
    assert sure.sum() > 10
    assert (gW[1][sure & (h > 0)] == np.inf).all()
    assert np.isfinite(gW[[0, 2]]).all()


def test_running_sums_past_the_range():
    """Partial sums of +-3e38 in the order + + - -: an FP32 running sum overflows at the
    second one, the sum itself is that of one contact."""
    pb = Problem(None, lattice_scene(15, 6))
    assert ROWS * 148 + 100 < pb.Nc <= ROWS * 4 * 150
    params = torch.zeros_like(learned.init_params(1))
    B = 2.0 ** 100
    params[OFF_B3:OFF_WO] = B  # h3 = B everywhere, outputs 0
    d = 3e38 / ROWS / B * 1.5 * pb.Nc
    part = np.arange(pb.Nc) // ROWS
    sign = np.where(part < 148, np.where(part % 4 < 2, 1.0, -1.0), 0.0)
    sign[-1] = 0.25
    y = np.zeros((pb.Nc, 3), np.float32)
    y[:, 2] = -d * sign
    g = torch.empty_like(params)
    loss = pb.ctx.mpnn_grad(params, SCALE, torch.tensor(y.reshape(-1), device="cuda"), g)
    got = to_np(g).astype(np.float64)
    dO = np.float64(np.float32(2) * np.float32(0.25 * d) / np.float32(3 * pb.Nc))
    # the partial sums cancel to the bit (the same sums with the other sign); FP32 rounds the rest
    assert abs(got[OFF_BO + 2] - dO) <= 1e-6 * dO
    gW = got[OFF_WO:OFF_BO].reshape(3, 64)
    assert (np.abs(gW[2] - dO * B) <= 1e-6 * dO * B).all() and not gW[:2].any()
    assert abs(loss - (y.astype(np.float64) ** 2).mean()) <= 1e-6 * loss
