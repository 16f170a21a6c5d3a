"""QTT products whose cores are contracted several a pass: the sizes and ranks where
the passes' cuts fall differently (sizes below and at the first possible pass, odd
remainders, ranks at and past each padding, ranks that rise and fall, a core too wide
in the middle), FP32, BF16 and FP64 cores, against the oracle entry by entry."""
import numpy as np
import pytest
import torch

from gpu_common import assert_close, to_np
from oracle import tt
from paper_1808_02558_gb300 import binding

pytestmark = pytest.mark.gpu


def ranks_of(d, r):
    if isinstance(r, int):
        return [min(r, 4 ** min(k, d - k)) for k in range(d + 1)]
    return [1] + [min(r[k % len(r)], 4 ** min(k, d - k)) for k in range(1, d)] + [1]


CASES = [(1, 2), (4, 7), (5, 3), (9, 10), (10, 10), (10, 4), (11, 10), (12, 9), (12, 11), (13, 16), (13, 17), (14, 8),
         (14, (3, 9, 1, 14)), (15, (10, 10, 20, 10)), (16, (5, 12)), (17, 10), (18, 10)]


@pytest.mark.parametrize("d,r", CASES, ids=[f"d{d}-r{r}".replace(" ", "") for d, r in CASES])
@pytest.mark.parametrize("kind", ["f64", "f32", "bf16", "f64cores"])
def test_product_against_oracle(d, r, kind):
    rng = np.random.default_rng(100 * d + (r if isinstance(r, int) else sum(r)))
    ranks = ranks_of(d, r)
    cores = [rng.standard_normal((ranks[k], 4, ranks[k + 1])) / np.sqrt(2 * ranks[k + 1]) for k in range(d)]
    ctx = binding.Context()
    A = ctx.qtt_from_cores(cores)
    vdt = torch.float64 if kind == "f64" else torch.float32
    cdt = {"f64": binding.QP_F64, "f32": binding.QP_F32, "bf16": binding.QP_BF16, "f64cores": binding.QP_F64}[kind]
    if kind in ("f32", "f64cores"):
        cores = [c.astype(np.float32).astype(np.float64) for c in cores]
    elif kind == "bf16":
        cores = [torch.tensor(c, dtype=torch.float32).to(torch.bfloat16).to(torch.float64).numpy() for c in cores]
    x = torch.tensor(rng.standard_normal(1 << d), dtype=vdt, device="cuda")
    # one element past an aligned address: the caller's vectors carry no alignment
    buf = torch.full((2 + (1 << d),), float("nan"), dtype=vdt, device="cuda")
    y = buf[1:-1]
    ctx.qtt_set_tensor_cores(0)
    ctx.qtt_apply(A, x, y, cdt, binding.QP_F64 if kind == "f64" else binding.QP_F32)
    want = tt.qtt_matvec(cores, to_np(x).astype(np.float64))
    size = tt.qtt_matvec([np.abs(c) for c in cores], np.abs(to_np(x)).astype(np.float64))
    # each of the d contractions sums 2 r products: (2 r + 1) roundings of half an ulp,
    # carried by the later ones; |G_1| .. |G_d| |x| bounds the terms
    eps = 2.0 ** -53 if kind == "f64" else 2.0 ** -24
    assert_close(to_np(y), want, eps * sum(2 * q + 1 for q in ranks[1:]) * 1.01, scale=size, what=f"d={d} r={r} {kind}")
    assert bool(torch.isnan(buf[0])) and bool(torch.isnan(buf[-1]))
    A.free()
    ctx.close()
