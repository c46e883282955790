"""Backward ops at the ends of the FP32 range: what lies below or near the ends of it in between, while inputs and
result are ordinary numbers, has to come out as in exact arithmetic on every path."""
import numpy as np
import pytest
import torch

from paper_2609_01864_gb300 import credit as C

import parity_util as U

pytestmark = pytest.mark.gpu
PLANS = {"planned": None, "one_cta": C.make_plan(C.PATH_TWO_PASS, ctas_per_row=1),
         "split": C.make_plan(C.PATH_TWO_PASS, ctas_per_row=3),
         "rows_over_cluster": C.make_plan(C.PATH_CLUSTER, 4, retain=C.RETAIN_ROW)}


@pytest.fixture(scope="module", autouse=True)
def _init():
    from paper_2609_01864_gb300 import build as B
    B.build()
    C.init()


def softmax64(z):
    e = np.exp(z - z.max(1, keepdims=True))
    return e / e.sum(1, keepdims=True)


@pytest.mark.parametrize("plan", sorted(PLANS))
@pytest.mark.parametrize("op", [C.SOFTMAX_LOGITS_BWD, C.XENT_BWD])
@pytest.mark.parametrize("cols", [5000, 5003])
def test_logits_far_below_the_maximum(op, plan, cols):
    """Probabilities below the normal numbers reach the gradient: each of the two to three roundings on the way is
    at most 2^-150 there, times factors of at most 2, or one part in 10^5 where the numbers are normal.  One row has
    a dy so large that such a term decides the sum."""
    rows = 7
    z = torch.zeros(rows, cols)
    z[:, 1:] = -torch.linspace(80, 104, cols - 1)
    d = torch.zeros(rows, cols)
    kw = {}
    big = int((z[0] > -95).sum())
    if op == C.XENT_BWD:
        d[:, 0] = 1.0
        kw["scale"] = torch.full((rows,), 1.5, device="cuda")
    else:
        d[:, 0], d[:, 1::2], d[:, 2::2] = 1.0, 0.5, -1.0
        d[3, 1:] = 0.0
        d[3, big] = 2.0 ** 126
    dx = torch.full((rows, cols), float("nan"), device="cuda")
    C.run_bwd(op, z.cuda(), d.cuda(), dx, plan=PLANS[plan], **kw)
    torch.cuda.synchronize()
    assert C.device_error() == C.OK
    y, d64 = softmax64(z.double().numpy()), d.double().numpy()
    if op == C.XENT_BWD:
        ref = 1.5 * (y * d64.sum(1, keepdims=True) - d64)
    else:
        ref = y * (d64 - (y * d64).sum(1, keepdims=True))
    bound = 2.0 ** -147 + 1e-5 * np.abs(ref)
    bound[:, 0] = 4e-7  # at the maximum 1 - T / S cancels: three roundings of numbers near 1
    bound[3, big] += 2.0 ** -22
    err = np.abs(dx.cpu().double().numpy() - ref)
    assert np.isfinite(err).all() and (err <= bound).all(), (err / bound).max()


@pytest.mark.parametrize("plan", ["planned", "one_cta", "split"])
@pytest.mark.parametrize("op", [C.LAYERNORM_BWD, C.RMSNORM_BWD])
@pytest.mark.parametrize("scale", [1e-25, 1e19, 1e23, 1e36])
@pytest.mark.parametrize("cols", [4096, 4099])
def test_norm_rows_of_any_scale(op, plan, scale, cols):
    """Saved statistics of rows so small or large that rstd^2, or a sum of x g, leaves FP32 (the result does not)."""
    rows = 9
    _, dy, gamma, _, _ = U.bwd_inputs(op, C.F32, rows, cols, seed=3)
    a = torch.randn(rows, cols, generator=torch.Generator().manual_seed(11), dtype=torch.float64).mul(scale).float()
    a64 = a.double()
    mean = a64.mean(1).float() if op == C.LAYERNORM_BWD else None
    rstd = (1.0 / (a64.std(1, correction=0) if op == C.LAYERNORM_BWD else a64.square().mean(1).sqrt())).float()
    kw = {k: v.cuda() for k, v in dict(gamma=gamma, mean=mean, rstd=rstd).items() if v is not None}
    dx = torch.full((rows, cols), float("nan"), device="cuda")
    C.run_bwd(op, a.cuda(), dy.cuda(), dx, plan=PLANS[plan], **kw)
    torch.cuda.synchronize()
    assert C.device_error() == C.OK
    ref = U.bwd_reference(op, C.F32, a, dy, gamma, mean, rstd, rows, cols)
    assert torch.isfinite(dx).all()
    assert U.bwd_error(op, C.F32, U.to64(dx), ref, a, dy, gamma, mean, rstd, cols) <= 1.0
