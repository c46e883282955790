"""GPU parity of rows over warps (plans with RETAIN_WARPS: softmax, log-sum-exp and int8) where it can go wrong: widths
around a segment of half and of all a warp's buffer, rows with fewer groups than warps, one row to many turns per
warp, any start on the 16-byte grid, in place, infinities, and what it refuses."""
import numpy as np
import pytest
import torch

from paper_2609_01864_gb300 import credit as C

import parity_util as U

pytestmark = pytest.mark.gpu
SHAPES = [(1, 16), (1, 8), (2, 8), (4, 8), (8, 8), (8, 16), (16, 8), (16, 16)]  # CTAs, warps of each


@pytest.fixture(scope="module", autouse=True)
def _init():
    from paper_2609_01864_gb300 import build as B
    B.build()
    C.init()


def plan_of(P, W):
    return C.make_plan(C.PATH_ONE_CTA if P == 1 else C.PATH_CLUSTER, P, retain=C.RETAIN_WARPS, threads=32 * W)


def check(op, dt, rows, cols, plan, off_in=0, off_out=0, seed=0):
    x, _ = U.make_input(dt, rows, cols, kind="outliers" if op == C.QUANT_INT8 else "normal", seed=seed)
    buf = torch.empty(off_in + rows * cols, dtype=x.dtype, device="cuda")
    d = buf[off_in:].view(rows, cols)
    d.copy_(x)
    out_dt = C.F32 if op == C.LOGSUMEXP else C.INT8 if op == C.QUANT_INT8 else dt
    n = rows if op == C.LOGSUMEXP else rows * cols
    guard = torch.full((off_out + n + 16,), 77, device="cuda").to(C.TORCH_DTYPE[out_dt])
    y = guard[off_out:off_out + n]
    sc = torch.zeros(rows, device="cuda")
    C.run_ex(op, d, y, plan=plan, rows=rows, cols=cols, in_dtype=dt, out_dtype=out_dt,
             out_scale=sc if op == C.QUANT_INT8 else None)
    torch.cuda.synchronize()
    assert C.device_error() == C.OK
    if op == C.QUANT_INT8:  # the two-pass path's codes and scales, bit for bit
        y2, s2 = torch.zeros_like(y), torch.zeros_like(sc)
        C.run_ex(op, d, y2, plan=C.make_plan(C.PATH_TWO_PASS), rows=rows, cols=cols, in_dtype=dt, out_dtype=out_dt,
                 out_scale=s2)
        torch.cuda.synchronize()
        assert torch.equal(y, y2) and torch.equal(sc, s2)
    else:
        ref = U.reference(op, dt, x)
        err = U.error_metric(op, out_dt, U.to64(y if op == C.LOGSUMEXP else y.view(rows, cols)), ref)
        assert err <= 1.0, err
    assert (guard[:off_out].float() == 77).all() and (guard[off_out + n:].float() == 77).all()


@pytest.mark.parametrize("op", [C.SOFTMAX, C.LOGSUMEXP, C.QUANT_INT8])
@pytest.mark.parametrize("dt", [C.F32, C.BF16])
@pytest.mark.parametrize("P,W", SHAPES)
def test_widths(op, dt, P, W):
    V = 4 if dt == C.F32 else 8
    check(op, dt, 40, 5 * V + 1, plan_of(P, W), 1, 3)                 # hardly a group per warp
    check(op, dt, 9, 440 * P * V + 3, plan_of(P, W), 3, 0)            # segments of half a buffer and a little more
    check(op, dt, 9, 880 * P * V - 1, plan_of(P, W), 0, 1)
    check(op, dt, 700 if P <= 4 else 90, 220 * P * V, plan_of(P, W))  # many turns
    check(op, dt, 5, 870 * P * W * V - 2, plan_of(P, W), 1, 1)        # the widest


@pytest.mark.parametrize("dt", [C.F32, C.BF16])
def test_in_place_and_strided(dt):
    rows, cols, ld = 300, 70001, 70016
    x, _ = U.make_input(dt, rows, ld, seed=4)
    d = x.cuda()
    want = torch.empty_like(d)
    kw = dict(rows=rows, cols=cols, ld_in=ld, ld_out=ld, in_dtype=dt, out_dtype=dt)
    C.run_ex(C.SOFTMAX, d, want, plan=plan_of(8, 8), **kw)
    C.run_ex(C.SOFTMAX, d, d, plan=plan_of(8, 8), **kw)
    torch.cuda.synchronize()
    assert torch.equal(want[:, :cols], d[:, :cols]) and torch.equal(d[:, cols:].cpu(), x[:, cols:])


def test_infinities():
    x = torch.randn(3, 60000)
    x[0, :59990] = -torch.inf
    x[1] = -torch.inf
    x[2, 7] = torch.inf
    y, _ = U.run_gpu(C.SOFTMAX, x, None, plan=plan_of(4, 8))
    lse, _ = U.run_gpu(C.LOGSUMEXP, x, None, plan=plan_of(4, 8))
    torch.cuda.synchronize()
    assert torch.allclose(y[0].cpu().double(), torch.softmax(x[0].double(), 0), rtol=1e-5, atol=0)
    assert torch.isnan(y[1]).all() and torch.isnan(y[2, 7])
    assert abs(lse[0].item() - torch.logsumexp(x[0].double(), 0).item()) < 1e-5 and lse[1].item() == -np.inf


@pytest.mark.parametrize("P,W", [(1, 16), (4, 8)])
def test_subnormal_outputs(P, W):
    """Outputs below the normal numbers: within one unit of 2^-149 and one part in 10^5 of the oracle."""
    x = torch.zeros(4, 5003)
    x[:, 1:] = -torch.linspace(80, 104, 5002)
    y, _ = U.run_gpu(C.SOFTMAX, x, None, plan=plan_of(P, W))
    torch.cuda.synchronize()
    ref = torch.softmax(x.double(), 1)
    assert ((y.cpu().double() - ref).abs() <= 2.0 ** -149 + 1e-5 * ref).all()


def test_planned_and_refused():
    for op, dt, cols in ((C.SOFTMAX, C.BF16, 131072), (C.QUANT_INT8, C.F32, 50001), (C.LOGSUMEXP, C.BF16, 32003)):
        p = C.plan(op, 1300, cols, dt, C.INT8 if op == C.QUANT_INT8 else None)
        assert p.retain == C.RETAIN_WARPS
        check(op, dt, 20, cols, p)
    x = torch.zeros(2, 4096, device="cuda")
    for bad in (C.make_plan(C.PATH_ONE_CTA, retain=C.RETAIN_WARPS, threads=1024),
                C.make_plan(C.PATH_ONE_CTA, retain=C.RETAIN_WARPS, ring_chunks=2)):
        assert C.plan_check(C.SOFTMAX, x, x, bad) == C.ERR_UNSUPPORTED
    assert C.plan_check(C.RMSNORM, x, x, plan_of(2, 8)) == C.ERR_UNSUPPORTED       # no such kernel
    w = torch.zeros(1, 880 * 8 * 4 + 64, device="cuda")
    assert C.plan_check(C.SOFTMAX, w, w, plan_of(1, 8)) == C.ERR_UNSUPPORTED       # too wide for one CTA's warps
