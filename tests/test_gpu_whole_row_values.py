"""The whole-row kernels on the values that the general paths are tested on: E4M3 rows under negative, zero, tiny and
large scales, logits of a masked vocabulary, NaN, gradients written over their inputs, and second gradients between
guards."""
import numpy as np
import pytest
import torch

from paper_2609_01864_gb300 import credit as C

import parity_util as U
from test_gpu_bwd_team import shifted

pytestmark = pytest.mark.gpu
G1 = C.make_plan(C.PATH_TWO_PASS, ctas_per_row=1)
ROWS = {"one_cta": C.make_plan(C.PATH_ONE_CTA, retain=C.RETAIN_ROW),
        "cluster4": C.make_plan(C.PATH_CLUSTER, 4, retain=C.RETAIN_ROW)}
BWD_ROWS = {"one_cta": G1, "cluster4": C.make_plan(C.PATH_CLUSTER, 4, retain=C.RETAIN_ROW, threads=0)}


@pytest.fixture(scope="module", autouse=True)
def _init():
    from paper_2609_01864_gb300 import build as B
    B.build()
    C.init()


def e4m3(rows, cols, seed):
    """Codes over the whole range (no NaN), +-448, the smallest subnormal and -0 in the first columns."""
    g = torch.Generator().manual_seed(seed)
    codes = torch.randint(0, 256, (rows, cols), generator=g, dtype=torch.int16)
    codes = torch.where((codes & 0x7F) == 0x7F, codes - 1, codes).to(torch.uint8)
    codes[:, :4] = torch.tensor([0x7E, 0xFE, 0x01, 0x80], dtype=torch.uint8)
    return codes.view(torch.float8_e4m3fn)


@pytest.mark.parametrize("plan", sorted(ROWS))
@pytest.mark.parametrize("cols", [4096, 20011])
@pytest.mark.parametrize("op,tout", [(C.SOFTMAX, C.FP8_E4M3), (C.SOFTMAX, C.F32), (C.LOGSUMEXP, C.F32),
                                     (C.LAYERNORM, C.FP8_E4M3), (C.RMSNORM, C.BF16)])
def test_fp8_rows_with_negative_and_zero_scales(op, tout, cols, plan):
    x = e4m3(12, cols, 21)
    sc = torch.tensor([-1.0, 0.0, 1e-3, -1e-3, 0.25, -0.25, 0.05, -0.02, 2.0 ** -20, -(2.0 ** -20), 0.01, -0.5])
    if op == C.SOFTMAX and tout == C.F32:
        sc = sc.clamp(-0.05, 0.05)  # |x - max| <= 45: every probability a normal FP32 number
    assert C.plan_kernel(op, x.cuda(), torch.empty(12, cols, device="cuda", dtype=C.TORCH_DTYPE[tout]), ROWS[plan],
                         in_scale=sc.cuda(), out_scale=sc.cuda(), out_dtype=tout) == "k_row_team"
    U.check_against_oracle(op, x, sc, out_dtype=tout, plan=ROWS[plan])


@pytest.mark.parametrize("plan", sorted(ROWS))
@pytest.mark.parametrize("op,tout", [(C.SOFTMAX, C.FP8_E4M3), (C.SOFTMAX, C.F32), (C.LOGSUMEXP, C.F32)])
def test_fp8_rows_whose_maximum_lies_below_the_scale_bound(op, tout, plan):
    spec = [(0x80, 0xFE, 0.1), (0x00, 0x60, 0.05), (0x00, 0x70, 0.01), (0x00, 0x7E, -0.1), (0x80, 0xFE, -0.002),
            (0x38, 0x48, 0.5), (0x40, 0x40, 0.3), (0x00, 0x68, 0.02)]  # lowest and highest code, scale
    g = torch.Generator().manual_seed(33)
    codes = torch.empty(len(spec), 20011, dtype=torch.uint8)
    for r, (lo, hi, _) in enumerate(spec):
        codes[r] = torch.randint(lo, hi + 1, (20011,), generator=g, dtype=torch.int16).to(torch.uint8)
    U.check_against_oracle(op, codes.view(torch.float8_e4m3fn), torch.tensor([s for _, _, s in spec]), out_dtype=tout,
                           plan=ROWS[plan])


def logits_reference(op, z, d, w):
    y = torch.softmax(z.double(), 1)
    d = d.double()
    if op == C.XENT_BWD:
        return w[:, None].double() * (y * d.sum(1, keepdim=True) - d)
    return y * (d - (y * d).sum(1, keepdim=True))


@pytest.mark.parametrize("plan", sorted(BWD_ROWS))
@pytest.mark.parametrize("op", [C.SOFTMAX_LOGITS_BWD, C.XENT_BWD])
@pytest.mark.parametrize("dtype", [C.F32, C.BF16])
@pytest.mark.parametrize("cols", [5000, 20003])
def test_masked_logits_and_nan(op, dtype, cols, plan):
    """-inf logits have the gradient -w t (0 from the softmax); whole slices of them, all but one, all (NaN), and a NaN
    that stays in its row.  Error: 1e-5 of the row's largest term, plus a BF16 ulp of it for BF16."""
    rows = 40
    a, dy, _, _, w = U.bwd_inputs(op, dtype, rows, cols, seed=cols)
    w = torch.ones(rows) if w is None else w
    z = a.clone()
    z[0, cols // 2:] = z[1, ::2] = z[2, :cols - 1] = z[3, 1:] = z[4] = z[5, cols // 4:cols // 2] = -torch.inf
    z[6, 7] = torch.nan
    z[7, 11] = torch.inf
    dx = torch.full((rows, cols), 7.0, device="cuda", dtype=z.dtype)
    kw = dict(scale=w.cuda()) if op == C.XENT_BWD else {}
    assert C.bwd_plan_kernel(op, z.cuda(), dy.cuda(), dx, BWD_ROWS[plan], **kw) == "k_bwd_team"
    C.run_bwd(op, z.cuda(), dy.cuda(), dx, plan=BWD_ROWS[plan], **kw)
    torch.cuda.synchronize()
    assert C.device_error() == C.OK
    ref, got = logits_reference(op, z, dy, w), dx.cpu().double()
    assert torch.equal(torch.isnan(got), torch.isnan(ref))
    ok = ~torch.isnan(ref).any(1)
    assert int(ok.sum()) == rows - 3
    y = torch.softmax(z.double(), 1)
    d = dy.double()
    if op == C.XENT_BWD:  # the terms w y sum(t) and w t
        S = w.double() * (y.amax(1) * d.sum(1).abs() + d.abs().amax(1))
    else:  # y dy and y sum(y dy)
        S = y.amax(1) * ((d * y).abs().sum(1) + d.abs().amax(1))
    bound = (1e-5 + (2.0 ** -8 if dtype == C.BF16 else 0.0)) * S[:, None] * torch.ones_like(ref)
    assert ((got - ref).abs() <= bound)[ok].all(), ((got - ref).abs() / bound)[ok].max()


@pytest.mark.parametrize("op", [C.LAYERNORM_BWD, C.SOFTMAX_LOGITS_BWD, C.XENT_BWD, C.WVAR_BWD, C.PEARSON_BWD])
@pytest.mark.parametrize("dtype", [C.F32, C.BF16])
@pytest.mark.parametrize("cols", [11, 4096, 5003])
def test_gradients_over_their_inputs(op, dtype, cols):
    rows = 400
    pair = op in (C.WVAR_BWD, C.PEARSON_BWD)
    if pair:
        a, dy, g = U.pair_inputs(op, dtype, rows, cols, seed=1)
        kw = dict(scale=g.cuda())
    else:
        a, dy, g, m, r = U.bwd_inputs(op, dtype, rows, cols, seed=1)
        kw = dict(scale=r.cuda()) if op == C.XENT_BWD else {
            k: v.cuda() for k, v in dict(gamma=g, mean=m, rstd=r).items() if v is not None}
    want, want2 = torch.empty(rows, cols, device="cuda", dtype=a.dtype), torch.empty(rows, cols, device="cuda", dtype=a.dtype)
    if pair:
        kw["dx2"] = want2
    ga, gd = a.cuda(), dy.cuda()
    assert C.bwd_plan_kernel(op, ga, gd, want, G1, **kw) == "k_bwd_team"
    C.run_bwd(op, ga, gd, want, plan=G1, **kw)
    for first in (True, False):  # dx over a (and dx2 over dy), dx over dy (and dx2 over a)
        x, d = a.cuda(), dy.cuda()
        if pair:
            kw["dx2"] = d if first else x
        C.run_bwd(op, x, d, x if first else d, plan=G1, **kw)
        torch.cuda.synchronize()
        assert torch.equal(x if first else d, want)
        assert not pair or torch.equal(d if first else x, want2)
    assert C.device_error() == C.OK


@pytest.mark.parametrize("op", [C.WVAR_BWD, C.PEARSON_BWD])
@pytest.mark.parametrize("dtype", [C.F32, C.BF16])
@pytest.mark.parametrize("rows,cols", [(330, 5), (330, 1021), (9, 40003)])
@pytest.mark.parametrize("off,off1,off2", [(0, 0, 0), (1, 1, 1), (3, 0, 2)])
def test_second_gradient_between_guards(op, dtype, rows, cols, off, off1, off2):
    """Nothing is written outside either gradient, each at its own phase of the 16-byte grid."""
    a, dy, g = U.pair_inputs(op, dtype, rows, cols, seed=cols)
    n = rows * cols
    bufs = [torch.full((o + n + 16,), float("nan"), device="cuda", dtype=a.dtype) for o in (off1, off2)]
    out = [b[o:o + n].view(rows, cols) for b, o in zip(bufs, (off1, off2))]
    C.run_bwd(op, shifted(a, off), shifted(dy, off), out[0], plan=G1, dx2=out[1], scale=g.cuda())
    torch.cuda.synchronize()
    assert C.device_error() == C.OK
    r1, r2 = U.pair_reference(op, a, dy, g, cols)
    assert U.pair_error(op, dtype, U.to64(out[0]), U.to64(out[1]), r1, r2, a, dy, g, cols) <= 1.0
    for b, o in zip(bufs, (off1, off2)):
        assert torch.isnan(b[:o].float()).all() and torch.isnan(b[o + n:].float()).all()
        assert not np.isnan(U.to64(b[o:o + n])).any()
