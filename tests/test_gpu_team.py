"""GPU parity of the whole-row team kernel (one-CTA plans with CREDIT_RETAIN_ROW) where it can go wrong: rows
shorter than a 16-byte group, one group and one thread short of or past a team's threads, the widths at which the
threads per row, the stages and the place of gamma / beta change, one row to many rows per team, and rows that
start and end anywhere on the 16-byte grid of either tensor."""
import pytest
import torch

from paper_2609_01864_gb300 import credit as C
from paper_2609_01864_gb300 import synth

import parity_util as U

pytestmark = pytest.mark.gpu
ROW = C.make_plan(C.PATH_ONE_CTA, retain=C.RETAIN_ROW)
OPS = [C.SOFTMAX, C.LOGSUMEXP, C.LAYERNORM, C.RMSNORM]
SIZE = {C.F32: 4, C.BF16: 2, C.FP8_E4M3: 1}


@pytest.fixture(scope="module", autouse=True)
def _init():
    from paper_2609_01864_gb300 import build as B
    B.build()
    C.init()


def _case(op, tin, tout, rows, cols, seed):
    norm = op in (C.LAYERNORM, C.RMSNORM)
    x, s = U.make_input(tin, rows, cols, kind="outliers" if norm else "normal", std=3.0, seed=seed)
    g, b = synth.gamma_beta(cols, seed=seed + 1) if norm else (None, None)
    return x, s, g, (b if op == C.LAYERNORM else None)


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("tin,tout", [(C.F32, C.F32), (C.BF16, C.BF16), (C.FP8_E4M3, C.FP8_E4M3), (C.BF16, C.FP8_E4M3),
                                      (C.FP8_E4M3, C.BF16)])
@pytest.mark.parametrize("kib16", [0, 1, 127, 128, 1024, 1025, 4096])  # 16-byte groups of a row
@pytest.mark.parametrize("extra", [-1, 0, 3])
def test_widths(op, tin, tout, kib16, extra):
    cols = kib16 * 16 // SIZE[tin] + extra
    if cols < 1:
        cols = 1 if extra < 0 else 2
    rows = 700 if kib16 <= 128 else 310 if kib16 <= 1025 else 5
    if op == C.LOGSUMEXP:
        tout = C.F32
    x, s, g, b = _case(op, tin, tout, rows, cols, cols * 3 + tin)
    U.check_against_oracle(op, x, s, out_dtype=tout, plan=ROW, gamma=g, beta=b)


@pytest.mark.parametrize("op", [C.SOFTMAX, C.LAYERNORM, C.RMSNORM])
@pytest.mark.parametrize("rows,cols", [(1, 1000), (151, 1000), (153, 1000), (5000, 1000), (9, 24500)])
@pytest.mark.parametrize("stages", [0, 1, 3, 4])
def test_rows_and_stages(op, rows, cols, stages):
    x, s, g, b = _case(op, C.BF16, C.BF16, rows, cols, rows)
    plan = C.make_plan(C.PATH_ONE_CTA, retain=C.RETAIN_ROW, ring_chunks=stages)
    U.check_against_oracle(op, x, s, plan=plan, gamma=g, beta=b)


@pytest.mark.parametrize("op", [C.SOFTMAX, C.LAYERNORM, C.RMSNORM])
@pytest.mark.parametrize("tin,tout", [(C.F32, C.F32), (C.BF16, C.BF16), (C.BF16, C.FP8_E4M3)])
@pytest.mark.parametrize("off_in,off_out,ld_in,ld_out", [(1, 0, 0, 0), (0, 1, 0, 0), (3, 3, 4099, 4101), (0, 0, 4096, 4099)])
def test_any_phase(op, tin, tout, off_in, off_out, ld_in, ld_out):
    """Rows at every element offset of the 16-byte grid, the output's offset unlike the input's, gamma / beta off
    the grid too, and nothing outside a row written."""
    rows, cols = 320, 4093
    x, _, g, b = _case(op, tin, tout, rows, cols, off_in + 7 * off_out)
    li, lo = ld_in or cols, ld_out or cols
    buf = torch.zeros(off_in + rows * li, dtype=x.dtype, device="cuda")
    xin = buf[off_in:].view(rows, li)
    xin[:, :cols] = x.cuda()
    guard = torch.full((off_out + rows * lo,), 3.0, device="cuda").to(C.TORCH_DTYPE[tout])
    y = guard[off_out:].view(rows, lo)
    osc = torch.empty(rows, device="cuda") if tout == C.FP8_E4M3 else None
    gd = None if g is None else torch.cat([g[:1], g]).cuda()[1:]
    bd = None if b is None else torch.cat([b[:1], b]).cuda()[1:]
    C.run_ex(op, xin, y, plan=ROW, rows=rows, cols=cols, ld_in=ld_in, ld_out=ld_out, in_dtype=tin, out_dtype=tout,
             out_scale=osc, gamma=gd, beta=bd)
    torch.cuda.synchronize()
    assert C.device_error() == C.OK
    ref = U.reference(op, tin, x, None, g, b)
    m = U.error_metric(op, tout, U.to64(y[:, :cols]), ref, None if osc is None else osc.cpu().numpy(),
                       x64=U.decoded(x) if op == C.LAYERNORM else None, gamma=g, beta=b)
    assert m <= 1.0
    assert (guard[:off_out].float() == 3.0).all() and (y[:, cols:].float() == 3.0).all()


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("tin,tout", [(C.F32, C.F32), (C.BF16, C.BF16), (C.FP8_E4M3, C.FP8_E4M3), (C.BF16, C.FP8_E4M3)])
@pytest.mark.parametrize("P", [2, 4, 8, 16])
@pytest.mark.parametrize("groups,extra,rows", [(32, 0, 700), (131, 3, 700), (1023, 1, 90), (2049, -1, 7)])
def test_clusters(op, tin, tout, P, groups, extra, rows):
    """Rows split over a cluster: `groups` 16-byte groups per CTA (32: the fewest the plan takes as such), slices of
    unlike sizes, several rows per team so that every exchange slot and stage is reused, rows off the grid."""
    cols = P * groups * 16 // SIZE[tin] + extra
    if op == C.LOGSUMEXP:
        tout = C.F32
    x, s, g, b = _case(op, tin, tout, rows, cols, cols + P)
    plan = C.make_plan(C.PATH_CLUSTER, P, retain=C.RETAIN_ROW)
    y = torch.empty(1, device="cuda")
    if C.plan_check(op, x.cuda(), y, plan, out_dtype=tout, in_scale=None if s is None else s.cuda(),
                    out_scale=y) != C.OK:
        pytest.skip("gamma / beta and a slice exceed shared memory, and so does AUTO")
    U.check_against_oracle(op, x, s, out_dtype=tout, plan=plan, gamma=g, beta=b)


@pytest.mark.parametrize("op", [C.SOFTMAX, C.LAYERNORM, C.RMSNORM])
@pytest.mark.parametrize("dt", [C.F32, C.BF16])
def test_planned_rows_off_the_grid(op, dt):
    """The planner's choice on wide rows off the 16-byte grid is a cluster of this kernel
    (softmax: of rows over warps) and matches the oracle."""
    cols = 140 * 1024 // SIZE[dt] - 3
    p = C.plan(op, 700, cols, dt)
    assert (p.path, p.retain) == (C.PATH_CLUSTER, C.RETAIN_WARPS if op == C.SOFTMAX else C.RETAIN_ROW)
    x, s, g, b = _case(op, dt, dt, 48, cols, 5)
    U.check_against_oracle(op, x, s, gamma=g, beta=b)


@pytest.mark.parametrize("dt", [C.F32, C.BF16])
@pytest.mark.parametrize("cols", [8, 100, 4096, 20001, 60001])
def test_int8_and_in_place(dt, cols):
    import numpy as np
    import oracle as O
    x, _ = U.make_input(dt, 200, cols, kind="outliers", seed=cols)
    x[5] = 0
    d = x.cuda()
    y, sc = torch.empty(200, cols, dtype=torch.int8, device="cuda"), torch.empty(200, device="cuda")
    plan = ROW if cols < 60000 else C.make_plan(C.PATH_CLUSTER, 4, retain=C.RETAIN_ROW)
    C.run_ex(C.QUANT_INT8, d, y, plan=plan, in_dtype=dt, out_dtype=C.INT8, out_scale=sc)
    codes, scales = O.quant_int8(x.float().numpy())
    assert np.array_equal(y.cpu().numpy(), codes) and np.array_equal(sc.cpu().numpy(), scales)
    z = torch.empty_like(d)
    C.run_ex(C.SOFTMAX, d, z, plan=plan)
    C.run_ex(C.SOFTMAX, d, d, plan=plan)  # in == out
    assert torch.equal(d, z)


def test_rows_of_infinities():
    """-inf everywhere gives NaN outputs and a log-sum-exp of -inf; some -inf are zeros of the softmax; a NaN makes
    its own row NaN and no other."""
    x = torch.randn(64, 5000)
    x[3], x[9, ::2], x[11, 77] = -float("inf"), -float("inf"), float("nan")
    for op in (C.SOFTMAX, C.LOGSUMEXP):
        y, _ = U.run_gpu(op, x, None, plan=ROW)
        ref = torch.softmax(x.double(), 1) if op == C.SOFTMAX else torch.logsumexp(x.double(), 1)
        y = y.cpu().double()
        assert torch.equal(torch.isnan(y), torch.isnan(ref))
        ok = torch.isfinite(ref)
        assert torch.equal(torch.isfinite(y), ok) and (y - ref)[ok].abs().max() <= 1e-5 * ref[ok].abs().max()
