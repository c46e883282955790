"""GPU parity of the backward ops' whole-row team kernel (one-CTA two-pass plans on rows that fit shared memory)
where it can go wrong: rows shorter than a 16-byte group, around a team's threads and around the widths at which the
number of teams changes, one row to many rows per team, rows that start anywhere on the 16-byte grid, and arrays at
unlike phases (which leave it).  Wider rows off the grid take the split path's shifted groups."""
import pytest
import torch

from paper_2609_01864_gb300 import credit as C

import parity_util as U

pytestmark = pytest.mark.gpu
OPS = [C.SOFTMAX_BWD, C.LAYERNORM_BWD, C.RMSNORM_BWD, C.SOFTMAX_LOGITS_BWD, C.XENT_BWD, C.WVAR_BWD, C.PEARSON_BWD]
PAIR = (C.WVAR_BWD, C.PEARSON_BWD)
G1 = C.make_plan(C.PATH_TWO_PASS, ctas_per_row=1)


@pytest.fixture(scope="module", autouse=True)
def _init():
    from paper_2609_01864_gb300 import build as B
    B.build()
    C.init()


def shifted(t, off):
    """t's values on the device, starting `off` elements after a 16-byte boundary."""
    buf = torch.empty(off + t.numel(), dtype=t.dtype, device="cuda")
    v = buf[off:].view(t.shape)
    v.copy_(t)
    return v


def check(op, dtype, rows, cols, plan, off=(0, 0, 0), seed=0):
    if op in PAIR:
        a, dy, g = U.pair_inputs(op, dtype, rows, cols, seed=seed)
        kw = dict(scale=g.cuda())
    else:
        a, dy, g, m, r = U.bwd_inputs(op, dtype, rows, cols, seed=seed)
        kw = dict(scale=r.cuda()) if op == C.XENT_BWD else {
            k: v.cuda() for k, v in dict(gamma=g, mean=m, rstd=r).items() if v is not None}
    ga, gd = shifted(a, off[0]), shifted(dy, off[1])
    guard = torch.full((2, off[2] + rows * cols + 16), float("nan"), device="cuda").to(a.dtype)
    out = [b[off[2]:off[2] + rows * cols].view(rows, cols) for b in guard]
    if op in PAIR:
        # the second output a whole number of 16-byte groups into its buffer plus the same offset
        kw["dx2"] = shifted(out[1], off[2])
    C.run_bwd(op, ga, gd, out[0], plan=plan, rows=rows, cols=cols, **kw)
    torch.cuda.synchronize()
    assert C.device_error() == C.OK
    if op in PAIR:
        r1, r2 = U.pair_reference(op, a, dy, g, cols)
        err = U.pair_error(op, dtype, U.to64(out[0]), U.to64(kw["dx2"]), r1, r2, a, dy, g, cols)
    else:
        ref = U.bwd_reference(op, dtype, a, dy, g, m, r, rows, cols)
        err = U.bwd_error(op, dtype, U.to64(out[0]), ref, a, dy, g, m, r, cols)
    assert err <= 1.0, err
    assert torch.isnan(guard[0, :off[2]].float()).all() and torch.isnan(guard[0, off[2] + rows * cols:].float()).all()


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("dtype", [C.F32, C.BF16])
@pytest.mark.parametrize("groups", [1, 127, 128, 1024, 1664, 4096, 6144])  # 16-byte groups of a row of one array
@pytest.mark.parametrize("extra", [-1, 0, 3])
def test_widths(op, dtype, groups, extra):
    rows = 640 if groups <= 128 else 330 if groups <= 1664 else 4
    check(op, dtype, rows, groups * (4 if dtype == C.F32 else 8) + extra, G1, seed=groups + extra)


@pytest.mark.parametrize("op", [C.LAYERNORM_BWD, C.XENT_BWD, C.PEARSON_BWD])
@pytest.mark.parametrize("rows,cols", [(1, 900), (151, 900), (153, 900), (6000, 900), (320, 12000)])
def test_rows(op, rows, cols):
    check(op, C.BF16, rows, cols, None, seed=rows)


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("off", [(3, 3, 3), (1, 1, 0), (2, 5, 2)])
@pytest.mark.parametrize("cols", [4093, 50021, 70001])  # the last two pass the team kernel's width in FP32
def test_any_phase(op, off, cols):
    for dtype in (C.F32, C.BF16):
        check(op, dtype, 9, cols, None, off=off, seed=cols)


@pytest.mark.parametrize("op", [C.LAYERNORM_BWD, C.SOFTMAX_LOGITS_BWD, C.WVAR_BWD])
def test_split_rows_off_the_grid(op):
    for dtype in (C.F32, C.BF16):
        check(op, dtype, 11, 90001, C.make_plan(C.PATH_TWO_PASS, ctas_per_row=3), off=(1, 1, 1), seed=5)


@pytest.mark.parametrize("op", [C.SOFTMAX_BWD, C.RMSNORM_BWD])
def test_in_place(op):
    a, dy, g, m, r = U.bwd_inputs(op, C.F32, 400, 5003, seed=2)
    kw = {k: v.cuda() for k, v in dict(gamma=g, rstd=r).items() if v is not None}
    ga, gd = a.cuda(), dy.cuda()
    out = torch.empty_like(ga)
    C.run_bwd(op, ga, gd, out, **kw)
    C.run_bwd(op, ga, gd, gd, **kw)
    assert torch.equal(out, gd)


# rows split over clusters: several rows at a time per CTA, one CTA per row's slice up to 16
@pytest.mark.parametrize("op", [C.SOFTMAX_BWD, C.SOFTMAX_LOGITS_BWD, C.XENT_BWD])
@pytest.mark.parametrize("dtype", [C.F32, C.BF16])
@pytest.mark.parametrize("P,rows,kb,extra", [(2, 5, 70, 1), (2, 700, 64, 0), (4, 320, 96, 3), (16, 130, 64, -1),
                                             (16, 7, 900, 5), (8, 1, 200, 0)])
def test_cluster_rows(op, dtype, P, rows, kb, extra):
    plan = C.make_plan(C.PATH_CLUSTER, P, retain=C.RETAIN_ROW, threads=0)
    cols = kb * 1024 // (4 if dtype == C.F32 else 2) + extra
    check(op, dtype, rows, cols, plan, off=(1, 1, 2) if extra else (0, 0, 0), seed=rows)


@pytest.mark.parametrize("op", [C.SOFTMAX_BWD, C.SOFTMAX_LOGITS_BWD, C.XENT_BWD])
def test_cluster_rows_chosen(op):
    for dtype in (C.F32, C.BF16):
        cols = 150 * 1024 // (4 if dtype == C.F32 else 2) + 1
        check(op, dtype, 640, cols, None, seed=1)
        check(op, dtype, 6, cols, None, off=(1, 2, 1), seed=2)  # unlike phases: another path


def test_cluster_rows_refused():
    x = torch.zeros(4, 40000, device="cuda")
    m = torch.zeros(4, device="cuda")
    plan = C.make_plan(C.PATH_CLUSTER, 4, retain=C.RETAIN_ROW, threads=0)
    n0 = C.launch_count()
    assert C.run_bwd_status(C.RMSNORM_BWD, x, x, x, plan=plan, rstd=m) == C.ERR_UNSUPPORTED
    odd = torch.zeros(4 * 40000 + 1, device="cuda")[1:].view(4, 40000)
    assert C.run_bwd_status(C.XENT_BWD, x, odd, x, plan=plan) == C.ERR_UNSUPPORTED
    assert C.launch_count() == n0
