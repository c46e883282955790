"""GPU parity of the two-pass norms whose gamma / beta lie off the 16-byte grid (shifted vectors, at another phase in
every row): every phase, the array's ends, null gamma or beta, every type, one CTA and several per row; and of the
calls that the planner gives the two-pass path for it."""
import pytest
import torch

from paper_2609_01864_gb300 import credit as C
from paper_2609_01864_gb300 import synth

import parity_util as U

pytestmark = pytest.mark.gpu
TYPES = [(C.F32, C.F32), (C.BF16, C.BF16), (C.BF16, C.FP8_E4M3), (C.FP8_E4M3, C.FP8_E4M3), (C.FP8_E4M3, C.F32)]


@pytest.fixture(scope="module", autouse=True)
def _init():
    from paper_2609_01864_gb300 import build as B
    B.build()
    C.init()


def check(op, tin, tout, rows, cols, plan, g_off=0, b_off=0, affine="gb", seed=0):
    x, sc = U.make_input(tin, rows, cols, seed=seed)
    g, b = synth.gamma_beta(cols, seed=seed + 1)
    g, b = (g if "g" in affine else None), (b if "b" in affine and op == C.LAYERNORM else None)

    def at(t, off):  # the array starts `off` floats after a 16-byte boundary, between NaNs
        if t is None:
            return None
        buf = torch.full((off + cols + 8,), float("nan"), device="cuda")
        buf[off:off + cols] = t.cuda()
        return buf[off:off + cols]

    y, osc = U.run_gpu(op, x, sc, out_dtype=tout, plan=plan, gamma=at(g, g_off), beta=at(b, b_off))
    torch.cuda.synchronize()
    assert C.device_error() == C.OK
    ref = U.reference(op, tin, x, sc, g, b)
    err = U.error_metric(op, tout, U.to64(y), ref, None if osc is None else osc.cpu().numpy(),
                         x64=U.decoded(x, sc) if op == C.LAYERNORM else None, gamma=g, beta=b)
    assert err <= 1.0, err


@pytest.mark.parametrize("op", [C.LAYERNORM, C.RMSNORM])
@pytest.mark.parametrize("tin,tout", TYPES)
@pytest.mark.parametrize("cols", [1, 19, 67, 4097, 9003])
@pytest.mark.parametrize("G", [1, 3])
def test_phases(op, tin, tout, cols, G):
    if cols == 1 and op == C.LAYERNORM:
        pytest.skip("x - mean of a single column is rounding alone, times 1 / sqrt(eps): the bounds do not cover it")
    plan = C.make_plan(C.PATH_TWO_PASS, ctas_per_row=G)
    for g_off, b_off in ((0, 0), (1, 2), (3, 0)):
        check(op, tin, tout, 17, cols, plan, g_off, b_off, seed=cols)
    check(op, tin, tout, 5, cols, plan, 1, 3, affine="b", seed=cols)
    check(op, tin, tout, 5, cols, plan, 3, 1, affine="g", seed=cols)


@pytest.mark.parametrize("op,tin,tout,cols", [(C.LAYERNORM, C.F32, C.F32, 400001), (C.LAYERNORM, C.BF16, C.FP8_E4M3, 500003),
                                              (C.LAYERNORM, C.FP8_E4M3, C.FP8_E4M3, 400001)])
def test_wide_rows_as_planned(op, tin, tout, cols):
    assert C.plan(op, 12, cols, tin, tout).path == C.PATH_TWO_PASS
    check(op, tin, tout, 12, cols, None)


@pytest.mark.parametrize("tin,cols", [(C.F32, 280001), (C.BF16, 600001)])
def test_wide_int8_rows_as_planned(tin, cols):
    """int8 rows off the grid: codes and scales equal those of the same rows on the grid (padded stride)."""
    x, _ = U.make_input(tin, 9, cols, seed=3)
    ld = (cols + 15) // 16 * 16
    out = []
    for stride, plan in ((cols, None), (ld, C.make_plan(C.PATH_TWO_PASS, ctas_per_row=1))):
        xs = torch.zeros(9, stride, dtype=x.dtype, device="cuda")
        xs[:, :cols] = x.cuda()
        y = torch.zeros(9, stride, dtype=torch.int8, device="cuda")
        s = torch.zeros(9, device="cuda")
        C.run_ex(C.QUANT_INT8, xs, y, plan=plan, in_dtype=tin, out_dtype=C.INT8, out_scale=s, rows=9, cols=cols,
                 ld_in=stride, ld_out=stride)
        torch.cuda.synchronize()
        out.append((y[:, :cols].cpu(), s.cpu()))
    assert C.device_error() == C.OK
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
