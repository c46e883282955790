"""credit_set_trace on launches of whole rows and of rows over warps: the stamps of the first 32 CTAs' first rows, in the
order of a row's phases, and nothing else written."""
import pytest
import torch

from paper_2609_01864_gb300 import credit as C

pytestmark = pytest.mark.gpu
CTAS, FIELDS, R = 32, 8, 3


@pytest.fixture(scope="module", autouse=True)
def _init():
    from paper_2609_01864_gb300 import build as B
    B.build()
    C.init()
    yield
    C.set_trace(None)


@pytest.mark.parametrize("op,retain,P,cols", [(C.RMSNORM, C.RETAIN_ROW, 1, 1000), (C.LAYERNORM, C.RETAIN_ROW, 2, 20001),
                                              (C.LOGSUMEXP, C.RETAIN_ROW, 1, 12000), (C.SOFTMAX, C.RETAIN_WARPS, 1, 4001),
                                              (C.SOFTMAX, C.RETAIN_WARPS, 8, 70000),
                                              (C.LOGSUMEXP, C.RETAIN_WARPS, 1, 16384)])
def test_stamps(op, retain, P, cols):
    x = torch.randn(40000 if P == 1 else 3000, cols, device="cuda").bfloat16()
    y = torch.empty(x.shape[0], device="cuda") if op == C.LOGSUMEXP else torch.empty_like(x)
    plan = C.make_plan(C.PATH_ONE_CTA if P == 1 else C.PATH_CLUSTER, P, retain=retain)
    buf = torch.zeros(CTAS * R * FIELDS + 8, dtype=torch.int64, device="cuda")
    C.set_trace(buf[:CTAS * R * FIELDS])
    try:
        C.run_ex(op, x, y, plan=plan)
        torch.cuda.synchronize()
    finally:
        C.set_trace(None)
    assert C.device_error() == C.OK
    t = buf[:CTAS * R * FIELDS].view(CTAS, R, FIELDS).cpu()
    assert (buf[CTAS * R * FIELDS:] == 0).all() and (t[..., [1, 2, 6, 7]] == 0).all()
    phases = t[..., [0, 5, 3, 4]]
    assert (phases > 0).all()
    assert (phases.diff(dim=2) >= 0).all() and (t[:, 1:, 0] >= t[:, :-1, 4]).all()
    assert int(phases.max() - phases.min()) < 100_000_000  # one launch: well under a tenth of a second
    buf.zero_()
    C.run_ex(op, x, y, plan=plan)  # off again
    torch.cuda.synchronize()
    assert (buf == 0).all()
