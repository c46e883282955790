"""What the library says about plans of whole rows and of rows over warps."""
import pytest
import torch

from paper_2609_01864_gb300 import credit as C

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _init():
    from paper_2609_01864_gb300 import build as B
    B.build()
    C.init()


@pytest.mark.parametrize("P,W,cols", [(1, 16, 20000), (1, 8, 20000), (2, 8, 50000), (8, 8, 200000), (8, 16, 300000),
                                      (16, 16, 880000)])
def test_max_clusters_of_rows_over_warps(P, W, cols):
    """One CTA of 16 warps per SM, or two of 8: all SMs at P = 1, and no cluster more than its CTAs' places (the GPC
    boundaries leave some of them out; at least half are there)."""
    x = torch.empty(2, cols, device="cuda")
    plan = C.make_plan(C.PATH_ONE_CTA if P == 1 else C.PATH_CLUSTER, P, retain=C.RETAIN_WARPS, threads=32 * W)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    places = sms * (16 // W) // P
    n = C.max_clusters(C.SOFTMAX, x, x, plan)
    assert n == places if P == 1 else places // 2 <= n <= places
    assert C.max_clusters(C.RMSNORM, x, x, plan) == 0  # no such kernel


def test_max_clusters_of_the_planned_plans():
    for op, rows, cols, dt in ((C.SOFTMAX, 2400, 131072, C.BF16), (C.LOGSUMEXP, 2400, 32003, C.BF16),
                               (C.RMSNORM, 16384, 4096, C.BF16)):
        x = torch.empty(rows, cols, device="cuda", dtype=C.TORCH_DTYPE[dt])
        y = torch.empty(rows, device="cuda") if op == C.LOGSUMEXP else x
        p = C.plan(op, rows, cols, dt)
        assert p.retain in (C.RETAIN_ROW, C.RETAIN_WARPS)
        assert C.plan_check(op, x, y, p) == C.OK and C.max_clusters(op, x, y, p) > 0
