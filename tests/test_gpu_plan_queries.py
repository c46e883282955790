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


SIZE = {C.F32: 4, C.BF16: 2, C.FP8_E4M3: 1}
TYPES = [(C.F32, C.F32), (C.BF16, C.BF16), (C.FP8_E4M3, C.FP8_E4M3), (C.BF16, C.FP8_E4M3), (C.FP8_E4M3, C.BF16)]
OPS = [C.SOFTMAX, C.LOGSUMEXP, C.LAYERNORM, C.RMSNORM]


def kernel_of(op, tin, tout, rows, cols, plan, off=0):
    x = torch.empty(rows * cols + off, device="cuda", dtype=C.TORCH_DTYPE[tin])[off:].view(rows, cols)
    y = torch.empty(rows, cols, device="cuda", dtype=C.TORCH_DTYPE[tout])
    s = torch.empty(rows, device="cuda")
    return C.plan_kernel(op, x, y, plan, in_dtype=tin, out_dtype=C.F32 if op == C.LOGSUMEXP else tout, in_scale=s,
                         out_scale=s)


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("tin,tout", TYPES)
def test_whole_rows_run_as_whole_rows(op, tin, tout):
    """One CTA's rows: the team kernel at every width of the parity tests (a stage of 64 KiB and, where gamma / beta do
    not fit beside it, reads through L2), and the ring beyond shared memory."""
    for groups in (0, 1, 127, 128, 1024, 1025, 4096):
        for extra in (-1, 0, 3):
            cols = max(groups * 16 // SIZE[tin] + extra, 1)
            for rows, stages in ((5, 0), (310, 0), (700, 1), (5000, 4)) if groups <= 1025 else ((5, 0), (310, 1)):
                p = C.make_plan(C.PATH_ONE_CTA, retain=C.RETAIN_ROW, ring_chunks=stages)
                assert kernel_of(op, tin, tout, rows, cols, p, off=extra % 4) == "k_row_team", (groups, extra, rows)
    wide = 232448 // SIZE[tin]  # the opt-in shared memory of a CTA, control area and all
    assert kernel_of(op, tin, tout, 2, wide, C.make_plan(C.PATH_ONE_CTA, retain=C.RETAIN_ROW)) != "k_row_team"


@pytest.mark.parametrize("op", OPS)
@pytest.mark.parametrize("tin,tout", TYPES[:4])
@pytest.mark.parametrize("P", [2, 4, 8, 16])
@pytest.mark.parametrize("groups,extra,rows", [(32, 0, 700), (131, 3, 700), (1023, 1, 90), (2049, -1, 7)])
def test_clusters_run_as_whole_rows(op, tin, tout, P, groups, extra, rows):
    """Rows over a cluster: the team kernel wherever a slice and its gamma / beta fit shared memory beside at most 34 KiB
    of barriers and exchange, another one where the two alone do not."""
    cols = P * groups * 16 // SIZE[tin] + extra
    nab = {C.LAYERNORM: 2, C.RMSNORM: 1}.get(op, 0)
    need = groups * 16 + nab * groups * 16 // SIZE[tin] * 4
    k = kernel_of(op, tin, tout, rows, cols, C.make_plan(C.PATH_CLUSTER, P, retain=C.RETAIN_ROW))
    if need + (36 << 10) <= 232448:
        assert k == "k_row_team"
    elif need > 232448:
        assert k in ("", "k_ring", "k_ring_tm")


@pytest.mark.parametrize("op", [C.SOFTMAX_BWD, C.LAYERNORM_BWD, C.RMSNORM_BWD, C.SOFTMAX_LOGITS_BWD, C.XENT_BWD, C.WVAR_BWD,
                                C.PEARSON_BWD])
@pytest.mark.parametrize("dt", [C.F32, C.BF16])
def test_backward_rows_run_as_whole_rows(op, dt):
    """Backward: one CTA's rows up to 96 KiB per array, any phase that a and dy share; clusters for the ops that have
    them."""
    v = torch.empty(700, device="cuda")
    kw = dict(scale=v, mean=v, rstd=v)

    def kernel(rows, cols, plan, off=(0, 0)):
        t = [torch.empty(rows * cols + 8, device="cuda", dtype=C.TORCH_DTYPE[dt])[o:o + rows * cols].view(rows, cols)
             for o in (off[0], off[1], off[0])]
        return C.bwd_plan_kernel(op, *t, plan, dx2=t[2], **kw)
    g1 = C.make_plan(C.PATH_TWO_PASS, ctas_per_row=1)
    V = 16 // SIZE[dt]
    for groups in (1, 127, 128, 1024, 1664, 4096, 6144):
        for rows in (4, 700) if groups < 2000 else (4,):
            assert kernel(rows, groups * V, g1) == kernel(rows, groups * V - 1, g1, (1, 1)) == "k_bwd_team"
    assert kernel(9, 999, g1, (1, 2)) == kernel(9, 6144 * V + 1, g1) == "k_bwd_tp_fused"
    has = op in (C.SOFTMAX_BWD, C.SOFTMAX_LOGITS_BWD, C.XENT_BWD)
    for P, kb in ((2, 70), (4, 96), (16, 900)):
        p = C.make_plan(C.PATH_CLUSTER, P, retain=C.RETAIN_ROW, threads=0)
        assert kernel(7, kb * 1024 // SIZE[dt] + 1, p, (1, 1)) == ("k_bwd_team" if has else "")
    assert kernel(5, 1024, C.make_plan(C.PATH_CLUSTER, 2)) == "k_bwd_staged"
    assert kernel(5, 1024, C.make_plan(C.PATH_TWO_PASS, ctas_per_row=3)) == "k_bwd_tp_stats"


def test_kernels_of_other_plans():
    x = torch.empty(8, 65536, device="cuda")
    for plan, want in ((C.make_plan(C.PATH_CLUSTER, 4, retain=C.RETAIN_SMEM), "k_ring"),
                       (C.make_plan(C.PATH_CLUSTER, 4, retain=C.RETAIN_TMEM), "k_ring_tm"),
                       (C.make_plan(C.PATH_CLUSTER, 8, retain=C.RETAIN_WARPS), "k_row_warps"),
                       (C.make_plan(C.PATH_TWO_PASS), "k_tp_fused"),
                       (C.make_plan(C.PATH_TWO_PASS, ctas_per_row=4), "k_tp_stats"),
                       (C.make_plan(C.PATH_CLUSTER, 3, retain=C.RETAIN_WARPS), "")):
        assert C.plan_kernel(C.SOFTMAX, x, x, plan) == want


@pytest.mark.parametrize("op,dt,rows,nbytes,warps", [
    (C.SOFTMAX, C.F32, 600, 98 << 10, True), (C.SOFTMAX, C.F32, 400, 128 << 10, True), (C.SOFTMAX, C.F32, 304, 128 << 10, False),
    (C.SOFTMAX, C.F32, 600, 288 << 10, True), (C.SOFTMAX, C.F32, 600, 448 << 10, False), (C.SOFTMAX, C.F32, 600, 560 << 10, True),
    (C.SOFTMAX, C.F32, 600, 1024 << 10, False), (C.SOFTMAX, C.BF16, 2600, 88 << 10, False),
    (C.SOFTMAX, C.BF16, 2600, (88 << 10) + 2, True), (C.SOFTMAX, C.BF16, 600, 88 << 10, True),
    (C.SOFTMAX, C.BF16, 600, 1024 << 10, True), (C.SOFTMAX, C.BF16, 600, 1740 << 10, True),
    (C.QUANT_INT8, C.F32, 600, 98 << 10, True), (C.QUANT_INT8, C.F32, 600, 896 << 10, False),
    (C.QUANT_INT8, C.F32, 600, 1000 << 10, True), (C.QUANT_INT8, C.F32, 600, 1024 << 10, False),
    (C.QUANT_INT8, C.BF16, 200, (160 << 10) + 2, False), (C.QUANT_INT8, C.BF16, 400, (160 << 10) + 2, True),
    (C.LOGSUMEXP, C.F32, 600, 128 << 10, False), (C.LOGSUMEXP, C.F32, 1300, 128 << 10, True),
    (C.LOGSUMEXP, C.BF16, 600, 36 << 10, False), (C.LOGSUMEXP, C.BF16, 600, 48 << 10, True),
    (C.LOGSUMEXP, C.BF16, 600, 57 << 10, True), (C.LOGSUMEXP, C.F32, 600, 57 << 10, False)])
def test_rows_over_warps_are_planned_by_their_buffers(op, dt, rows, nbytes, warps):
    """Both sides of the planner's lines: how many warps' buffers a row takes, and how full they are."""
    p = C.plan(op, rows, nbytes // SIZE[dt], dt, C.INT8 if op == C.QUANT_INT8 else None)
    assert (p.retain == C.RETAIN_WARPS) == warps


@pytest.mark.parametrize("dt,rows,nbytes,P", [
    (C.BF16, 1300, 66 << 10, 2), (C.BF16, 1300, 112 << 10, 0), (C.BF16, 1300, 116 << 10, 4), (C.BF16, 1300, 192 << 10, 4),
    (C.BF16, 1300, 224 << 10, 0), (C.BF16, 1300, 256 << 10, 8), (C.BF16, 1300, 264 << 10, 0), (C.BF16, 1300, 300 << 10, 8),
    (C.BF16, 300, 192 << 10, 0), (C.BF16, 300, 300 << 10, 8), (C.F32, 1300, 256 << 10, 0), (C.F32, 1300, 264 << 10, 8),
    (C.F32, 300, 420 << 10, 16), (C.F32, 1300, 1000 << 10, 0)])
def test_logits_rows_over_clusters_are_planned_by_their_slices(dt, rows, nbytes, P):
    """Both sides of the backward planner's lines: how much of shared memory the slices in flight fill."""
    p = C.plan_bwd(C.XENT_BWD, rows, nbytes // SIZE[dt], dt)
    assert (p.cluster_size if p.retain == C.RETAIN_ROW else 0) == P
