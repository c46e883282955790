"""What making a ragged batch has to leave behind: the work list on the device before any launch reads it."""
import pytest
import torch

from paper_2609_01864_gb300 import credit as C

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _init():
    from paper_2609_01864_gb300 import build as B
    B.build()
    C.init()


@pytest.mark.parametrize("threads", ["256", "512"])
def test_run_on_another_stream_right_after_making(monkeypatch, threads):
    """Handles made and run one after the other, each with another row table over the same data."""
    monkeypatch.setenv("CREDIT_RAGGED_THREADS", threads)
    n, total = 4000, 1 << 20
    x = torch.randn(total, device="cuda")
    want = {}
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    for k in range(12):
        w = 200 + 7 * (k % 3)
        rows = [((i * 211 + k % 3) % (total - w), i * w, w, C.SOFTMAX) for i in range(n)]
        y = torch.zeros(n * w, device="cuda")
        torch.cuda.synchronize()
        R = C.Ragged(rows, C.F32, x, y, tune=False)
        R.run(stream)
        torch.cuda.synchronize()
        assert C.device_error() == C.OK
        R.close()
        if k < 3:
            ref = torch.softmax(torch.stack([x[i:i + w] for i, _, _, _ in rows]).double(), 1)
            assert (y.view(n, w).double() - ref).abs().max().item() < 1e-5
            want[k] = y
        else:
            assert torch.equal(y, want[k % 3])


@pytest.mark.parametrize("rows,lo,hi", [(3000, 20000, 500000)])
def test_autotuning_costs_a_bounded_number_of_runs(rows, lo, hi):
    """Shapes that fall behind are not run to the end: 74 shapes in fewer than 330 runs' time of the chosen one."""
    import math
    import random
    import time
    rng = random.Random(7)
    table, off = [], 0
    for _ in range(rows):
        w = int(lo * 2 ** (rng.random() * math.log2(hi / lo)))
        table.append((off, off, w, C.SOFTMAX if rng.random() < 0.5 else C.RMSNORM))
        off += w
    x = torch.randn(off, device="cuda").bfloat16()
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    C.Ragged(table[:50], C.BF16, x, y).close()  # kernels loaded
    t0 = time.perf_counter()
    R = C.Ragged(table, C.BF16, x, y)
    made = time.perf_counter() - t0
    for _ in range(3):
        R.run()
    torch.cuda.synchronize()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    for _ in range(10):
        R.run()
    b.record()
    torch.cuda.synchronize()
    one = a.elapsed_time(b) / 10 * 1e-3
    R.close()
    assert made < 330 * one, (made, one)


@pytest.mark.parametrize("W", [8, 16])
def test_info_of_rows_over_warps(monkeypatch, W):
    """threads = 512 marks the kind; staging_bytes are those of the launch's own CTAs, of W buffers of 14080 bytes."""
    for k, v in dict(THREADS=512, P=0, W=W).items():
        monkeypatch.setenv("CREDIT_RAGGED_" + k, str(v))
    x = torch.zeros(9000, device="cuda")
    R = C.Ragged([(0, 0, 9000, C.RMSNORM)], C.F32, x, x, tune=False)
    info = R.info()
    R.close()
    assert (info["threads"], info["staging_bytes"], info["tuned_us"]) == (512, W * 14080, 0.0)
