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
