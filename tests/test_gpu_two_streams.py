"""Calls on several streams at a time, eager and captured: the planned split two-pass calls of wide rows off the 16-byte
grid exchange partials through device memory, which no two streams may share."""
import pytest
import torch

from paper_2609_01864_gb300 import credit as C
from paper_2609_01864_gb300 import synth

pytestmark = pytest.mark.gpu
CASES = [(C.LAYERNORM, C.F32, C.F32, 40, 300001), (C.QUANT_INT8, C.BF16, C.INT8, 40, 1200001)]


@pytest.fixture(scope="module", autouse=True)
def _init():
    from paper_2609_01864_gb300 import build as B
    B.build()
    C.init()


def calls(op, tin, tout, rows, cols, n):
    """n independent calls: (run(stream), outputs)."""
    out = []
    g, b = (t.cuda() for t in synth.gamma_beta(cols))
    for k in range(n):
        x = synth.outliers(rows, cols, seed=k, device="cuda").mul_(k + 1.0).to(C.TORCH_DTYPE[tin])
        y = torch.zeros(rows, cols, device="cuda", dtype=C.TORCH_DTYPE[tout])
        sc = torch.zeros(rows, device="cuda")
        kw = dict(in_dtype=tin, out_dtype=tout)
        kw.update(dict(gamma=g, beta=b) if op == C.LAYERNORM else dict(out_scale=sc))
        out.append((lambda s, x=x, y=y, kw=kw: C.run_ex(op, x, y, stream=s, **kw), (y, sc)))
    return out


@pytest.mark.parametrize("op,tin,tout,rows,cols", CASES)
def test_eager_and_captured_calls_overlap(op, tin, tout, rows, cols):
    C.load_model(str(__import__("pathlib").Path(C.__file__).parent / "data" / "gb300.calib"))
    p = C.plan(op, rows, cols, tin, tout)
    assert p.path == C.PATH_TWO_PASS and p.ctas_per_row > 1
    cs = calls(op, tin, tout, rows, cols, 4)
    streams = [torch.cuda.Stream() for _ in cs]
    want = []
    for run, outs in cs:  # one after the other
        run(None)
        torch.cuda.synchronize()
        want.append([t.clone() for t in outs])
        for t in outs:
            t.zero_()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        cs[3][0](None)
    torch.cuda.synchronize()
    for _ in range(25):
        for k in range(3):
            cs[k][0](streams[k])
        with torch.cuda.stream(streams[3]):
            graph.replay()
    torch.cuda.synchronize()
    assert C.device_error() == C.OK
    for (_, outs), w in zip(cs, want):
        assert all(torch.equal(a, b) for a, b in zip(outs, w))
