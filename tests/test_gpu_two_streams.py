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


MANY = r"""
import ctypes, sys, torch
from paper_2609_01864_gb300 import credit as C
C.init()
x = torch.randn(8, 120001, device="cuda") * 3
want, y = torch.empty_like(x), torch.empty_like(x)
split = C.make_plan(C.PATH_TWO_PASS, ctas_per_row=3)
C.run_ex(C.SOFTMAX, x, want, plan=split)
whole = torch.empty_like(x)
C.run_ex(C.SOFTMAX, x, whole, plan=C.make_plan(C.PATH_TWO_PASS))
torch.cuda.synchronize()
rt = ctypes.CDLL(next(l.split()[-1] for l in open("/proc/self/maps") if "libcudart" in l))
for k in range(560):  # more streams than workspaces: the one used longest ago goes to the new one
    s = ctypes.c_void_p()
    assert rt.cudaStreamCreateWithFlags(ctypes.byref(s), 1) == 0
    y.zero_()
    torch.cuda.synchronize()
    C.run_ex(C.SOFTMAX, x, y, plan=split, stream=s.value)
    assert rt.cudaStreamSynchronize(s) == 0 and rt.cudaStreamDestroy(s) == 0
    assert torch.equal(y, want), k
n = torch.randn(40, 300001, device="cuda").bfloat16()
g = torch.ones(300001, device="cuda")
p = C.plan(C.LAYERNORM, 40, 300001, C.BF16)
assert p.path == C.PATH_TWO_PASS and p.ctas_per_row > 1
ref = torch.layer_norm(n.double(), (300001,)).float()
z = torch.empty_like(n)
for k in range(530):  # more captures than workspaces: a planned call then runs one CTA per row
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        C.run_ex(C.LAYERNORM, n, z, gamma=g)
    if k % 40 == 0 or k > 505:
        z.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert (z.float() - ref).abs().max().item() <= 2.0 ** -6 * ref.abs().max().item(), k
assert C.device_error() == C.OK
print("ok")
"""


def test_more_streams_and_captures_than_workspaces():
    """In a process of its own: captured calls keep their workspaces for good."""
    import subprocess
    import sys
    r = subprocess.run([sys.executable, "-c", MANY], capture_output=True, text=True, timeout=300,
                       cwd=__import__("pathlib").Path(C.__file__).resolve().parents[1])
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stderr[-2000:]
