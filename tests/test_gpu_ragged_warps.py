"""GPU parity of the ragged batches' rows-over-warps launch, row by row against the FP64 oracle, where it can go
wrong: widths around a segment of half and of all a warp's buffer at every number of warps, rows without a whole
16-byte group, classes with fewer rows than groups of warps, rows that start anywhere on the 16-byte grid, outputs at
another phase than their inputs, rows of infinities, and the refusal of rows too wide for it."""
import numpy as np
import pytest
import torch

from paper_2609_01864_gb300 import credit as C

import parity_util as U

pytestmark = pytest.mark.gpu
HALF, WARPS = 440, 16  # 16-byte groups of half a warp's buffer, warps per CTA


@pytest.fixture(scope="module", autouse=True)
def _init():
    from paper_2609_01864_gb300 import build as B
    B.build()
    C.init()


def shape(monkeypatch, P=0, q=4, tight=0, spread=0, W=WARPS):
    for k, v in dict(THREADS=32 * WARPS, P=P, W=W, Q=q, TIGHT=tight, SPREAD=spread).items():
        monkeypatch.setenv("CREDIT_RAGGED_" + k, str(v))


def run(x, rows, dtype, out_len):
    d_in, d_out = x.cuda(), torch.full((out_len,), float("nan"), device="cuda").to(x.dtype)
    R = C.Ragged(rows, dtype, d_in, d_out, tune=False)
    for _ in range(2):  # the second run finds the first one's results
        R.run()
    torch.cuda.synchronize()
    info = R.info()
    R.close()
    assert C.device_error() == C.OK and info["threads"] == 32 * WARPS and info["items"] == len(rows)
    return d_out.cpu(), info


def batch(widths, seed, dtype, out_shift=0):
    rng = np.random.default_rng(seed)
    rows, i, o = [], 0, out_shift
    for w in rng.permutation(widths):
        rows.append((i, o, int(w), C.SOFTMAX if rng.random() < 0.5 else C.RMSNORM))
        i += int(w)
        o += int(w)
    g = torch.Generator().manual_seed(seed)
    return (torch.randn(i, generator=g) * 2.0).to(C.TORCH_DTYPE[dtype]), rows, o


def check(x, y, rows, dtype):
    written = torch.zeros(y.numel(), dtype=torch.bool)
    for i, o, w, op in rows:
        ref = U.reference(op, dtype, x[i:i + w].reshape(1, w))
        assert U.error_metric(op, dtype, U.to64(y[o:o + w].reshape(1, w)), ref) <= 1.0, (w, op)
        written[o:o + w] = True
    assert torch.isnan(y.float()[~written]).all()


def widths_for(dtype, most):
    V = 4 if dtype == C.F32 else 8
    out = [1, 2, V - 1, V, V + 1, 31 * V + 1, 32 * V]
    u = 1
    while u <= most:
        out += [V * HALF * u - V - 1, V * HALF * u, V * HALF * u + 3]
        u *= 2
    return out


@pytest.mark.parametrize("q,tight,spread,W", [(1, 0, 0, 16), (4, 0, 0, 8), (16, 0, 0, 16), (2, 1, 0, 8), (8, 1, 0, 16),
                                              (8, 1, 0, 8), (2, 0, 2, 16)])
@pytest.mark.parametrize("dtype", [C.F32, C.BF16])
def test_widths(monkeypatch, dtype, q, tight, spread, W):
    shape(monkeypatch, 0, q, tight, spread, W)
    widths = widths_for(dtype, 256)
    x, rows, n = batch(widths + [int(w) for w in widths[3:16]] * 3, q, dtype)
    y, info = run(x, rows, dtype, n)
    assert info["wide_items"] > 0 and info["huge_items"] == 0
    check(x, y, rows, dtype)


@pytest.mark.parametrize("P,spread", [(1, 0), (1, 4), (2, 0), (4, 3), (8, 0), (16, 0), (16, 8)])
def test_one_cluster_size(monkeypatch, P, spread):
    shape(monkeypatch, P, 1, 0, spread)
    for dtype in (C.F32, C.BF16):
        widths = widths_for(dtype, 8 * P)
        x, rows, n = batch(widths * 2, P, dtype, out_shift=3)
        y, info = run(x, rows, dtype, n + 5)
        assert info["cluster_size"] == P
        check(x, y, rows, dtype)


@pytest.mark.parametrize("q", [1, 16])
def test_many_rows_per_warp(monkeypatch, q):
    shape(monkeypatch, 0, q)
    rng = np.random.default_rng(q)
    widths = [int(2 ** rng.uniform(3, 13)) for _ in range(6000)] + [int(2 ** rng.uniform(14, 18)) for _ in range(300)]
    x, rows, n = batch(widths, 5, C.BF16)
    y, _ = run(x, rows, C.BF16, n)
    for i, o, w, op in rows[::17]:
        ref = U.reference(op, C.BF16, x[i:i + w].reshape(1, w))
        assert U.error_metric(op, C.BF16, U.to64(y[o:o + w].reshape(1, w)), ref) <= 1.0, (w, op)
    assert not torch.isnan(y.float()).any()


def test_infinities(monkeypatch):
    shape(monkeypatch, 0, 2)
    n = 40000
    x = torch.randn(3 * n)
    x[:n - 5] = -torch.inf        # most segments without a finite element
    x[n:2 * n] = -torch.inf       # none in the row: NaN
    x[2 * n + 7] = torch.inf      # NaN at the maximum
    y, _ = run(x, [(k * n, k * n, n, C.SOFTMAX) for k in range(3)], C.F32, 3 * n)
    ref = torch.softmax(x.view(3, n).double(), 1)
    assert torch.allclose(y[:n].double(), ref[0], rtol=1e-5, atol=0)
    assert torch.isnan(y[n:2 * n]).all() and torch.isnan(y[2 * n + 7])


def test_too_wide_is_refused(monkeypatch):
    shape(monkeypatch, 2, 1)
    n = 2 * WARPS * 2 * HALF * 4 + 64
    x = torch.zeros(n, device="cuda")
    with pytest.raises(C.CreditError):
        C.Ragged([(0, 0, n, C.SOFTMAX)], C.F32, x, x, tune=False)
