"""The one-launch power method at the edges of its partition, against the
oracle: odd trailing sizes (rows off 16-byte boundaries, partial pieces),
modes of size one, fewer outputs than blocks, leading modes with many blocks
per entry, modes longer than a block's threads, contracted modes beyond 64
rows per thread, slab scales, elements outside the exact FP64 window, tensors
off 16-byte boundaries, the stopping rule, failures, and graph capture."""
import math

import numpy as np
import pytest
import torch

import oracle
import synth
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

tg = pytest.importorskip("paper_2501_03121_gb300")

SHAPES = [(2, 3, 64), (1, 1, 70), (5, 1, 65), (1, 40, 1, 67), (3, 4, 5, 6, 16), (13, 44, 25, 6), (700, 9, 33), (9, 700, 65),
          (4, 3, 2100), (2, 2, 2, 2, 2, 2, 64), (130, 17, 31), (40, 41, 131), (2, 1500, 70)]
CODES = [tg.F64, tg.F32, tg.BF16, tg.E4M3, tg.F16]
IDS = ["f64", "f32", "bf16", "e4m3", "f16"]


def starts(dims, dt):
    return [np.full(n, 1.0 / math.sqrt(n)).astype(dt) for n in dims]


def tensor(dims, code):
    """A tensor with a dominant rank-1 part, so that the iteration contracts."""
    if code == tg.F64:
        A = synth.tensor("u64", 2, dims) + 0.75
        return A, A, None
    src = synth.tensor("u32", 2, dims) + np.float32(0.75)
    if code == tg.F32:
        return src, src, None
    codes, scales = oracle.quantise(src, code)
    return codes, codes, scales


def placed(A, shift):
    flat = gu.to_dev(A).reshape(-1)
    buf = torch.zeros(flat.numel() + 32, dtype=flat.dtype, device=gu.DEV)
    buf[shift:shift + flat.numel()] = flat
    return buf[shift:shift + flat.numel()]


def compare(A, Ao, scales, dims, code, sweeps, shift=0, x=None):
    x = x or starts(dims, np.float64 if code == tg.F64 else np.float32)
    ref = oracle.hopm(Ao, [v.astype(np.float64) for v in x], sweeps, scales=scales)
    r = tg.hopm(placed(A, shift), [gu.to_dev(v) for v in x], sweeps, shape=dims,
                scales=None if scales is None else gu.to_dev(scales)).check()
    tol = gu.TOL[code]
    assert int(r.sweeps.item()) == sweeps
    assert abs(r.lam.item() - ref["lam"]) <= tol * abs(ref["lam"])
    for got, want in zip(r.x, ref["x"]):
        assert gu.rel_l2(got.cpu().numpy(), want) <= 10 * tol


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("code", CODES, ids=IDS)
@pytest.mark.parametrize("dims", SHAPES, ids=lambda d: "x".join(map(str, d)))
def test_against_oracle(dims, code, shift):
    compare(*tensor(dims, code), dims, code, 4, shift)


@pytest.mark.parametrize("dims", [(20, 30, 64), (20, 30, 33)])
def test_fp64_elements_outside_the_window(dims):
    A = synth.tensor("u64", 2, dims) + 0.75
    A[::3, 1] = 0.0
    A[2, 3, 4] = 2.0 ** -300
    A[5, 7, 9] = 2.0 ** 70
    compare(A, A, None, dims, tg.F64, 3)


def test_single_double():
    dims = (30, 21, 50)
    A = (synth.tensor("u32", 2, dims) + np.float32(0.75)).astype(np.float32)
    x = starts(dims, np.float64)
    ref = oracle.hopm(A, x, 4)
    r = tg.hopm(gu.to_dev(A), [gu.to_dev(v) for v in x], 4).check()
    assert abs(r.lam.item() - ref["lam"]) <= 1e-12 * ref["lam"]


def test_stopping_rule_and_failures():
    dims = (12, 13, 64)
    A = gu.to_dev(synth.tensor("u64", 2, dims) + 0.75)
    x = [gu.to_dev(v) for v in starts(dims, np.float64)]
    full = tg.hopm(A, x, 30).check()
    r = tg.hopm(A, x, 30, 1e-6).check()
    t = int(r.sweeps.item())
    hist = full.lam_hist.cpu().numpy()
    want = next(i + 1 for i in range(1, 30) if abs(hist[i] - hist[i - 1]) <= 1e-6 * hist[i])
    assert t == want and r.lam.item() == hist[t - 1]
    z = tg.hopm(torch.zeros(dims, dtype=torch.float64, device=gu.DEV), x, 3)
    torch.cuda.synchronize()
    assert int(z.status.item()) != 0 and int(z.sweeps.item()) == 0
    assert all(torch.equal(a, b) for a, b in zip(z.x, x))
    A[3, 4, 5] = float("nan")
    n = tg.hopm(A, x, 3)
    torch.cuda.synchronize()
    assert int(n.status.item()) not in (0, int(z.status.item()))


def test_graph_replay_and_streams():
    dims = (40, 41, 128)
    A = gu.to_dev(synth.tensor("u32", 2, dims) + np.float32(0.75))
    x = [gu.to_dev(v) for v in starts(dims, np.float32)]
    ws = torch.empty(tg.hopm_workspace_size(dims, tg.F32), dtype=torch.uint8, device=gu.DEV)
    ref = tg.hopm(A, x, 5, workspace=ws).check()
    xg = [v.clone() for v in x]
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        with torch.cuda.graph(g, stream=s):
            r = tg.hopm(A, xg, 5, workspace=ws, inplace=True, stream=s)
    torch.cuda.current_stream().wait_stream(s)
    for _ in range(2):
        for a, b in zip(xg, x):
            a.copy_(b)
        g.replay()
        torch.cuda.synchronize()
        assert r.lam.item() == ref.lam.item()
        assert all(torch.equal(a, b) for a, b in zip(xg, ref.x))
    # two runs at once, each on its own stream and workspace
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    out = []
    for st in streams:
        with torch.cuda.stream(st):
            out.append(tg.hopm(A, x, 20, stream=st))
    torch.cuda.synchronize()
    one = tg.hopm(A, x, 20).check()
    assert all(o.lam.item() == one.lam.item() for o in out)
