"""An infinite element gives the infinities that plain addition gives, in every
output that meets it and in no other, whichever kernel a shape takes: sums
held as compensated pairs, splits, phases, rows off 16-byte boundaries."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu

tg = pytest.importorskip("paper_2501_03121_gb300")

DTYPES = [torch.float64, torch.float32, torch.bfloat16, torch.float16]
INF = float("inf")
# (dims, mode): rows and columns at both alignments, few outputs, slabs, a single row
CASES = [((50, 63), 1), ((5000, 63), 1), ((300, 128), 1), ((4, 20001), 1), ((4096, 32), 0), ((4100, 33), 0), ((20000, 2), 0),
         ((5, 64, 130), 1), ((60, 2049), 0), ((40, 41, 200), 1), ((3000, 50, 3), 1), ((500, 19, 16), 1), ((70, 1000, 65), 1)]


def tensor(dims, dt, seed=0):
    """Positive entries, one +Inf; and the index of the Inf as (i, j, l) of mode k's view."""
    g = torch.Generator().manual_seed(seed)
    A = (torch.rand(dims, generator=g, dtype=torch.float64) + 0.5).to(dt).cuda()
    at = A.numel() // 3
    A.view(-1)[at] = INF
    return A, at


def where(dims, k, at):
    v, nk = math.prod(dims[k + 1:]), dims[k]
    return at // (nk * v), at // v % nk, at % v


def vec(n, dt):
    return torch.ones(n, dtype=torch.float64 if dt == torch.float64 else torch.float32, device="cuda")


@pytest.mark.parametrize("dt", DTYPES, ids=str)
@pytest.mark.parametrize("dims,k", CASES, ids=lambda d: "x".join(map(str, d)) if isinstance(d, tuple) else None)
def test_contraction_and_adjoint(dims, k, dt):
    A, at = tensor(dims, dt)
    i, j, l = where(dims, k, at)
    v = math.prod(dims[k + 1:])
    y = tg.tvc(A, k, vec(dims[k], dt)).view(-1)
    assert y[i * v + l] == INF and int(torch.isfinite(y).sum()) == y.numel() - 1
    gy = vec(y.numel(), dt)
    gx, _ = tg.tvc_backward(A, k, None, gy, need_A=False)
    assert gx[j] == INF and int(torch.isfinite(gx).sum()) == dims[k] - 1
    gy.neg_()
    gx, _ = tg.tvc_backward(A, k, None, gy, need_A=False)
    assert gx[j] == -INF
    A.view(-1)[at - at % v + (l + 1) % v if v > 1 else at - at % dims[k] + (j + 1) % dims[k]] = -INF
    if v == 1:  # both infinities in one row
        assert math.isnan(tg.tvc(A, k, vec(dims[k], dt)).view(-1)[i])


@pytest.mark.parametrize("R", [3, 8, 13, 33])
@pytest.mark.parametrize("dt", DTYPES, ids=str)
@pytest.mark.parametrize("dims,k", CASES, ids=lambda d: "x".join(map(str, d)) if isinstance(d, tuple) else None)
def test_tensor_matrix(dims, k, dt, R):
    A, at = tensor(dims, dt)
    i, j, l = where(dims, k, at)
    X = vec(R * dims[k], dt).view(R, dims[k])
    X[1::2] = -1.0
    Y = tg.tmc(A, k, X).view(-1, R, math.prod(dims[k + 1:]))
    assert torch.equal(Y[i, :, l], torch.tensor([INF, -INF], dtype=Y.dtype, device="cuda").repeat(R)[:R])
    assert int(torch.isfinite(Y).sum()) == Y.numel() - R


@pytest.mark.parametrize("R", [2, 16])
@pytest.mark.parametrize("dt", DTYPES, ids=str)
def test_mttkrp(dt, R):
    dims = (20, 30, 40)
    A, at = tensor(dims, dt)
    F = [vec(n * R, dt).view(n, R) for n in dims]
    for k in range(3):
        M = tg.mttkrp(A, k, F)
        row = where(dims, k, at)[1]
        assert bool((M[row] == INF).all()) and int(torch.isfinite(M).sum()) == M.numel() - R


@pytest.mark.parametrize("dims,k", [((3, 7, 32), 1), ((2, 513, 34), 1), ((40, 31, 50, 9), 2), ((700, 31), 1), ((2049, 64), 1),
                                    ((300, 257), 1), ((17, 1025), 0)])
def test_batch(dims, k):
    A, at = tensor(dims, torch.float32)
    i, j, l = where(dims, k, at)
    v, n = math.prod(dims[k + 1:]), dims[k]
    x, gy = vec(n, torch.float32), vec(A.numel() // n, torch.float32)
    y, gx, gA = torch.zeros_like(gy), torch.zeros_like(x), torch.zeros_like(A)
    tg.TVCBatch([dict(A=A, mode=k, x=x, y=y, gy=gy, gx=gx, gA=gA)]).run()
    torch.cuda.synchronize()
    assert y[i * v + l] == INF and int(torch.isfinite(y).sum()) == y.numel() - 1
    assert gx[j] == INF and int(torch.isfinite(gx).sum()) == n - 1
    assert bool((gA == 1).all())


def test_sums_beyond_binary32():
    A = torch.full((64, 100, 40), 3e38, device="cuda")
    for k in range(3):
        x = torch.ones(A.shape[k], device="cuda")
        assert bool((tg.tvc(A, k, x) == INF).all())
        assert bool((tg.tmc(A, k, torch.stack([x, -x])) == torch.tensor([INF, -INF], device="cuda").view(
            [2 if i == k else 1 for i in range(3)])).all())
