"""Few-output contractions (phases of rows within a block) and the adjoint
kernels at the edges of their tiles, against the oracle: one to many pieces of
outputs, rows around the phases, splits and shared-memory chunks of x, rows
off 16-byte boundaries, partial pieces; gx with chunks of rows and elements
outside the exact FP64 window; gA in 16-byte pieces that cross rows and slabs."""
import math

import numpy as np
import pytest
import torch

import oracle
import synth
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

tg = pytest.importorskip("paper_2501_03121_gb300")

CODES = [tg.F64, tg.F32, tg.BF16, tg.E4M3, tg.F16]
IDS = ["f64", "f32", "bf16", "e4m3", "f16"]
FEW = [(4096, 32), (4100, 33), (9001, 64), (20000, 2), (5000, 7), (4097, 31), (3, 4099, 40), (70000, 35), (30011, 5)]
SMALL = [(128, 128), (8, 32), (9, 33), (17, 100), (300, 7, 33), (5, 64, 130), (1023, 50), (1025, 47), (60, 2049)]


def placed(A, shift):
    flat = gu.to_dev(A).reshape(-1)
    buf = torch.zeros(flat.numel() + 32, dtype=flat.dtype, device=gu.DEV)
    buf[shift:shift + flat.numel()] = flat
    return buf[shift:shift + flat.numel()]


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("code", CODES, ids=IDS)
@pytest.mark.parametrize("dims", FEW + SMALL, ids=lambda d: "x".join(map(str, d)))
def test_contraction(dims, code, shift):
    A, Ao, scales = gu.inputs(dims, code)
    k = len(dims) - 2
    x = gu.vec(code, dims[k], synth.stream_x(k))
    st = None if scales is None else gu.to_dev(scales)
    y0 = gu.vec(code, math.prod(dims) // dims[k], 99)
    y = gu.to_dev(y0).clone()
    tg.tvc(placed(A, shift), k, gu.to_dev(x), y=y, scales=st, alpha=-1.5, beta=0.5, shape=dims)
    ref = -1.5 * oracle.tvc(Ao, k, x, scales=scales).ravel() + 0.5 * y0.astype(np.float64)
    assert gu.rel_l2(y.cpu().numpy(), ref) <= gu.TOL[code]


@pytest.mark.parametrize("dims", [(5000, 40), (200, 64)])
def test_contraction_single_double_and_window(dims):
    A = synth.tensor("u64", 3, dims)
    A[::5, 3] = 0.0
    A[7, 9] = 2.0 ** -200
    A[11, 2] = 2.0 ** 65
    x = synth.vector("u64", 4, 1, dims[0])
    x[13] = 2.0 ** -40
    got = tg.tvc(gu.to_dev(A), 0, gu.to_dev(x)).cpu().numpy()
    assert gu.rel_l2(got, oracle.tvc(A, 0, x)) <= 1e-12
    F = synth.tensor("u32", 3, dims).astype(np.float32)
    got = tg.tvc(gu.to_dev(F), 0, gu.to_dev(x)).cpu().numpy()
    assert gu.rel_l2(got, oracle.tvc(F, 0, x)) <= 1e-12


GRADS = [((5, 300, 33), 1), ((257, 9), 0), ((2, 255, 70), 1), ((700, 3, 5), 1), ((40, 17, 31), 1), ((3, 513, 64), 1),
         ((6000, 7), 1), ((31, 5, 128), 1), ((900,), 0), ((12, 8, 2), 2), ((4, 1000, 1, 2), 1)]


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("code", CODES, ids=IDS)
@pytest.mark.parametrize("dims,k", GRADS, ids=lambda d: "x".join(map(str, d)) if isinstance(d, tuple) else None)
def test_adjoints(dims, k, code, shift):
    A, Ao, scales = gu.inputs(dims, code)
    N, n = math.prod(dims), dims[k]
    x = gu.vec(code, n, synth.stream_x(k))
    gy = gu.vec(code, N // n, 77)
    st = None if scales is None else gu.to_dev(scales)
    buf = torch.full((N + 4,), float("nan"), dtype=gu.to_dev(x).dtype, device=gu.DEV)
    gA = buf[shift:shift + N]
    gx, _ = tg.tvc_backward(placed(A, shift), k, gu.to_dev(x), gu.to_dev(gy), scales=st, gA=gA, shape=dims, code=code)
    tol = gu.TOL[code]
    assert gu.rel_l2(gx.cpu().numpy(), oracle.tvc_grad_x(Ao, k, gy, scales=scales)) <= tol
    want = oracle.tvc_grad_A(dims, k, x, gy).ravel()
    assert gu.rel_l2(gA.cpu().numpy(), want) <= tol
    assert torch.isnan(buf[:shift]).all() and torch.isnan(buf[shift + N:]).all()
    tg.tvc_backward(None, k, gu.to_dev(x), gu.to_dev(gy), need_x=False, gA=gA, beta_A=0.5, shape=dims, code=code)
    assert gu.rel_l2(gA.cpu().numpy(), 1.5 * want) <= tol


@pytest.mark.parametrize("dims,k", [((40, 21, 64), 1), ((40, 21, 33), 1)])
def test_grad_x_outside_the_window(dims, k):
    A = synth.tensor("u64", 3, dims)
    A[::7, 2] = 0.0
    A[3, 4, 5] = 2.0 ** -200
    A[8, 9, 10] = 2.0 ** 66
    gy = synth.vector("u64", 4, 1, math.prod(dims) // dims[k])
    gy[17] = 0.0
    gy[33] = 2.0 ** -50
    gx, _ = tg.tvc_backward(gu.to_dev(A), k, None, gu.to_dev(gy), need_A=False)
    assert gu.rel_l2(gx.cpu().numpy(), oracle.tvc_grad_x(A, k, gy)) <= 1e-12
