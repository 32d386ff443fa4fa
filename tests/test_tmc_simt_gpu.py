"""Register-blocked tensor-matrix contraction at the edges of its tiles,
against the oracle: every count of rows of X around the passes, columns and
rows at every alignment and remainder of the four-element windows, n_k around
the stages, the folds and the splits, slab scales, alpha and beta."""
import math

import numpy as np
import pytest
import torch

import oracle
import synth
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

tg = pytest.importorskip("paper_2501_03121_gb300")

CODES = [tg.F32, tg.BF16, tg.E4M3, tg.F16]
IDS = ["f32", "bf16", "e4m3", "f16"]
# (dims, mode): columns (v > 1), then rows (v == 1)
CASES = [((3, 5, 4), 1), ((2, 64, 5), 1), ((4, 65, 7), 1), ((300, 33), 0), ((1100, 6), 0), ((2, 63, 130), 1), ((5, 129, 9), 1),
         ((7, 4), 1), ((70, 5), 1), ((33, 63), 1), ((129, 129), 1), ((9, 513), 1), ((130, 1030), 1), ((2, 3, 127), 2),
         ((5, 4001), 1)]


def placed(A, shift):
    flat = gu.to_dev(A).reshape(-1)
    buf = torch.zeros(flat.numel() + 32, dtype=flat.dtype, device=gu.DEV)
    buf[shift:shift + flat.numel()] = flat
    return buf[shift:shift + flat.numel()]


def check(dims, k, code, R, shift, alpha=1.0, beta=0.0):
    A, Ao, scales = gu.inputs(dims, code)
    X = synth.tensor("u32", 4, (R, dims[k])).astype(np.float32)
    out = tuple(R if i == k else n for i, n in enumerate(dims))
    Y = synth.tensor("u32", 5, out).astype(np.float32)
    st = None if scales is None else gu.to_dev(scales)
    got = tg.tmc(placed(A, shift), k, gu.to_dev(X), Y=gu.to_dev(Y), scales=st, alpha=alpha, beta=beta, shape=dims)
    ref = alpha * oracle.tmc(Ao, k, X.astype(np.float64), scales=scales) + beta * Y.astype(np.float64)
    assert gu.rel_l2(got.cpu().numpy(), ref) <= 1e-5  # the parity bound of the TMC tests


@pytest.mark.parametrize("shift", [0, 1, 3])
@pytest.mark.parametrize("code", CODES, ids=IDS)
@pytest.mark.parametrize("dims,k", CASES, ids=lambda d: "x".join(map(str, d)) if isinstance(d, tuple) else None)
def test_windows(dims, k, code, shift):
    check(dims, k, code, 13, shift)


@pytest.mark.parametrize("R", [1, 3, 4, 5, 8, 9, 12, 13, 16, 17, 24, 25, 31, 32, 33, 40, 65])
@pytest.mark.parametrize("dims,k", [((6, 70, 35), 1), ((70, 131), 1)], ids=["cols", "rows"])
def test_rows_of_x(dims, k, R):
    check(dims, k, tg.F32, R, 1, alpha=-0.5, beta=2.0)
    check(dims, k, tg.BF16, R, 0)
