"""Contractions whose rows start off 16-byte boundaries, against the oracle:
column pieces cut at every offset (row lengths 33 and up, tensors shifted by
elements), partial last pieces, row counts around the rows in flight and the
fold, split n_k; rows of every lane count from 16 bytes up; neighbours that
are NaN must not leak into a row or column."""
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
COLS = [(3, 5, 33), (2, 6, 34), (2, 7, 35), (4, 12, 37), (1, 70, 47), (9, 64, 49), (2, 131, 63), (1, 999, 65), (7, 1, 101),
        (1, 4, 4099)]
ROWS = [(9, 5), (50, 11), (33, 13), (70, 16 + 3), (31, 33), (40, 63), (129, 75), (64, 100), (11, 175), (10, 250), (6, 501),
        (5, 979), (1, 4095), (3, 20001), (700, 47)]


def shifted(A, shift):
    """The tensor on the GPU, `shift` elements past a 16-byte boundary."""
    flat = gu.to_dev(A).reshape(-1)
    buf = torch.zeros(flat.numel() + 32, dtype=flat.dtype, device=gu.DEV)
    buf[shift:shift + flat.numel()] = flat
    return buf[shift:shift + flat.numel()]


@pytest.mark.parametrize("shift", [0, 1, 3])
@pytest.mark.parametrize("code", CODES, ids=IDS)
@pytest.mark.parametrize("dims", COLS + ROWS, ids=lambda d: "x".join(map(str, d)))
def test_against_oracle(dims, code, shift):
    A, Ao, scales = gu.inputs(dims, code)
    k = len(dims) - 2 if dims in COLS else len(dims) - 1
    x = gu.vec(code, dims[k], synth.stream_x(k))
    ref = oracle.tvc(Ao, k, x, scales=scales)
    st = None if scales is None else gu.to_dev(scales)
    got = tg.tvc(shifted(A, shift), k, gu.to_dev(x), scales=st, shape=dims).cpu().numpy()
    assert gu.rel_l2(got, ref) <= 1e-5  # the parity bound of FP32 accumulation


@pytest.mark.parametrize("dims,k", [((6, 9, 37), 1), ((12, 43), 1), ((8, 333), 1)])
def test_nan_neighbours_stay_out(dims, k):
    rng = np.random.default_rng(3)
    A = rng.uniform(-1, 1, size=dims).astype(np.float32)
    A[3] = np.nan  # the slab or row between its neighbours
    if k == 1 and len(dims) == 3:
        A[1, :, 5] = np.nan  # one column
    x = rng.uniform(-1, 1, size=dims[k]).astype(np.float32)
    got = tg.tvc(gu.to_dev(A), k, gu.to_dev(x)).cpu().numpy()
    ref = np.tensordot(A.astype(np.float64), x.astype(np.float64), axes=(k, 0))
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    ok = ~np.isnan(ref)
    assert gu.rel_l2(got[ok], ref[ok]) <= 1e-5
