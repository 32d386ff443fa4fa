"""gx with FP64 arithmetic (FP64 and single-double storage): its error, and
elements and entries of gy outside the exact window of the products."""
import math

import numpy as np
import pytest
import torch

import synth
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

tg = pytest.importorskip("paper_2501_03121_gb300")

CODES = [tg.F64, tg.F32D]
IDS = ["f64", "f32d"]
# (dims, mode): rows on and off 16-byte boundaries, one and several pieces per thread, rows around the chunks of 128
CASES = [((480, 161), 0), ((106, 117), 0), ((7, 65), 0), ((1, 3, 64), 1), ((2, 8, 3, 9), 2), ((27, 57), 0), ((9, 129, 64), 1),
         ((300, 128, 33), 1), ((40, 21, 6000), 1), ((5, 7, 40000), 1), ((3, 300, 31), 1), ((900,), 0), ((129, 2), 0)]


def terms(A, k, gy):
    u, v = math.prod(A.shape[:k]), math.prod(A.shape[k + 1:])
    return A.reshape(u, -1, v).astype(np.longdouble) * gy.reshape(u, 1, v).astype(np.longdouble)


def gx_of(A, k, gy, code):
    return tg.tvc_backward(gu.to_dev(A), k, None, gu.to_dev(gy), need_A=False, code=code)[0].cpu().numpy()


def inputs(dims, k, code):
    A = synth.tensor("u64" if code == tg.F64 else "u32", 3, dims)
    return A, synth.vector("u64", 4, 1, math.prod(dims) // dims[k])


@pytest.mark.parametrize("code", CODES, ids=IDS)
@pytest.mark.parametrize("dims,k", CASES, ids=lambda d: "x".join(map(str, d)) if isinstance(d, tuple) else None)
def test_error(dims, k, code):
    # A thread's pair of at most 8 products is off by a few units of 2^-49 of
    # their root sum of squares, independently of other threads; FP64 sums
    # join them.  4 units bound the norm over all entries.
    A, gy = inputs(dims, k, code)
    t = terms(A, k, gy)
    err = gx_of(A, k, gy, code) - t.sum((0, 2))
    assert np.sqrt((err**2).sum()) <= 4 * 2.0**-49 * np.sqrt((t**2).sum())


@pytest.mark.parametrize("kind", ["zeros", "tiny gy", "tiny A", "mixed"])
@pytest.mark.parametrize("code", CODES, ids=IDS)
@pytest.mark.parametrize("dims,k", [((40, 21, 640), 1), ((40, 21, 33), 1), ((300, 70), 0)])
def test_outside_the_window(dims, k, code, kind):
    A, gy = inputs(dims, k, code)
    rng = np.random.default_rng(1)
    if kind == "zeros":
        A[rng.random(dims) < 0.3] = 0.0
        gy[rng.random(gy.shape) < 0.3] = 0.0
    if kind == "tiny gy":
        gy *= 2.0**-200
    if kind == "tiny A":
        A *= A.dtype.type(2.0**-80)
    if kind == "mixed":
        A[rng.random(dims) < 0.1] *= A.dtype.type(2.0**-90)
        A.reshape(-1)[17] = 2.0**70
        gy *= np.exp2(rng.integers(-60, 60, gy.shape).astype(np.float64))
    t = terms(A, k, gy)
    err = gx_of(A, k, gy, code) - t.sum((0, 2))
    assert np.sqrt((err**2).sum()) <= 4 * 2.0**-49 * np.sqrt((t**2).sum())


@pytest.mark.parametrize("code", CODES, ids=IDS)
def test_infinite_entries(code):
    A, gy = inputs((6, 5, 40), 1, code)
    A[3, 2, 7] = 0.0
    gy = gy.reshape(6, 40)
    gy[3, 7] = np.inf
    with np.errstate(invalid="ignore"):
        want = np.einsum("ijl,il->j", A.astype(np.float64), gy)
    got = gx_of(A, 1, gy, code)
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.isnan(got[2])  # 0 * Inf
    assert np.array_equal(np.isinf(got), np.isinf(want)) and np.array_equal(np.sign(got[:2]), np.sign(want[:2]))
