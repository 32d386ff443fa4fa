"""Batched power methods on both sides of the line between one block and one
cluster per tensor: tiny, small and mid sizes, few and many, matrices; vectors
beyond shared memory on a workspace that is only 8-byte aligned."""
import ctypes
import math

import numpy as np
import pytest
import torch

import oracle
import synth
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

tg = pytest.importorskip("paper_2501_03121_gb300")


def batch(shapes, sweeps, shift=0):
    items, host = [], []
    for b, dims in enumerate(shapes):
        A = (synth.tensor("u32", 8, dims, synth.stream_batch(b)) + np.float32(0.75)).astype(np.float32)
        x = [np.full(n, 1.0 / math.sqrt(n), dtype=np.float32) for n in dims]
        items.append(dict(A=gu.to_dev(A), x=[gu.to_dev(v) for v in x], lam=torch.zeros(1, dtype=torch.float64, device=gu.DEV),
                          status=torch.full((1,), -1, dtype=torch.int32, device=gu.DEV)))
        host.append((A, x))
    plan = tg.HOPMBatch(items, sweeps)
    if shift:
        plan._buffer = torch.empty(plan.workspace.numel() + 16, dtype=torch.uint8, device=gu.DEV)
        plan.workspace = plan._buffer[shift:shift + plan.workspace.numel()]
    plan.run()
    torch.cuda.synchronize()
    assert all(int(it["status"].item()) == 0 for it in items)
    for it, (A, x) in list(zip(items, host))[:12] + list(zip(items, host))[-4:]:
        ref = oracle.hopm(A, [v.astype(np.float64) for v in x], sweeps)
        assert abs(it["lam"].item() - ref["lam"]) <= 1e-5 * abs(ref["lam"])
        for got, want in zip(it["x"], ref["x"]):
            assert gu.rel_l2(got.cpu().numpy(), want) <= 1e-4  # the bounds of the single power method


TINY = [(3, 4, 5), (1, 1), (2, 3), (9, 8, 7, 6), (1, 130, 3), (65, 2, 33), (31, 33), (4, 4, 4, 4, 4), (3, 3, 3, 3, 3, 3)]


@pytest.mark.parametrize("shapes", [
    TINY * 30, [(127, 129), (2, 515)] * 3, [(24, 25, 26), (40, 40, 40), (16, 16, 16, 16)], [(41, 40, 41), (64, 33, 30)],
    [(64, 33, 30), (60, 61, 60)] * 32, [(100, 100), (99, 101)], [(130, 131)], [(96, 95, 94), (2, 2)], [(300, 401), (2, 2)]],
    ids=["tiny", "matrices", "small", "mid-few", "mid-many", "matrix-limit", "matrix-above", "large", "large-matrix"])
def test_against_oracle(shapes):
    batch(shapes, 3)


def test_vectors_in_memory_on_an_8_byte_boundary():
    batch([(3100, 3), (5, 3200), (3, 4, 5)], 2, shift=8)
