"""Cluster kernel of the batched power method at the shapes where its tiling
can go wrong, against the oracle: column counts around the block's chunks and
the cluster's split (fewer columns than blocks, odd counts, whole 8- and
16-byte pieces), row counts around the rows in flight and beyond one
reduction range, trailing modes of size one, order 2 and high order, vectors
too long for shared memory, tensors that start off a 16-byte boundary, and
batches that select every cluster width."""
import math

import numpy as np
import pytest
import torch

import oracle
import synth
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

tg = pytest.importorskip("paper_2501_03121_gb300")

SHAPES = [(2, 2), (1, 5), (33, 1), (7, 3, 1), (3, 1, 1, 4), (17, 9), (15, 31, 33), (16, 32, 32), (9, 64, 130),
          (8, 63, 129), (5, 257, 66), (1100, 6), (600, 3, 5), (2, 3001, 4), (4, 3, 2500), (31, 2, 3, 5, 7),
          (3, 2, 2, 2, 2, 2, 3), (40, 1, 513), (128, 20, 51)]


def run(shapes, sweeps, shift=0):
    items, host = [], []
    for b, dims in enumerate(shapes):
        N = math.prod(dims)
        A = synth.tensor("u32", 3, dims, synth.stream_batch(b)) + np.float32(0.5)  # a dominant rank-1 part
        buf = torch.zeros(N + 4, dtype=torch.float32, device=gu.DEV)
        buf[shift:shift + N] = gu.to_dev(A).reshape(-1)
        xs = [torch.full((n,), 1.0 / math.sqrt(n), dtype=torch.float32, device=gu.DEV) for n in dims]
        items.append(dict(A=buf[shift:shift + N], shape=dims, x=xs,
                          lam=torch.zeros(1, dtype=torch.float64, device=gu.DEV),
                          status=torch.full((1,), -1, dtype=torch.int32, device=gu.DEV)))
        host.append(A)
    tg.HOPMBatch(items, sweeps).run()
    torch.cuda.synchronize()
    for it, A, dims in zip(items, host, shapes):
        ref = oracle.hopm(A, [np.ones(n) / math.sqrt(n) for n in dims], sweeps)
        assert int(it["status"].item()) == ref["status"] == 0, dims
        # FP32 storage and products: the parity bound of the FP32 kernels
        assert abs(it["lam"].item() - ref["lam"]) <= 1e-5 * ref["lam"], dims
        for xg, xr in zip(it["x"], ref["x"]):
            assert gu.rel_l2(xg.cpu().numpy(), xr) <= 1e-5, dims


@pytest.mark.parametrize("shift", [0, 1, 2])
def test_shapes_and_alignments(shift):
    run(SHAPES, 4, shift)


@pytest.mark.parametrize("count", [1, 24, 60, 120, 400])
def test_every_cluster_width(count):
    # equal tensors: the batch alone decides the blocks per cluster (16, 16, 8, 4, 2)
    run([(6, 40, 21)] * count, 3)


def test_stops_on_zero_norm():
    x = [torch.full((n,), 1.0, dtype=torch.float32, device=gu.DEV) for n in (4, 5, 6)]
    keep = [v.clone() for v in x]
    it = dict(A=torch.zeros(4, 5, 6, dtype=torch.float32, device=gu.DEV), x=x,
              lam=torch.ones(1, dtype=torch.float64, device=gu.DEV),
              status=torch.zeros(1, dtype=torch.int32, device=gu.DEV))
    tg.HOPMBatch([it], 3).run()
    torch.cuda.synchronize()
    assert int(it["status"].item()) != 0 and it["lam"].item() == 0.0
    assert all(torch.equal(a, b) for a, b in zip(x, keep))
