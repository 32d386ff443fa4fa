"""Fused items of the batched contractions (y, gx and gA from one read of A)
at the edges of their tiles, against the oracle: columns of every load width
(16-, 8- and 4-byte pieces, tensors off 16-byte boundaries), row counts around
the rows in flight and the fusion limit, rows of v == 1 around the chunk and
length limits, and every subset of the wanted results."""
import itertools
import math

import numpy as np
import pytest
import torch

import oracle
import synth
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

tg = pytest.importorskip("paper_2501_03121_gb300")

SPEC = [((3, 7, 32), 1), ((3, 8, 33), 1), ((2, 9, 130), 1), ((5, 16, 64), 1), ((17, 1025), 0), ((4, 511, 36), 1),
        ((2, 512, 35), 1), ((2, 513, 34), 1), ((1, 1, 40), 1), ((40, 31, 50, 9), 2), ((70, 12, 11), 1),  # v >= 32, v < 32
        ((700, 31), 1), ((700, 32), 1), ((260, 33), 1), ((2049, 64), 1), ((300, 255), 1), ((300, 256), 1),
        ((300, 257), 1), ((3, 5, 100), 2), ((5000, 8), 1), ((333, 17), 1), ((50, 1000), 1)]  # v == 1


def run(spec, wanted, shift):
    items, host = [], []
    for b, (dims, mode) in enumerate(spec):
        N, n = math.prod(dims), dims[mode]
        A = synth.tensor("u32", 5, dims, synth.stream_batch(b))
        x = synth.vector("u32", 6, synth.stream_batch(b), n)
        gy = synth.vector("u32", 7, synth.stream_batch(b), N // n)
        bufs = {}
        for k, size in (("A", N), ("gA", N)):
            t = torch.full((N + 4,), float("nan"), dtype=torch.float32, device=gu.DEV)
            bufs[k] = t[shift:shift + size]
        bufs["A"].copy_(gu.to_dev(A).reshape(-1))
        it = dict(A=bufs["A"], shape=dims, mode=mode, x=gu.to_dev(x), gy=gu.to_dev(gy))
        if "y" in wanted:
            it["y"] = torch.full((N // n,), float("nan"), dtype=torch.float32, device=gu.DEV)
        if "gx" in wanted:
            it["gx"] = torch.full((n,), float("nan"), dtype=torch.float32, device=gu.DEV)
        if "gA" in wanted:
            it["gA"] = bufs["gA"]
        items.append(it)
        host.append((A, x, gy))
    batch = tg.TVCBatch(items)
    for _ in range(2):  # the second run finds the counters reset
        batch.run()
    torch.cuda.synchronize()
    for it, (A, x, gy), (dims, mode) in zip(items, host, spec):
        # the parity bounds of the FP32 kernels
        if "y" in wanted:
            assert gu.rel_l2(it["y"].cpu().numpy(), oracle.tvc(A, mode, x)) <= 1e-5, dims
        if "gx" in wanted:
            assert gu.rel_l2(it["gx"].cpu().numpy(), oracle.tvc_grad_x(A, mode, gy)) <= 1e-5, dims
        if "gA" in wanted:
            assert gu.rel_l2(it["gA"].cpu().numpy(), oracle.tvc_grad_A(dims, mode, x, gy)) <= 1e-6, dims


@pytest.mark.parametrize("shift", [0, 1, 2])
def test_all_results_every_alignment(shift):
    run(SPEC, ("y", "gx", "gA"), shift)


@pytest.mark.parametrize("wanted", [w for r in (1, 2) for w in itertools.combinations(("y", "gx", "gA"), r)])
def test_subsets(wanted):
    run(SPEC, wanted, 0)
