"""A batch holds on to the tensors whose addresses its descriptors carry, as
long as it can run (host side; the constructors take CPU tensors too)."""
import gc
import weakref

import torch

import paper_2501_03121_gb300 as tg


def test_power_method_batch_keeps_its_tensors():
    xs = [torch.ones(n) for n in (3, 4, 5)]
    item = dict(A=torch.ones(3, 4, 5), x=xs, lam=torch.zeros(1, dtype=torch.float64))
    refs = [weakref.ref(t) for t in (item["A"], item["lam"], *xs)]
    batch = tg.HOPMBatch([item], 2)
    xs.clear()
    del item, xs
    gc.collect()
    assert all(r() is not None for r in refs)
    del batch
    gc.collect()
    assert all(r() is None for r in refs)


def test_contraction_batch_keeps_its_tensors():
    A = torch.ones(3, 4)
    ref = weakref.ref(A)
    batch = tg.TVCBatch([dict(A=A, mode=0, x=torch.ones(3), y=torch.zeros(4))])
    del A
    gc.collect()
    assert ref() is not None and batch.count == 1
