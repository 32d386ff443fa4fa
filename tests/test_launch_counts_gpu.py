"""How many kernels a call launches, where the route promises one: phases of rows
(few outputs unsplit, small tensors), the power method of small tensors, the
batches; and the queued power method beyond its line."""
import pytest
import torch

pytestmark = pytest.mark.gpu

tg = pytest.importorskip("paper_2501_03121_gb300")


def launches(f):
    before = tg.kernel_launches()
    f()
    torch.cuda.synchronize()
    return tg.kernel_launches() - before


@pytest.mark.parametrize("dt,dims,mode,count", [
    (torch.float32, (128, 128, 128), 0, 1), (torch.bfloat16, (128, 128, 128), 1, 1), (torch.float8_e4m3fn, (128, 128, 128), 0, 1),
    (torch.float64, (70, 128, 128), 1, 1),
    (torch.float64, (128, 128, 128), 0, 3),   # x split, columns, reduction
    (torch.float32, (1000000, 64), 0, 2)])    # phases over one wave, reduction
def test_contraction(dt, dims, mode, count):
    vt = torch.float64 if dt == torch.float64 else torch.float32
    A, x = torch.zeros(dims, dtype=dt, device="cuda"), torch.zeros(dims[mode], dtype=vt, device="cuda")
    assert launches(lambda: tg.tvc(A, mode, x)) == count


@pytest.mark.parametrize("dt,dims,one", [
    (torch.float64, (128, 128, 128), True), (torch.float32, (20, 30, 64), True), (torch.bfloat16, (130, 17, 62), True),
    (torch.float8_e4m3fn, (130, 17, 64), True), (torch.float16, (9, 700, 65), True),
    (torch.float16, (130, 17, 31), False),          # rows of less than four pieces
    (torch.float32, (4, 20, 948, 502), False),      # W_1 of 38 MB
    (torch.float32, (300, 300, 300), False)])       # beyond 104 MB
def test_power_method(dt, dims, one):
    vt = torch.float64 if dt == torch.float64 else torch.float32
    A = torch.ones(dims, device="cuda").to(dt)
    xs = [torch.full((n,), n**-0.5, dtype=vt, device="cuda") for n in dims]
    got = launches(lambda: tg.hopm(A, xs, 2).check())
    assert (got == 1) if one else (got > 2 * len(dims))


def test_batches():
    A = torch.ones(20, 30, 40, device="cuda")
    xs = [torch.ones(n, device="cuda") for n in A.shape]
    contraction = tg.TVCBatch([dict(A=A, mode=1, x=xs[1], y=torch.empty(800, device="cuda"))] * 3)
    assert launches(contraction.run) == 1
    assert launches(tg.HOPMBatch([dict(A=A, x=xs)], 2).run) == 1
