"""FP32 sums that meet one large term early: the small terms behind it are kept
by compensated pairs and lost by plain running sums.  Terms of 1 beside 2^25
(spacing 4) or 2^31 (spacing 256) vanish one by one."""
import pytest
import torch

pytestmark = pytest.mark.gpu

tg = pytest.importorskip("paper_2501_03121_gb300")


def batch_gx(dims, mode, at, big):
    A = torch.ones(dims, device="cuda")
    A.view(-1)[at] = big
    gy = torch.ones(A.numel() // dims[mode], device="cuda")
    x = torch.ones(dims[mode], device="cuda")
    y, gx = torch.zeros_like(gy), torch.zeros_like(x)
    tg.TVCBatch([dict(A=A, mode=mode, x=x, y=y, gy=gy, gx=gx)]).run()
    torch.cuda.synchronize()
    return gx.double()


@pytest.mark.parametrize("nk", [1, 2, 3])
def test_batched_gx_of_columns(nk):
    # A warp adds 128 columns (at most half the spacing of 2^31 is lost there,
    # and half of it in the result), then its compensated row sums.
    n = 1 << 17
    gx = batch_gx((1, nk, n), 1, 0, 2.0**31)
    assert abs(gx[0].item() - (2.0**31 + n - 1)) <= 512
    assert bool((gx[1:] == n).all())


def test_batched_gx_of_rows():
    # At most 64 products per plain partial sum: 63 terms lost beside 2^25, and
    # half its spacing per join of the eight warps and the result.
    n = 1 << 14
    gx = batch_gx((n, 64), 1, 0, 2.0**25)
    assert abs(gx[0].item() - (2.0**25 + n - 1)) <= 63 + 4 * 2
    assert bool((gx[1:] == n).all())


@pytest.mark.parametrize("dims", [(2, 2, 1200, 1200), (2, 2, 1450, 1000)])
def test_power_method_of_few_leading_entries(dims):
    # z_0[0] = 2^25 + n - 1 and z_0[1] = n: their quotient, to the rounding (2^-24
    # each) of the two entries of x_0 and of z_0[0], and of the tree over a block's
    # threads (nine levels of half a spacing of 2^25).  A plain chain loses one per
    # product of the thread that holds the large one, about 37.
    n = dims[2] * dims[3]
    A = torch.ones(dims, device="cuda")
    A.view(-1)[0] = 2.0**25
    one = torch.zeros(dims[1], device="cuda")
    one[0] = 1.0
    xs = [torch.ones(dims[0], device="cuda"), one] + [torch.ones(m, device="cuda") for m in dims[2:]]
    ws = torch.empty(tg.hopm_workspace_size(dims, tg.F32), dtype=torch.uint8, device="cuda")
    before = tg.kernel_launches()
    r = tg.hopm(A, xs, 1, workspace=ws).check()
    assert tg.kernel_launches() - before == 1  # the one-launch kernel
    got = r.x[0][0].double().item() / r.x[0][1].double().item()
    want = (2.0**25 + n - 1) / n
    assert abs(got - want) <= 3 * 2.0**-24 * want + 9 * 2 / n
