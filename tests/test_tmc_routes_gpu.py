"""Tensor-matrix contractions on both sides of the lines between the
register-blocked and the one-element kernels: few outputs over long modes, many
columns of short and long modes, rows, odd widths, slab scales, alpha and
beta."""
import pytest
import torch

pytestmark = pytest.mark.gpu

tg = pytest.importorskip("paper_2501_03121_gb300")

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16, "e4m3": torch.float8_e4m3fn}
# (u, n_k, v, R)
CASES = [(1, 127, 31, 13), (1, 128, 31, 13), (3, 70, 30, 5), (3, 1000, 42, 9), (3, 1000, 43, 9), (2, 9000, 60, 12), (1, 8191, 5, 8), (1, 8192, 5, 8),
         (2500, 16, 253, 13), (2500, 15, 253, 13), (613, 9, 2049, 16), (5, 600, 131072, 9), (130, 300, 2021, 17),
         (9000, 3, 517, 33), (9000, 2, 517, 33), (700, 64, 901, 6), (16, 600, 4099, 12),
         (127, 40, 1, 16), (128, 32, 1, 16), (128, 31, 1, 16), (70, 64, 1, 13), (511, 100, 1, 6), (512, 100, 1, 6), (3, 70001, 1, 5)]


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("dt", DTYPES)
@pytest.mark.parametrize("u,nk,v,R", CASES)
def test_against_64_bits(u, nk, v, R, dt, shift):
    g = torch.Generator(device="cuda").manual_seed(u + nk + v)
    flat = torch.zeros(u * nk * v + 16, dtype=DTYPES[dt], device="cuda")
    A = flat[shift:shift + u * nk * v]
    A.copy_((torch.rand(u * nk * v, generator=g, device="cuda") * 2 - 1).to(DTYPES[dt]))
    X = torch.rand(R, nk, generator=g, device="cuda") * 2 - 1
    Y = torch.rand(u, R, v, generator=g, device="cuda")
    scales = torch.rand(u, generator=g, device="cuda") + 0.5 if dt != "f32" else None
    ref = 0.5 * Y.double()
    step = max(1, (1 << 25) // (nk * v))
    for i in range(0, u, step):
        j = min(u, i + step)
        a = A[i * nk * v:j * nk * v].double().view(j - i, nk, v)
        y = -1.5 * torch.matmul(X.double(), a)
        ref[i:j] = 0.5 * Y[i:j].double() + (y if scales is None else y * scales[i:j].double().view(-1, 1, 1))
    got = tg.tmc(A, 1, X, Y=Y.clone(), scales=scales, alpha=-1.5, beta=0.5, shape=(u, nk, v)).view(u, R, v).double()
    assert float((got - ref).norm() / ref.norm()) <= 1e-5  # the parity bound of the TMC tests
