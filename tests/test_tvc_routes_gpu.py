"""Contractions on both sides of the lines between the kernels: columns and rows
off 16-byte boundaries, phases of rows for few outputs and small tensors, splits
of n_k, every storage type, slab scales, against 64 bits."""
import pytest
import torch

pytestmark = pytest.mark.gpu

tg = pytest.importorskip("paper_2501_03121_gb300")

DTYPES = {"f64": torch.float64, "f32": torch.float32, "f32d": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16,
          "e4m3": torch.float8_e4m3fn}
TOL = {"f64": 1e-12, "f32d": 1e-12}  # the rest: the parity bound of FP32 accumulation
# (u, n_k, v) by what decides: ragged columns (pieces x rows), rows (row and tensor bytes), few outputs, small tensors
CASES = [(1, 513, 24401), (1, 512, 24335), (1, 129, 78001), (2, 40, 155701), (1, 7, 1600003), (1, 511, 3001), (9, 126, 4333),
         (5, 130, 38939),
         (20011, 101, 1), (2001, 101, 1), (41000, 99, 1), (1851, 534, 1), (8100, 501, 1), (16400, 979, 1), (30, 20011, 1),
         (5, 70001, 1), (300, 31, 1), (999, 17, 1),
         (1, 4096, 64), (1, 70000, 16), (1, 70001, 15), (1, 600000, 7), (1, 600001, 8), (1, 100000, 42), (2, 33000, 64),
         (1, 16846, 441), (1, 4096, 2001), (3, 9000, 12),
         (300, 15, 40), (300, 16, 40), (300, 16, 33), (40, 31, 128), (40, 32, 128), (40, 63, 131), (40, 64, 131), (9000, 20, 33),
         (1, 300, 64), (6, 13, 1134)]


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("dt", DTYPES)
@pytest.mark.parametrize("u,nk,v", CASES)
def test_contraction(u, nk, v, dt, shift):
    N = u * nk * v
    g = torch.Generator(device="cuda").manual_seed(u + nk + v)
    vt = torch.float64 if dt in ("f64", "f32d") else torch.float32
    flat = torch.zeros(N + 16, dtype=DTYPES[dt], device="cuda")
    A = flat[shift:shift + N]
    A.copy_((torch.rand(N, generator=g, dtype=vt if dt == "f64" else torch.float32, device="cuda") * 2 - 1).to(DTYPES[dt]))
    x = torch.rand(nk, generator=g, dtype=vt, device="cuda") * 2 - 1
    y = torch.rand(u * v, generator=g, dtype=vt, device="cuda")
    scales = torch.rand(u, generator=g, device="cuda") + 0.5 if dt in ("bf16", "f16", "e4m3") else None
    ref = (A.double().view(u, nk, v) * x.double().view(1, nk, 1)).sum(1)
    if scales is not None:
        ref = ref * scales.double().view(u, 1)
    ref = -1.5 * ref.reshape(-1) + 0.5 * y.double()
    shape = (u, nk, v) if v > 1 else (u, nk)
    got = tg.tvc(A, 1, x, y=y.clone(), scales=scales, alpha=-1.5, beta=0.5, shape=shape).view(-1).double()
    assert float((got - ref).norm() / ref.norm()) <= TOL.get(dt, 1e-5)


@pytest.mark.parametrize("dt", DTYPES)
@pytest.mark.parametrize("u,nk,v", [(1, 130, 26), (1, 369, 205), (3, 7, 39), (1, 26103, 1), (1, 261039, 1), (1, 9, 1), (200, 300, 5),
                                    (1, 20, 8191), (2, 2561, 33), (1, 1379, 984)])
def test_adjoint_of_few_pieces(u, nk, v, dt):
    g = torch.Generator(device="cuda").manual_seed(u + nk + v)
    vt = torch.float64 if dt in ("f64", "f32d") else torch.float32
    A = (torch.rand((u, nk, v), generator=g, dtype=vt if dt == "f64" else torch.float32, device="cuda") * 2 - 1).to(DTYPES[dt])
    gy = torch.rand(u * v, generator=g, dtype=vt, device="cuda") * 2 - 1
    ref = (A.double() * gy.double().view(u, 1, v)).sum((0, 2))
    scales = torch.rand(nk if u == 1 else u, generator=g, device="cuda") + 0.5 if dt in ("bf16", "f16", "e4m3") else None
    if scales is not None and u == 1:
        ref = ref * scales.double()
    elif scales is not None:
        ref = (A.double() * gy.double().view(u, 1, v) * scales.double().view(u, 1, 1)).sum((0, 2))
    shape, k = ((nk,), 0) if u == v == 1 else ((nk, v), 0) if u == 1 else ((u, nk, v), 1)
    got, _ = tg.tvc_backward(A.view(shape), k, None, gy, need_A=False, scales=scales,
                             code=tg._with_vectors(tg.dtype_code(A), gy))
    assert float((got.double() - ref).norm() / ref.norm()) <= TOL.get(dt, 1e-5)
