"""The workloads whose running time counts, each through the package's public calls.

kinds
  tvc     y_k = A x_k x_k along every mode k of one tensor: what the bandwidth
          sweep and the Table 1 measurement do with each tensor.
  hopm    a power method of a fixed number of sweeps.
  adjoint forward and backward of the contraction through autograd, every
          mode: gradients with respect to the tensor and to the vector.
  batch   many FP32 tensors of uneven order and shape, one contraction and both
          adjoints each, in one persistent launch.
  hbatch  a power method on each of many such tensors, in one launch.
  mttkrp  M_k = A_(k) (Khatri-Rao of the other factors) for every mode k: the
          tensor work of one sweep of CP-ALS.

Every input is made from the seed with torch's own generator.  Narrow storage
is made with torch's own conversions, so that the values in 64 bits are known
without this package: bfloat16 and float16 by rounding, E4M3 by dividing each
slab A[i_0, ...] by amax/448 and rounding.
"""
import math
import random

import torch

import paper_2501_03121_gb300 as tg

DEV = "cuda"
ELEM = {"f64": 8, "f32": 4, "f32d": 4, "bf16": 2, "f16": 2, "e4m3": 1}


def listed():
    return [
        # The plain method's tensor, FP64, three modes: the smallest calls, where
        # launches and host work count.
        {"name": "tvc_f64_128^3", "kind": "tvc", "dims": "128,128,128", "dtype": "f64"},
        # A Table 1 tensor (7.1 GB, FP64, odd dimensions): columns, slabs and rows
        # of 31 entries.
        {"name": "tvc_f64_31^6", "kind": "tvc", "dims": "31,31,31,31,31,31", "dtype": "f64"},
        # The same kind of tensor in FP32: 63^5, rows and slabs of 63.
        {"name": "tvc_f32_63^5", "kind": "tvc", "dims": "63,63,63,63,63", "dtype": "f32"},
        # Table 1 shapes in the paper's storage-only low precision: 175^4 in BF16
        # and 979^3 in E4M3 with per-slab scales; odd row lengths.
        {"name": "tvc_bf16_175^4", "kind": "tvc", "dims": "175,175,175,175", "dtype": "bf16"},
        {"name": "tvc_e4m3_979^3", "kind": "tvc", "dims": "979,979,979", "dtype": "e4m3"},
        # The plain method's power method: 20 sweeps from all-ones on a tensor
        # that fits L2; latency counts.
        {"name": "hopm_f64_128^3", "kind": "hopm", "dims": "128,128,128", "dtype": "f64", "sweeps": 20},
        # Planted rank-1 plus noise, 17 GB FP32: the largest tensor.
        {"name": "hopm_f32_256^4", "kind": "hopm", "dims": "256,256,256,256", "dtype": "f32", "sweeps": 10},
        # Low-precision power method, E4M3 with per-slab scales.
        {"name": "hopm_e4m3_2048^3", "kind": "hopm", "dims": "2048,2048,2048", "dtype": "e4m3", "sweeps": 10},
        # A training step of the contraction on a tensor of the bandwidth sweep.
        {"name": "adjoint_f32_128^4", "kind": "adjoint", "dims": "128,128,128,128", "dtype": "f32"},
        # The batched workload at an eighth of its 4096 tensors (three states have
        # to fit beside their gradients).
        {"name": "batch_512", "kind": "batch", "count": 512, "shapes": 0},
        {"name": "hbatch_512", "kind": "hbatch", "count": 512, "shapes": 0, "sweeps": 10},
        # CP-ALS with 16 components on the sweep's 1024^3 tensor.
        {"name": "mttkrp_f32_1024^3_r16", "kind": "mttkrp", "dims": "1024,1024,1024", "dtype": "f32", "rank": 16},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _dims(rng, order, N):
    """`order` dimensions of product at most N and near it, none below 2."""
    w = [rng.uniform(0.5, 1.5) for _ in range(order)]
    s = sum(w)
    dims = [max(2, int(round(N ** (v / s)))) for v in w]
    while math.prod(dims) > N:
        dims[dims.index(max(dims))] -= 1
    return dims


def draw(rng):
    kind = rng.choice(["tvc", "tvc", "tvc", "hopm", "hopm", "adjoint", "batch", "hbatch", "mttkrp"])
    if kind in ("batch", "hbatch"):
        c = {"kind": kind, "count": int(round(_log(rng, 24, 512))), "shapes": rng.randrange(1, 1 << 20)}
        if kind == "hbatch":
            c["sweeps"] = rng.randint(3, 10)
        return c
    if kind == "tvc":
        dtype, order = rng.choice(["f64", "f32", "bf16", "e4m3", "f16", "f32d"]), rng.randint(2, 8)
        N = _log(rng, 2e6, 8e8)
    elif kind == "hopm":
        dtype, order = rng.choice(["f64", "f32", "bf16", "e4m3"]), rng.randint(3, 5)
        N = _log(rng, 2e6, 2e9)
    elif kind == "adjoint":
        dtype, order = rng.choice(["f32", "f32", "f64"]), rng.randint(2, 5)
        N = _log(rng, 2e6, 2.6e8)
    else:
        dtype, order = rng.choice(["f32", "f32", "bf16"]), rng.randint(3, 4)
        N = _log(rng, 2e7, 1e9)
    dims = _dims(rng, order, N)
    c = {"kind": kind, "dims": ",".join(map(str, dims)), "dtype": dtype}
    if kind == "hopm":
        c["sweeps"] = rng.randint(4, 20) if N < 5e8 else rng.randint(3, 10)
    if kind == "mttkrp":
        c["rank"] = rng.randint(4, 32)
    return c


# ------------------------------------------------------------------ inputs


def _shape(case):
    return tuple(int(n) for n in case["dims"].split(","))


def _vec(dtype):
    return torch.float64 if dtype in ("f64", "f32d") else torch.float32


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _uniform(g, shape, dtype):
    return torch.rand(shape, generator=g, dtype=dtype, device=DEV).mul_(2).sub_(1)


def _unit(g, n):
    v = torch.randn(n, generator=g, dtype=torch.float64, device=DEV)
    return v / v.norm()


def _stored(src, dtype):
    """(codes or values, scales) of an FP32/FP64 source in the storage type."""
    if dtype in ("f64", "f32", "f32d"):
        return src, None
    if dtype == "bf16":
        return src.to(torch.bfloat16), None
    if dtype == "f16":
        return src.to(torch.float16), None
    scales = src.view(src.shape[0], -1).abs().amax(dim=1) / 448.0
    src.div_(scales.view(-1, *[1] * (src.dim() - 1)))
    return src.to(torch.float8_e4m3fn), scales


def _plant(A, us, noise):
    """A = noise * A + 10 u_0 (x) u_1 (x) ... in place."""
    rest = us[1].to(A.dtype)
    for u in us[2:]:
        rest = torch.outer(rest, u.to(A.dtype)).reshape(-1)
    A.mul_(noise)
    A.view(A.shape[0], -1).addr_(us[0].to(A.dtype), rest, alpha=10.0)


def _start(g, us, vt):
    """Start vectors that overlap the planted factors: u_j plus a unit Gaussian vector, normalised."""
    xs = []
    for u in us:
        v = u + _unit(g, u.numel())
        xs.append((v / v.norm()).to(vt))
    return xs


def _hopm_inputs(case, seed):
    shape, dtype = _shape(case), case["dtype"]
    g = _gen(seed)
    if dtype == "f64":  # the plain method: uniform entries, all-ones start
        A = _uniform(g, shape, torch.float64)
        return A, None, [torch.full((n,), 1 / math.sqrt(n), dtype=torch.float64, device=DEV) for n in shape]
    A = torch.empty(shape, dtype=torch.float32, device=DEV).normal_(generator=g)
    us = [_unit(g, n) for n in shape]
    _plant(A, us, 0.01)
    A, scales = _stored(A, dtype)
    return A, scales, _start(g, us, torch.float32)


def _dense_inputs(case, seed):
    """Tensor with uniform[-1, 1) entries in the case's storage, and one vector per mode."""
    shape, dtype = _shape(case), case["dtype"]
    g = _gen(seed)
    A, scales = _stored(_uniform(g, shape, torch.float64 if dtype == "f64" else torch.float32), dtype)
    return A, scales, [_uniform(g, (n,), _vec(dtype)) for n in shape], g


def _batch_shapes(case):
    """Order 3 or 4, dimensions uniform in [8, 192], redrawn above 2^24 elements; a random mode."""
    rng = random.Random(case["shapes"])
    spec = []
    for _ in range(case["count"]):
        d = rng.randint(3, 4)
        while True:
            dims = tuple(rng.randint(8, 192) for _ in range(d))
            if math.prod(dims) <= 1 << 24:
                break
        spec.append((dims, rng.randrange(d)))
    return spec


class _Pool:
    """One device buffer cut into pieces that start on 256-byte boundaries, as an allocator's would."""

    def __init__(self, sizes):
        self.at, off = [], 0
        for n in sizes:
            self.at.append((off, n))
            off += -(-n // 64) * 64
        self.flat = torch.zeros(off, dtype=torch.float32, device=DEV)
        self.parts = [self.flat[o:o + n] for o, n in self.at]


def _batch_inputs(case, seed):
    spec, g = _batch_shapes(case), _gen(seed)
    A = _Pool([math.prod(d) for d, _ in spec])
    x = _Pool([d[m] for d, m in spec])
    gy = _Pool([math.prod(d) // d[m] for d, m in spec])
    for p in (A, x, gy):
        p.flat.uniform_(-1, 1, generator=g)
    return spec, A, x, gy


def _hbatch_inputs(case, seed):
    spec, g = _batch_shapes(case), _gen(seed)
    A = _Pool([math.prod(d) for d, _ in spec])
    A.flat.normal_(generator=g)
    x0 = _Pool([n for d, _ in spec for n in d])
    at = 0
    for (d, _), a in zip(spec, A.parts):
        us = [_unit(g, n) for n in d]
        _plant(a.view(d), us, 0.01)
        for v in _start(g, us, torch.float32):
            x0.parts[at].copy_(v)
            at += 1
    return spec, A, x0


def _mttkrp_inputs(case, seed):
    A, _, _, g = _dense_inputs(case, seed)
    return A, [_uniform(g, (n, case["rank"]), torch.float32) for n in A.shape]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "tvc":
        A, scales, xs, _ = _dense_inputs(case, seed)
        return {"kind": kind, "A": A, "scales": scales, "xs": xs}
    if kind == "hopm":
        A, scales, xs = _hopm_inputs(case, seed)
        return {"kind": kind, "A": A, "scales": scales, "xs": xs, "sweeps": case["sweeps"]}
    if kind == "adjoint":
        A, _, xs, g = _dense_inputs(case, seed)
        gys = [_uniform(g, tuple(n for i, n in enumerate(A.shape) if i != k), A.dtype) for k in range(A.dim())]
        return {"kind": kind, "A": A.requires_grad_(), "xs": [x.requires_grad_() for x in xs], "gys": gys}
    if kind == "batch":
        spec, A, x, gy = _batch_inputs(case, seed)
        y, gx, gA = (_Pool([n for _, n in p.at]) for p in (gy, x, A))
        plan = tg.TVCBatch([
            dict(A=A.parts[b], shape=d, mode=m, x=x.parts[b], y=y.parts[b], gy=gy.parts[b], gx=gx.parts[b],
                 gA=gA.parts[b]) for b, (d, m) in enumerate(spec)])
        return {"kind": kind, "plan": plan, "out": [y.flat, gx.flat, gA.flat], "keep": (A, x, gy)}
    if kind == "hbatch":
        spec, A, x0 = _hbatch_inputs(case, seed)
        x = _Pool([n for _, n in x0.at])
        lam = torch.zeros(len(spec), dtype=torch.float64, device=DEV)
        items, at = [], 0
        for b, (d, _) in enumerate(spec):
            items.append(dict(A=A.parts[b], shape=d, x=x.parts[at:at + len(d)], lam=lam[b:b + 1]))
            at += len(d)
        return {"kind": kind, "plan": tg.HOPMBatch(items, case["sweeps"]), "x": x, "x0": x0, "lam": lam, "keep": A}
    A, factors = _mttkrp_inputs(case, seed)
    return {"kind": kind, "A": A, "factors": factors}


def run(s):
    kind = s["kind"]
    if kind == "tvc":
        return [tg.tvc(s["A"], k, x, scales=s["scales"]) for k, x in enumerate(s["xs"])]
    if kind == "hopm":
        r = tg.hopm(s["A"], s["xs"], s["sweeps"], scales=s["scales"])
        # lambda carries the precision of the vectors that it is the norm of
        return {"x": r.x, "lam": r.lam.to(r.x[0].dtype)}
    if kind == "adjoint":
        out = []
        for k, (x, gy) in enumerate(zip(s["xs"], s["gys"])):
            y = tg.tvc_autograd(s["A"], x, k)
            out.append((y.detach(),) + torch.autograd.grad(y, (s["A"], x), gy))
        return out
    if kind == "batch":
        s["plan"].run()
        return s["out"]
    if kind == "hbatch":
        s["x"].flat.copy_(s["x0"].flat)
        s["plan"].run()
        return {"x": s["x"].flat, "lam": s["lam"].float()}
    return [tg.mttkrp(s["A"], k, s["factors"]) for k in range(s["A"].dim())]


def work(case):
    kind = case["kind"]
    if kind in ("batch", "hbatch"):
        nbytes = flops = 0
        for dims, m in _batch_shapes(case):
            N = math.prod(dims)
            if kind == "batch":  # A for both products; gA, y and gx written
                nbytes += 4 * (2 * N + 2 * N // dims[m] + 2 * dims[m])
                flops += 5 * N
            else:  # A twice a sweep: x_0 needs x_1, and x_1 needs the new x_0
                nbytes += 4 * case["sweeps"] * 2 * N
                flops += 4 * N * case["sweeps"]
        return {"bytes": nbytes, "flops": flops}
    dims = _shape(case)
    N, es = math.prod(dims), ELEM[case["dtype"]]
    vs = 8 if _vec(case["dtype"]) == torch.float64 else 4
    if kind == "tvc":
        return {"bytes": sum(N * es + n * vs + N // n * vs for n in dims), "flops": 2 * N * len(dims)}
    if kind == "hopm":
        # a tensor that fits the 129 MB L2 has to come from memory once only
        times = 2 * case["sweeps"] if N * es > 100e6 else 1
        return {"bytes": N * es * times, "flops": 4 * N * case["sweeps"]}
    if kind == "adjoint":
        return {"bytes": sum(3 * N * es + 2 * n * vs + 2 * N // n * vs for n in dims), "flops": 5 * N * len(dims)}
    return {"bytes": len(dims) * N * es, "flops": 2 * N * case["rank"] * len(dims)}


# ------------------------------------------------------------------- exact


def _pieces(A, scales, most=1 << 27):
    """(first index, FP64 values) of runs of slabs of A of at most about `most` elements."""
    step = max(1, most // max(1, A[0].numel()))
    for i in range(0, A.shape[0], step):
        v = A[i:i + step].to(torch.float64)
        if scales is not None:
            v = v * scales[i:i + step].to(torch.float64).view(-1, *[1] * (A.dim() - 1))
        yield i, v


def _along(B, k, x):
    """B x_k x in FP64."""
    u, v = math.prod(B.shape[:k]), math.prod(B.shape[k + 1:])
    shape = tuple(n for i, n in enumerate(B.shape) if i != k)
    if v == 1:
        return torch.mv(B.reshape(u, -1), x).view(shape)
    return torch.matmul(x, B.reshape(u, B.shape[k], v)).view(shape)


def _tvc64(A, scales, k, x):
    x, out = x.to(torch.float64), []
    for i, v in _pieces(A, scales):
        out.append(_along(v, 0, x[i:i + v.shape[0]]) if k == 0 else _along(v, k, x))
    if k:
        return torch.cat(out)
    return torch.stack(out).sum(0)


def _hopm64(A, scales, xs, sweeps):
    xs = [x.to(torch.float64) for x in xs]
    lam = None
    for _ in range(sweeps):
        for j in range(len(xs)):
            k = 1 if j == 0 else 0
            B, left = _tvc64(A, scales, k, xs[k]), [m for m in range(len(xs)) if m != k]
            for m in reversed([m for m in left if m != j]):
                B = _along(B, left.index(m), xs[m])
                left.remove(m)
            lam = B.norm()
            xs[j] = B / lam
    return xs, lam


def exact(case, seed):
    kind = case["kind"]
    if kind == "tvc":
        A, scales, xs, _ = _dense_inputs(case, seed)
        return [_tvc64(A, scales, k, x) for k, x in enumerate(xs)]
    if kind == "hopm":
        A, scales, xs = _hopm_inputs(case, seed)
        xs, lam = _hopm64(A, scales, xs, case["sweeps"])
        return {"x": xs, "lam": lam.view(1)}
    if kind == "adjoint":
        A, _, xs, g = _dense_inputs(case, seed)
        out = []
        for k, x in enumerate(xs):
            gy = _uniform(g, tuple(n for i, n in enumerate(A.shape) if i != k), A.dtype).to(torch.float64).unsqueeze(k)
            shape = [1] * A.dim()
            shape[k] = -1
            gx = torch.zeros(A.shape[k], dtype=torch.float64, device=DEV)
            for i, v in _pieces(A, None):
                if k == 0:
                    gx[i:i + v.shape[0]] = torch.mv(v.reshape(v.shape[0], -1), gy.reshape(-1))
                else:
                    gx += (v * gy[i:i + v.shape[0]]).transpose(0, k).reshape(A.shape[k], -1).sum(1)
            out.append((_tvc64(A, None, k, x), gy * x.to(torch.float64).view(shape), gx))
        return out
    if kind == "batch":
        spec, A, x, gy = _batch_inputs(case, seed)
        y, gx, gA = (torch.zeros_like(p.flat, dtype=torch.float64) for p in (gy, x, A))
        for b, (d, m) in enumerate(spec):
            a, v = A.parts[b].view(d).to(torch.float64), x.parts[b].to(torch.float64)
            w = gy.parts[b].view(*d[:m], 1, *d[m + 1:]).to(torch.float64)
            shape = [1] * len(d)
            shape[m] = -1
            for out, p, r in ((y, gy, _along(a, m, v)),
                              (gx, x, (a * w).transpose(0, m).reshape(d[m], -1).sum(1)), (gA, A, w * v.view(shape))):
                o, n = p.at[b]
                out[o:o + n] = r.reshape(-1)
        return [y, gx, gA]
    if kind == "hbatch":
        spec, A, x0 = _hbatch_inputs(case, seed)
        x, lam, at = torch.zeros_like(x0.flat, dtype=torch.float64), [], 0
        for b, (d, _) in enumerate(spec):
            xs, sigma = _hopm64(A.parts[b].view(d), None, x0.parts[at:at + len(d)], case["sweeps"])
            for m, v in enumerate(xs):
                o, n = x0.at[at + m]
                x[o:o + n] = v
            at += len(d)
            lam.append(sigma)
        return {"x": x, "lam": torch.stack(lam)}
    A, factors = _mttkrp_inputs(case, seed)
    F = [f.to(torch.float64) for f in factors]
    out = []
    for k in range(A.dim()):
        M = torch.zeros(A.shape[k], case["rank"], dtype=torch.float64, device=DEV)
        for i, v in _pieces(A, None):
            G = [F[0][i:i + v.shape[0]]] + F[1:]
            other = [m for m in range(A.dim()) if m != k]
            K = G[other[0]]
            for m in other[1:]:
                K = (K[:, None, :] * G[m][None, :, :]).reshape(-1, case["rank"])
            part = v.movedim(k, 0).reshape(v.shape[k], -1) @ K
            if k == 0:
                M[i:i + v.shape[0]] = part
            else:
                M += part
        out.append(M)
    return out
