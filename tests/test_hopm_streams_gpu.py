"""Power methods of small tensors on several streams at once: a run leaves most
of the GPU to the others, so eight captured runs take far less than eight times
one."""
import time

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

tg = pytest.importorskip("paper_2501_03121_gb300")


def test_small_runs_overlap():
    dims, n = (32, 32, 32), 8
    A = torch.rand(dims, dtype=torch.float64, device="cuda") + 0.1
    one = [torch.full((m,), m**-0.5, dtype=torch.float64, device="cuda") for m in dims]
    want = tg.hopm(A, one, 20).check()
    runs = []
    for _ in range(n):
        s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        x = [v.clone() for v in one]
        ws = torch.empty(tg.hopm_workspace_size(dims, tg.F64), dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=s):
            r = tg.hopm(A, x, 20, workspace=ws, inplace=True, stream=s)
        runs.append((s, g, x, r, ws))

    def wall(k):
        best = float("inf")
        for _ in range(5):
            torch.cuda.synchronize()
            t = time.perf_counter()
            for s, g, x, r, ws in runs[:k]:
                with torch.cuda.stream(s):
                    g.replay()
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t)
        return best

    for _, _, x, _, _ in runs:
        for a, b in zip(x, one):
            a.copy_(b)
    wall(n)
    # measured 1.1x of one run; 8x when each takes the whole GPU
    assert wall(n) <= 4 * wall(1)
    for s, g, x, r, ws in runs:
        assert abs(r.lam.item() - want.lam.item()) <= 1e-12 * want.lam.item()
        assert all(np.allclose(a.cpu(), b.cpu(), rtol=1e-9, atol=1e-12) for a, b in zip(x, want.x))
