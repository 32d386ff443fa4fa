"""The batch's items do no more work than the wanted results need: y and gA
without gx share nothing, so they must not cost what all three results do."""
import math
import random

import pytest
import torch

pytestmark = pytest.mark.gpu

tg = pytest.importorskip("paper_2501_03121_gb300")


def test_y_and_gA_alone():
    rng = random.Random(9)
    items = []
    for _ in range(512):
        d = (rng.randint(20, 200), rng.randint(20, 200))
        k, N = rng.randrange(2), math.prod(d)
        items.append(dict(A=torch.rand(d, device="cuda"), mode=k, x=torch.rand(d[k], device="cuda"),
                          y=torch.empty(N // d[k], device="cuda"), gy=torch.rand(N // d[k], device="cuda"),
                          gx=torch.empty(d[k], device="cuda"), gA=torch.empty(d, device="cuda")))

    def us(names):
        b = tg.TVCBatch([{k: v for k, v in it.items() if k in names or k in ("A", "mode", "x", "gy")} for it in items])
        b.run()
        torch.cuda.synchronize()
        s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            for _ in range(5):
                b.run(stream=s)
        best = float("inf")
        for _ in range(5):
            e0, e1 = torch.cuda.Event(True), torch.cuda.Event(True)
            with torch.cuda.stream(s):
                e0.record()
                g.replay()
                e1.record()
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1))
        return best

    # measured 0.3; 0.95 with one kind of item for both
    assert us(("y", "gA")) <= 0.6 * us(("y", "gx", "gA"))
