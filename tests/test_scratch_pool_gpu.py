"""A warm-up call whose plan needs no scratch still prepares the library's
pool, so that a first captured call that does need some can be captured."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import torch
import paper_2501_03121_gb300 as tg
small = torch.ones(16, 16, 64, dtype=torch.float64, device="cuda")
tg.tvc(small, 0, torch.ones(16, dtype=torch.float64, device="cuda"))  # warm-up
A = torch.ones(500, 61, 40, dtype=torch.float64, device="cuda")
x = torch.ones(40, dtype=torch.float64, device="cuda")
y = torch.zeros(500, 61, dtype=torch.float64, device="cuda")
torch.cuda.synchronize()
s = torch.cuda.Stream()
g = torch.cuda.CUDAGraph()
with torch.cuda.stream(s):
    with torch.cuda.graph(g, stream=s):
        tg.tvc(A, 2, x, y=y, stream=s)
g.replay()
torch.cuda.synchronize()
assert torch.equal(y, torch.full_like(y, 40.0))
print("ok")
"""


def test_capture_after_a_call_without_scratch():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, cwd=root, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stderr
