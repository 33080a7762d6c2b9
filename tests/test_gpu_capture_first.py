"""The first call of a process may be made while its stream is captured: the scratch of the captured
call is the graph's."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import torch
from paper_2505_14399_gb300 import api, synthetic
dims = (4, 4, 4, 8)
U = torch.from_numpy(synthetic.haar_links(dims, 1)).to(torch.complex64).cuda()
x = torch.randn((2, 256, 4, 3), dtype=torch.complex64, device="cuda")
y = torch.empty_like(x)
graphs = []
for _ in range(2):                  # the first call of the process, then one with the pool in use
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        api.schur(x, U, dims, 0.12, out=y)
    graphs.append(g)
    for h in 2 * graphs:
        x.copy_(torch.randn_like(x))
        y.zero_()
        h.replay()
        z = api.schur(x, U, dims, 0.12)
        assert float((y - z).abs().max()) < 1e-5
print("ok")
"""


def test_first_call_under_capture():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True,
                       env=dict(os.environ, PYTHONPATH=ROOT), timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
