"""The memory that the library keeps between calls (scratch pool, freed blocks of closed handles)
goes back to the device on request, and calls after that work as before."""
import pytest
import torch

from paper_2505_14399_gb300 import api, synthetic
from gpu_common import to_dev

pytestmark = pytest.mark.gpu


def test_kept_memory_is_given_back():
    dims = (16, 16, 16, 16)
    U = torch.randn((4, 16 ** 4, 3, 3), dtype=torch.complex64, device="cuda")
    x = torch.randn((12, 16 ** 4 // 2, 4, 3), dtype=torch.complex64, device="cuda")
    y = api.schur(x, U, dims, 0.12)
    p = api.params(dims, (4, 4, 4, 4), 0.12, 4, 4, 1)
    links = to_dev(synthetic.unit_links(dims))
    api.Hierarchy(links, p, setup=False).close()
    z = torch.empty_like(x)
    torch.equal(z.zero_(), y)                    # torch has its code and memory by now
    torch.cuda.synchronize()
    api.release_memory()
    free0 = torch.cuda.mem_get_info()[0]
    api.schur(x, U, dims, 0.12, out=z)           # scratch: half of the field, 38 MB
    api.Hierarchy(links, p, setup=False).close()
    torch.cuda.synchronize()
    assert torch.equal(z, y)
    kept = free0 - torch.cuda.mem_get_info()[0]
    assert kept >= 100 << 20, kept
    api.release_memory()
    assert torch.cuda.mem_get_info()[0] >= free0 - (8 << 20)
