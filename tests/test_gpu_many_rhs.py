"""Transfers with more right-hand sides than a grid has rows (65 535)."""
import numpy as np
import pytest
import torch

from oracle import coarse
from paper_2505_14399_gb300 import api, synthetic
from gpu_common import orthonormal_tiles, rel, to_dev

pytestmark = pytest.mark.gpu


def test_prolong_beyond_the_grid_limit():
    dims = block = (2, 2, 2, 2)
    n, k = 65535 + 3, 2
    p = api.params(dims, block, 0.12, k, k, 1)
    h = api.Hierarchy(to_dev(synthetic.haar_links(dims, 1)), p, setup=False)
    P = orthonormal_tiles(1, 16, k, 2)
    h.set_prolongator(to_dev(P))
    rng = np.random.default_rng(3)
    vc = rng.standard_normal((n, 1, 2, k)) + 1j * rng.standard_normal((n, 1, 2, k))
    v = h.prolong(to_dev(vc))
    Pt = np.ascontiguousarray(np.swapaxes(P, 2, 3))
    for r in (0, 1, 65534, 65535, n - 1):
        assert rel(v[r].cpu().numpy(), coarse.prolong(Pt, vc[r], dims, block)) < 1e-13, r
    h.close()
