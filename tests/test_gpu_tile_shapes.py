"""The double-float Gram and update kernels of the streaming SVD at the edges of their launch rules
(odd column counts, an odd known block, one and several slices of column pairs, more than 40
columns, tiles shorter than a row chunk or ending inside one, every output-group width, extreme
scales) against the oracle's streaming SVD on the same vectors, at the bounds of svd_bounds."""
import numpy as np
import pytest

from oracle import icsvd
from paper_2505_14399_gb300 import api, synthetic
import svd_bounds
from gpu_common import to_dev
from test_gpu_setup_parity import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,block,k,r,n_s,scale", [
    ((2, 2, 2, 2), (1, 1, 2, 2), 3, 2, 3, 1.0),        # 24 rows, c = 2, 4, 5
    ((4, 4, 2, 2), (2, 2, 2, 2), 7, 9, 2, 1.0),        # 96 rows, odd known block (7), c = 9, 16
    ((6, 6, 6, 2), (3, 3, 3, 1), 1, 3, 3, 1.0),        # 162 rows, one column kept
    ((4, 4, 4, 4), (2, 2, 2, 4), 17, 16, 2, 1.0),      # 192 rows, c = 33, two slices
    ((4, 4, 4, 4), (4, 4, 2, 2), 32, 16, 3, 1.0),      # 384 rows, c = 48: four entries a thread
    ((6, 6, 6, 6), (3, 3, 3, 3), 10, 6, 2, 1.0),       # 486 rows: 15 chunks and 6 rows
    ((4, 4, 4, 4), (2, 2, 2, 2), 5, 5, 2, 1e-12),      # small and large fields
    ((4, 4, 4, 4), (2, 2, 2, 2), 8, 8, 2, 1e12),
])
def test_tile_shapes_match_oracle(dims, block, k, r, n_s, scale):
    U = synthetic.smooth_links(dims, 3)
    vec = (scale * synthetic.graded_fields(dims, r * n_s, 1.0, 4002)).astype(np.complex64)
    p = api.params(dims, block, 0.12, k, r, n_s, setup_dtype="c64", solve_dtype="c64")
    h = api.Hierarchy(to_dev(U), p, vectors=to_dev(vec))
    P, _ = h.prolongator()
    H = h.sigma_history().cpu().numpy()
    v = vec.astype(np.complex128)
    tiles = [icsvd.chiral_split(v[s * r:(s + 1) * r], dims, block) for s in range(n_s)]
    _check("tile_shapes", P.cpu().numpy(), H, tiles, k, svd_bounds.UDF)
    h.close()
