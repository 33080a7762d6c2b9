"""Streaming SVD on test vectors that are linearly dependent (a zero vector, a repeated one, a
combination of others), in every tile or in some: a kept direction of rounding noise, whose
eigenvalue is as often negative as positive, must not touch the accuracy of the others.  P against
the oracle's streaming SVD of the same vectors, at the double-float bounds of svd_bounds."""
import numpy as np
import pytest

from oracle import icsvd
from paper_2505_14399_gb300 import api, synthetic
import svd_bounds
from gpu_common import to_dev

pytestmark = pytest.mark.gpu


def _vectors(dims, r, n_s, kind):
    v = synthetic.graded_fields(dims, r * n_s, 1.0, 4010).reshape((n_s, r) + (-1, 4, 3))
    for s in range(n_s - 1):            # the last stream makes up the rank
        if kind == "zero":
            v[s, 1] = 0
        elif kind == "repeat":
            v[s, r - 1] = v[s, 0]
        elif kind == "combination":
            v[s, r - 1] = 0.5 * v[s, 0] - 2j * v[s, 1] + 0.25 * v[s, 2]
        else:                           # "local": equal on half of the lattice only
            n = v.shape[2] // 2
            v[s, r - 1, :n] = v[s, 0, :n]
    return v.reshape((n_s * r, -1, 4, 3)).astype(np.complex64)


@pytest.mark.parametrize("kind", ["zero", "repeat", "combination", "local"])
@pytest.mark.parametrize("dims,block,k,r,n_s", [
    ((4, 4, 4, 4), (2, 2, 2, 2), 8, 4, 3),       # 96 rows; 4 and 8 kept columns, then 12 -> 8
    ((4, 4, 4, 8), (2, 4, 2, 4), 12, 8, 3),      # 384 rows; 8, 12 of 16, 12 of 20
])
def test_other_columns_keep_their_accuracy(dims, block, k, r, n_s, kind):
    U = synthetic.smooth_links(dims, 3)
    vec = _vectors(dims, r, n_s, kind)
    p = api.params(dims, block, 0.12, k, r, n_s, setup_dtype="c64", solve_dtype="c64")
    h = api.Hierarchy(to_dev(U), p, vectors=to_dev(vec))
    P = h.prolongator()[0].cpu().numpy()
    S = h.sigma_history().cpu().numpy()[-1]
    h.close()
    v = vec.astype(np.complex128)
    tiles = [icsvd.chiral_split(v[s * r:(s + 1) * r], dims, block) for s in range(n_s)]
    Pt, So, _ = icsvd.icsvd_tiles(tiles, k)
    # the last stream's tiles have more independent columns than are kept, so the bounds hold for
    # P and for its singular values; a null value of an earlier stream is only known to the square
    # root of the Gram matrix's error and is not compared
    bp, bs = svd_bounds.vector_bounds(svd_bounds.stream_spectra(tiles, k), 0.0, svd_bounds.UDF,
                                      tiles[0].shape[2])[-1]
    ep = svd_bounds.projector_errors(P, Pt)
    assert np.all(ep <= bp), (ep / bp).max()
    assert np.all(np.abs(S - So).max(axis=-1) <= bs)
