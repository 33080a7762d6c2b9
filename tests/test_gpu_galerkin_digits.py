"""The tensor-pipe Galerkin contraction over its column counts, row remainders and digit extremes."""
import numpy as np
import pytest
import torch

from oracle import coarse
from paper_2505_14399_gb300 import api, synthetic
from gpu_common import orthonormal_tiles, rel, to_dev

pytestmark = pytest.mark.gpu

KAPPA, W, BC = 0.125, (1, 1, 1, 1 / 3.5), (1, 1, 1, -1)


def _compare(U, P, dims, block, k):
    p = api.params(dims, block, KAPPA, k, k, 1, hop_weight=W, bc=BC, setup_dtype="c128",
                   solve_dtype="c128", fp64_emulation=1)
    h = api.Hierarchy(to_dev(U), p, setup=False)
    h.set_prolongator(to_dev(P))
    h.coarse_build()
    X, Y = (t.cpu().numpy() for t in h.coarse_op())
    h.close()
    Xo, Yo = coarse.galerkin(np.ascontiguousarray(np.swapaxes(P, 2, 3)), U, dims, block, KAPPA, W, BC)
    return max(rel(X, Xo), rel(Y, Yo))


# every count of eight-column tiles with even, odd and full k; blocks one or three sites wide
# (passes without sites, passes of three), 4 n + 1 .. 3 sites per pass
@pytest.mark.parametrize("dims,block,k", [
    ((4, 4, 2, 4), (1, 2, 2, 4), 1), ((4, 4, 4, 4), (2, 2, 2, 2), 3), ((6, 4, 2, 4), (3, 2, 1, 2), 4),
    ((6, 6, 2, 2), (3, 3, 2, 2), 7), ((4, 4, 4, 4), (2, 4, 2, 2), 8), ((6, 4, 4, 4), (3, 4, 2, 2), 9),
    ((4, 4, 4, 8), (4, 4, 4, 4), 11), ((4, 4, 4, 4), (2, 2, 4, 4), 12), ((4, 4, 4, 4), (2, 2, 2, 4), 13),
    ((4, 4, 4, 6), (4, 2, 2, 3), 16), ((4, 4, 4, 4), (2, 2, 2, 4), 17), ((6, 4, 4, 4), (3, 2, 2, 4), 20),
    ((4, 4, 4, 4), (2, 2, 4, 4), 21), ((4, 4, 4, 6), (2, 4, 2, 3), 24)])
def test_column_counts_and_remainders(dims, block, k):
    """Orthonormal tiles and unitary links: digit truncation (2^-55 per factor), dropped digit
    pairs (2^-53) and double-float sums (2^-47 per addition) stay below 1e-12 of the blocks."""
    nd = int(np.prod(block))
    P = orthonormal_tiles(int(np.prod(dims)) // nd, nd, k, 21)
    assert _compare(synthetic.smooth_links(dims, 5), P, dims, block, k) < 1e-12


@pytest.mark.parametrize("k", [4, 12, 24])
@pytest.mark.parametrize("digit", [127, -127])
def test_largest_digits_sum_exactly(k, digit):
    """Every digit of every entry at its largest and unit links: the FP32 sums of a fold come
    within two per cent of 2^24 in the last weights and use 23 bits in the leading ones, so a bit
    lost by the accumulators would show at 2^-21 .. 2^-45; the same bound as above."""
    dims, block = (4, 4, 4, 8), (4, 4, 4, 4)
    nd, d = 256, 2
    v = sum(digit * 2.0 ** (-6 - 8 * i) for i in range(6))   # 48 bits: a double and a pair hold it
    P = np.full((d, 2, k, 6 * nd), v + 0j)
    U = np.zeros((4, int(np.prod(dims)), 3, 3), dtype=complex)
    U[...] = np.eye(3)
    assert _compare(U, P, dims, block, k) < 1e-12
