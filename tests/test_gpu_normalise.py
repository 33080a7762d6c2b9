"""FP32 Krylov vectors are normalised by the FP64 reciprocal of their norm, rounded once.

With kappa = 0 and unit links D is the identity, so one GMRES step on a vector with one non-zero
entry a leaves psi = a - y v with v = fl(f a), f = fl(1 / ||a||) and y the norm or, where v^2 > 1,
the norm over v^2; the aggregate's singular values are the |psi|, about 1e-8, which show one unit
in the last place of f.  (A clover term of 0 keeps the run off the fused first step, which
normalises nothing.)"""
import numpy as np
import pytest

from paper_2505_14399_gb300 import api, synthetic
from gpu_common import to_dev

pytestmark = pytest.mark.gpu
F = np.float32


def _psi(a, f):
    n = np.sqrt(float(F(a * a)))
    v = F(f * a)
    h = float(F(v * v))
    b2 = max(h - h * h, 0.0)
    y = F(n * h / (h * h + b2))
    return abs(float(F(float(a) - float(y) * float(v))))


def test_norm_reciprocal_is_rounded_once():
    dims = block = (4, 4, 4, 4)
    k = 32
    a = (1 + np.random.default_rng(5).random(k)).astype(F)
    vec = np.zeros((k, 256, 4, 3), dtype=np.complex64)
    for i in range(k):
        vec[i, 8 * i, 0, i % 3] = a[i]
    p = api.params(dims, block, 0.0, k, k, 1, sweeps=1, setup_dtype="c64", solve_dtype="c64", csw=1.0)
    h = api.Hierarchy(to_dev(synthetic.unit_links(dims)), p, vectors=to_dev(vec), smooth=True)
    S = h.prolongator()[1].cpu().numpy()[0, 0]
    h.close()
    n = np.sqrt((a * a).astype(np.float64))
    once = np.sort([_psi(x, F(1 / m)) for x, m in zip(a, n)])[::-1]
    twice = np.sort([_psi(x, F(1) / F(m)) for x, m in zip(a, n)])[::-1]
    assert np.abs(once - twice).max() > 1e-9       # the inputs tell the two apart
    assert np.abs(S - once).max() < 1e-12 + 1e-6 * once.max()


def test_norm_beyond_fp32_leaves_the_vectors_as_they_are():
    """Initial guesses phi whose squared norm overflows FP32 are not smoothed (as phi = 0 is not):
    the setup's results are those of phi itself, finite."""
    dims, block = (4, 4, 4, 4), (2, 2, 2, 2)
    v = (4e17 * synthetic.gaussian_rhs(dims, 6, 8)).astype(np.complex64)
    p = api.params(dims, block, 0.12, 4, 4, 2, setup_dtype="c64", solve_dtype="c64")
    out = []
    for smooth in (True, False):
        h = api.Hierarchy(to_dev(synthetic.smooth_links(dims, 5)), p, vectors=to_dev(v), smooth=smooth)
        out.append((h.prolongator()[0].cpu().numpy(), h.sigma_history().cpu().numpy()))
        h.close()
    assert np.all(np.isfinite(out[0][0])) and np.all(out[0][1] > 0)
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
