"""Every launch shape of the stencil, forced in a child process, for every storage type at every
accepted alignment (fields at odd multiples of 16 bytes, links at odd multiples of their element),
on lattices whose sites do not fill the last CTA and with a ragged last group of right-hand sides:
against the FP64 oracle, and an infinite component spreads in every shape as in the first one."""
import json
import os
import subprocess
import sys

import pytest

from paper_2505_14399_gb300 import api, synthetic

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import json, sys
sys.path.insert(0, "tests")
import numpy as np, torch
from oracle import wilson
from paper_2505_14399_gb300 import api, synthetic
from gpu_common import rel
from test_gpu_dslash_alignment import TOL, _dev, _host
W, BC = (1.0, 1.0, 1.0, 1 / 3.5), (1, 1, -1, -1)
EB = {"c128": 16, "c64": 8, "f16": 4, "bf16": 4}
out = {}
for dims in ((6, 10, 2, 6), (3, 5, 7, 2)):
    U = synthetic.haar_links(dims, 5)
    psi = synthetic.gaussian_rhs(dims, 6, 5)
    par = wilson.parity_of_sites(dims)
    for dtype in ("c128", "c64", "f16", "bf16"):
        for sf, sl in ((0, 0), (16, 0), (0, EB[dtype]), (16, EB[dtype])):
            Ud, pd = _dev(U, dtype, sl), _dev(psi, dtype, sf)
            Uh, ph = _host(Ud, dtype), _host(pd, dtype)
            w = (1.0,) * 4 if sl else W           # unit weights are left out of the arithmetic
            y = _host(api.dslash(pd, Ud, dims, 0.13, w, BC, dagger=sf > 0,
                                 out=_dev(psi, dtype, sf)), dtype)
            for r in range(5):
                e = rel(y[r], wilson.dslash(ph[r], Uh, dims, 0.13, w, BC, sf > 0))
                assert e < TOL[dtype], (dims, dtype, sf, sl, r, e)
            if dims[0] % 2 == 0:
                half = np.ascontiguousarray(psi[:, par == 0])
                hd = _dev(half, dtype, sf)
                hh = _host(hd, dtype)
                y = _host(api.dslash(hd, Ud, dims, 0.13, W, BC, parity=1,
                                     out=_dev(half, dtype, sf)), dtype)
                for r in range(5):
                    e = rel(y[r], wilson.dslash_parity(hh[r], Uh, dims, 0.13, 1, W, BC))
                    assert e < TOL[dtype], ("parity", dtype, sf, sl, r, e)
# the lane-contiguous copies of the half types, three and two rows per link
dims = (6, 10, 2, 6)
U, psi = synthetic.haar_links(dims, 9), synthetic.gaussian_rhs(dims, 6, 5)
for dtype in ("f16", "bf16"):
    for lc in (0, 1):
        p = api.params(dims, (2, 2, 2, 2), 0.13, 4, 4, 1, hop_weight=W, bc=BC, solve_dtype=dtype,
                       link_compress=lc)
        h = api.Hierarchy(torch.from_numpy(U).cuda(), p, setup=False)
        x = _dev(psi, dtype, 0)
        xh, y = _host(x, dtype), _host(h.apply_fine(x), dtype)
        h.close()
        for r in range(5):
            e = rel(y[r], wilson.dslash(xh[r], U, dims, 0.13, W, BC))
            assert e < TOL[dtype], ("lanes", dtype, lc, r, e)
# one infinite component at a time (every spin, both parts): which outputs are NaN, which infinite
dims = (6, 4, 6, 4)
U = synthetic.haar_links(dims, 7)
for dtype in ("c128", "c64"):
    psi = synthetic.gaussian_rhs(dims, 8, 8)
    for r in range(8):
        re, im = psi[r, 200, r // 2, 1].real, psi[r, 200, r // 2, 1].imag
        psi[r, 200, r // 2, 1] = complex(np.inf, im) if r % 2 else complex(re, -np.inf)
    Ud, pd = _dev(U, dtype, 0), _dev(psi, dtype, 0)
    for dag in (False, True):
        y = api.dslash(pd, Ud, dims, 0.13, W, BC, dagger=dag).cpu().numpy().view(
            np.float64 if dtype == "c128" else np.float32).ravel()
        out["%s_%d" % (dtype, dag)] = [int(np.isnan(y).sum()), int(np.isposinf(y).sum()),
                                       int(np.isneginf(y).sum()),
                                       int(np.flatnonzero(~np.isfinite(y)).sum())]
print(json.dumps(out))
"""


def _run(variant):
    env = dict(os.environ, WMG_DSLASH_VARIANT=str(variant), PYTHONPATH=ROOT)
    env.pop("WMG_AUTOTUNE_CACHE", None)
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    return json.loads(r.stdout.strip().splitlines()[-1])


@pytest.fixture(scope="module")
def first():
    return _run(0)


@pytest.mark.parametrize("variant", range(1, 9))
def test_forced_shape_every_storage_and_alignment(first, variant):
    assert _run(variant) == first


@pytest.mark.parametrize("shift_f,shift_l", [(16, 0), (0, 8), (16, 8)])
def test_less_aligned_calls_are_tuned_too(shift_f, shift_l):
    """Their shapes are candidates of the tuner as for aligned calls, under a key of their own."""
    from paper_2505_14399_gb300 import _lib
    from test_gpu_dslash_alignment import _dev
    dims = (10, 6, 4, 2 + shift_f // 8 + shift_l)           # keys of this test only
    U, psi = synthetic.haar_links(dims, 5), synthetic.gaussian_rhs(dims, 6, 3)
    count = _lib.lib().mg_kernel_launches
    for sf, sl in ((0, 0), (shift_f, shift_l)):
        Ud, x, y = _dev(U, "c64", sl), _dev(psi, "c64", sf), _dev(psi, "c64", sf)
        n = [count()]
        for _ in range(2):
            api.dslash(x, Ud, dims, 0.12, out=y)
            n.append(count())
        assert n[1] - n[0] > 1 and n[2] - n[1] == 1, (sf, sl, n)
