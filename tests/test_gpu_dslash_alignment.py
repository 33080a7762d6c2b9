"""The stencil's access forms against the FP64 oracle: 32-byte site accesses (aligned fields), the
16-byte forms (fields at an odd multiple of 16 bytes), ABI links at and off a 16-byte boundary
(windowed and element loads), on lattices whose CTA tiles are powers of two, ragged, or absent
(prime extents: consecutive sites)."""
import numpy as np
import pytest
import torch

from oracle import wilson
from paper_2505_14399_gb300 import api, synthetic
from gpu_common import from_half_pair, half_pair, rel, to_dev

pytestmark = pytest.mark.gpu

W, BC = (1.0, 1.0, 1.0, 1 / 3.5), (1, 1, -1, -1)
DIMS = [(2, 2, 2, 2), (16, 4, 2, 4), (6, 10, 4, 6), (34, 2, 2, 2)]      # every parity form
ODD = [(1, 1, 1, 1), (3, 5, 7, 2), (37, 1, 3, 2), (131, 1, 2, 1)]       # full lattice only
# bounds of the stencil's own parity tests; 16-bit storage: eight rounding errors of the inputs
TOL = {"c128": 1e-12, "c64": 1e-5, "f16": 8 * 2.0 ** -11, "bf16": 8 * 2.0 ** -8}
TORCH = {"c128": torch.complex128, "c64": torch.complex64, "f16": torch.float16,
         "bf16": torch.bfloat16}


def _dev(x, dtype, shift):
    """x on the device in storage `dtype`, `shift` bytes after a 256-byte boundary."""
    t = to_dev(x, TORCH[dtype]) if dtype[0] == "c" else half_pair(x, TORCH[dtype])
    n = t.numel() * t.element_size()
    buf = torch.empty(n + shift, dtype=torch.uint8, device=t.device)
    out = buf[shift:].view(t.dtype).reshape(t.shape)
    out.copy_(t)
    return out


def _host(t, dtype):
    return t.cpu().numpy().astype(np.complex128) if dtype[0] == "c" else from_half_pair(t)


@pytest.mark.parametrize("dtype", ["c128", "c64", "f16", "bf16"])
@pytest.mark.parametrize("dims", DIMS + ODD)
def test_alignment_forms_match_oracle(dims, dtype):
    eb = {"c128": 16, "c64": 8}.get(dtype, 4)
    U = synthetic.smooth_links(dims, 5)
    psi = synthetic.gaussian_rhs(dims, 6, 3)
    par = wilson.parity_of_sites(dims)
    for shift_f, shift_l in ((0, 0), (16, 0), (0, eb), (16, eb)):
        Ud, pd = _dev(U, dtype, shift_l), _dev(psi, dtype, shift_f)
        Uh, ph = _host(Ud, dtype), _host(pd, dtype)
        for dag in (False, True):
            out = _host(api.dslash(pd, Ud, dims, 0.13, W, BC, dagger=dag,
                                   out=_dev(psi, dtype, shift_f)), dtype)
            for r in range(3):
                assert rel(out[r], wilson.dslash(ph[r], Uh, dims, 0.13, W, BC, dag)) < TOL[dtype]
        if dims in DIMS:
            for p in (0, 1):
                half = np.ascontiguousarray(psi[:, par == 1 - p])
                hd = _dev(half, dtype, shift_f)
                hh = _host(hd, dtype)
                out = _host(api.dslash(hd, Ud, dims, 0.13, W, BC, parity=p,
                                       out=_dev(half, dtype, shift_f)), dtype)
                for r in range(3):
                    ref = wilson.dslash_parity(hh[r], Uh, dims, 0.13, p, W, BC)
                    assert rel(out[r], ref) < TOL[dtype]
