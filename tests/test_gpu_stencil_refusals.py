"""Fields and links less aligned than the stencil's accesses are refused with an error by every
entry point that reaches it, before anything is launched."""
import ctypes as C

import pytest
import torch

from paper_2505_14399_gb300 import _lib as L, api, synthetic
from gpu_common import to_dev

pytestmark = pytest.mark.gpu

DIMS = (4, 4, 4, 4)
DT = {"c128": (L.MG_C128, 16), "c64": (L.MG_C64, 8), "f16": (L.MG_F16, 4), "bf16": (L.MG_BF16, 4)}


def _calls(dtype, field, links):
    """(name, status) of the stencil's entry points on buffers at these byte offsets."""
    dt, eb = DT[dtype]
    size = 256 * 36 * 4 * 16 + 64
    x, y, u, c = (torch.zeros(size, dtype=torch.uint8, device="cuda") for _ in range(4))
    dims, w, bc = L.ivec(DIMS), L.dvec((1, 1, 1, 1)), L.ivec((1, 1, 1, 1))
    px, py, pu = x.data_ptr() + field, y.data_ptr() + field, u.data_ptr() + links
    lib, n0 = L.lib(), L.lib().mg_kernel_launches()
    yield "dslash", lib.wilson_dslash(py, px, pu, dims, 0.1, w, bc, -1, 0, dt, 1, None)
    yield "parity", lib.wilson_dslash(py, px, pu, dims, 0.1, w, bc, 1, 0, dt, 2, None)
    yield "schur", lib.wilson_schur(py, px, pu, dims, 0.1, w, bc, 0, dt, 1, None)
    if dtype[0] == "c":
        yield "clover", lib.wilson_clover_apply(py, px, pu, c.data_ptr(), dims, 0.1, w, bc, 0, dt, 1,
                                                None)
    if field:
        p = api.params(DIMS, (2, 2, 2, 2), 0.1, 4, 4, 1, solve_dtype=dtype)
        h = api.Hierarchy(to_dev(synthetic.unit_links(DIMS)), p, setup=False)
        n0 = lib.mg_kernel_launches()
        yield "fine", lib.mg_apply_fine(h._h, py, px, 1, dt, 0, None)
        h.close()
    assert lib.mg_kernel_launches() == n0


@pytest.mark.parametrize("dtype,field,links", [
    ("c128", 8, 0), ("c64", 8, 0), ("f16", 8, 0), ("bf16", 4, 0),
    ("c128", 0, 8), ("c64", 0, 4), ("f16", 0, 2), ("bf16", 0, 2)])
def test_misaligned_buffers_are_refused(dtype, field, links):
    for name, status in _calls(dtype, field, links):
        assert status == L.MG_EINVAL, name
        assert b"aligned" in L.lib().mg_last_error(), name
