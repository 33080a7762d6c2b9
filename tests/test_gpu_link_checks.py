"""The SU(3) check of the link copies: links with a NaN, an infinity or entries whose products
leave the FP32 range are not SU(3), wherever they stand."""
import numpy as np
import pytest

from paper_2505_14399_gb300 import _lib as L, api, synthetic
from gpu_common import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("emulation", [0, 1])        # without and with a double-float link copy
@pytest.mark.parametrize("value", [np.nan, np.inf, 1e25, 1e200])
@pytest.mark.parametrize("where", [0, 4, 8])
def test_non_su3_links_keep_three_rows(emulation, value, where):
    dims = (4, 4, 4, 4)
    U = synthetic.haar_links(dims, 3)
    U[2, 77].reshape(-1)[where] = value
    p = api.params(dims, (2, 2, 2, 2), 0.12, 4, 4, 1, fp64_emulation=emulation, link_compress=-1)
    h = api.Hierarchy(to_dev(U), p, setup=False)
    assert L.lib().mg_link_rows(h._h) == 3
    h.close()
    p.link_compress = 1
    with pytest.raises(Exception, match="SU\\(3\\)"):
        api.Hierarchy(to_dev(U), p, setup=False)
