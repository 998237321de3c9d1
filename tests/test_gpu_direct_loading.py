"""Loadings of the direct DC screen: the maximum, the count and the mask against
the flows it returns."""
import numpy as np
import pytest

import paper_1803_03290_gb300 as gp
from test_gpu_reduced import GRIDS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", list(GRIDS))
def test_dc_direct_loading(name):
    g = GRIDS[name]()
    out = np.random.default_rng(3).permutation(g.n_branch)[:151]
    with gp.GPCG(g, precision=gp.BATCHED_FP64) as c:
        full = c.n1_dc_screen(out, outputs=("flow", "max_loading", "n_overload", "overload"))
        some = c.n1_dc_screen(out, outputs=("max_loading", "n_overload"))
    ld = np.abs(full["flow"]) / g.rating
    # one product with the reciprocal rating in place of the quotient
    np.testing.assert_allclose(full["max_loading"], ld.max(1), rtol=1e-14)
    clear = ~(np.abs(ld - 1.0) < 1e-12).any(1)
    np.testing.assert_array_equal(full["n_overload"][clear], (ld > 1.0).sum(1)[clear])
    np.testing.assert_array_equal(gp.unpack_mask(full["overload"], g.n_branch)[clear],
                                  (ld > 1.0)[clear])
    for k in some:
        np.testing.assert_array_equal(some[k], full[k])
