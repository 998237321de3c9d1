"""The overload screen without flow outputs settles most branches on FP32 values
with an error bound: counts, masks and maxima have to be those of the FP64
evaluation that a call with flows makes, also for ratings within 1e-12 ... 1e-4
of the flows, on both sides, taps and islands included."""
import numpy as np
import pytest

import paper_1803_03290_gb300 as gp
from test_gpu_reduced import GRIDS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [2, 8])
@pytest.mark.parametrize("name", ["meshed_taps", "tree_no_pq", "spurs"])
def test_screen_without_flows(name, tile):
    g = GRIDS[name]()
    with gp.GPCG(g, tile=tile) as c:
        flow = c.base_solve()["flow"]
    rng = np.random.default_rng(6)
    off = rng.choice([-1, 1], g.n_branch) * 10.0 ** rng.uniform(-12, -4, g.n_branch)
    g.rating = np.abs(flow) * (1 + off) + 1e-9
    out = np.concatenate([np.arange(g.n_branch), np.arange(g.n_branch)[:3]])
    keys = ("status", "max_loading", "n_overload", "overload")
    with gp.GPCG(g, tile=tile, tol=1e-6) as c:
        c.base_solve()
        full = c.n1_screen(out, outputs=keys + ("flow",))
        for some in (keys, keys[:1] + keys[2:], ("n_overload",), ("max_loading",)):
            got = c.n1_screen(out, outputs=some)
            for k in some:
                np.testing.assert_array_equal(got[k], full[k], err_msg=f"{k} of {some}")
    assert (full["n_overload"] > 0).any()
