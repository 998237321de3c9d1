"""Launches of few scenarios (wide CTAs, one or two scenarios a tile): counts at
the rule's edges for 152 SMs, ragged last tiles, both precisions, grids with
fewer and more rows than threads -- against the same outages screened as part
of a long list, and the noalloc entry point's launch."""
import numpy as np
import pytest

import paper_1803_03290_gb300 as gp
from test_gpu_reduced import GRIDS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("n_bus", [300, 700, 1500])
def test_few_scenarios(n_bus, precision):
    import gridgen
    g = gridgen.make_grid(n_bus, int(1.4 * n_bus), 11, spur_frac=0.05, load_scale=0.03)
    keys = ("theta", "V", "flow", "label", "status", "n_overload", "max_loading")
    out = np.random.default_rng(2).integers(0, g.n_branch, 700).astype(np.int32)
    with gp.GPCG(g, tol=1e-10, max_outer=100, precision=precision) as c:
        c.base_solve()
        ref = c.n1_screen(out, outputs=keys)  # more than four scenarios per SM
        ok = np.isin(ref["status"], (0, 3))
        assert ok.mean() > 0.9
        sms = c.info()["num_sms"]
        for s in (1, 2, sms, sms + 1, 2 * sms - 1, 2 * sms + 1, 4 * sms):
            got = c.n1_screen(out[:s], outputs=keys)
            for k in ("status", "label"):
                np.testing.assert_array_equal(got[k], ref[k][:s])
            # the launches differ in the rounding of the inner solve only
            for k in ("theta", "V", "flow", "max_loading"):
                d = np.abs(got[k] - ref[k][:s])[ok[:s]]
                assert d.size == 0 or d.max() < 1e-6


@pytest.mark.parametrize("name", list(GRIDS))
def test_base_solve(name):
    """The base case, always a wide launch, against the oracle."""
    from oracle import powerflow as pf
    g = GRIDS[name]()
    th, V, k, st, _ = pf.base_case(g, tol=1e-11, max_outer=200)
    with gp.GPCG(g) as c:
        b = c.base_solve()
    assert np.abs(b["theta"] - th).max() < 1e-6 and np.abs(b["V"] - V).max() < 1e-6
