"""The reduced form of the adjoint (complete factor) where they can go wrong -- parallel circuits,
outages at the slack, bridges whose main island keeps no generator, ragged
tiles, no dense tail -- against the oracle, as the PCG form."""
import numpy as np
import pytest

import paper_1803_03290_gb300 as gp
from oracle import adjoint
from test_gpu_reduced import GRIDS

pytestmark = pytest.mark.gpu

@pytest.mark.parametrize("precond", [gp.PRECOND_EXACT, gp.PRECOND_IC0])
@pytest.mark.parametrize("name", list(GRIDS))
def test_adjoint_forms(name, precond):
    g = GRIDS[name]()
    outages = np.random.default_rng(4).permutation(g.n_branch)[:61]
    b = np.random.default_rng(5).uniform(0.8, 1.2, g.n_branch) / g.x
    L, gP, gb = adjoint.loss_and_grad(g, outages, g.P_sched, b)
    with gp.GPCG(g, precond=precond) as c:
        l, a, k = c.n1_adjoint(outages, P=g.P_sched, b=b)
        again = c.n1_adjoint(outages, P=g.P_sched, b=b)
    # solves to 1e-12 (tests/test_gpu_adjoint.py compares at the same bounds)
    assert abs(l - L) < 1e-9 * abs(L)
    assert np.abs(a - gP).max() < 1e-7 * np.abs(gP).max()
    # (on a tree dL/db is zero: the terms it is the difference of set the scale)
    assert np.abs(k - gb).max() < 1e-7 * max(np.abs(gb).max(), np.abs(gP).max())
    assert again[0] == l and np.array_equal(again[1], a) and np.array_equal(again[2], k)
