"""The direct forms of the DC screen (FP64, no iteration counts) and of the
adjoint (complete factor) where they can go wrong -- parallel circuits,
outages at the slack, bridges whose main island keeps no generator, ragged
tiles, no dense tail -- against the oracle and against the PCG forms."""
import numpy as np
import pytest

import paper_1803_03290_gb300 as gp
from oracle import adjoint, dc
from test_gpu_reduced import GRIDS

pytestmark = pytest.mark.gpu

KEYS = ("theta", "flow", "status", "max_loading", "n_overload", "overload")


@pytest.mark.parametrize("tail", [248, -1, 7])
@pytest.mark.parametrize("name", list(GRIDS))
def test_dc_direct(name, tail):
    g = GRIDS[name]()
    rng = np.random.default_rng(3)
    outages = rng.permutation(g.n_branch)[:151]
    outages = np.concatenate([outages, outages[:2]])  # an odd count, duplicates
    P = g.P_sched * rng.uniform(0.8, 1.2, g.n_bus)
    ref = dc.dc_screen(g, outages, P)
    with gp.GPCG(g, precision=gp.BATCHED_FP64, tail_rows=tail) as c:
        got = c.n1_dc_screen(outages, P=P, outputs=KEYS)
        pcg = c.n1_dc_screen(outages, P=P, outputs=KEYS + ("iters",))
        one = c.n1_dc_screen(outages[:1], P=P, outputs=KEYS)
    scale = max(1.0, np.abs(ref["theta"]).max())
    # FP64 direct solves: 1e-9 as the PCG's full-size test, to the angles' size
    assert np.abs(got["theta"] - ref["theta"]).max() < 1e-9 * scale
    assert np.abs(got["flow"] - ref["flow"]).max() < 1e-7 * scale
    assert np.abs(got["theta"] - pcg["theta"]).max() < 1e-9 * scale
    np.testing.assert_array_equal(got["status"], ref["status"])
    np.testing.assert_array_equal(got["status"], pcg["status"])
    tie = (np.abs(np.abs(ref["flow"]) / g.rating - 1.0) < 1e-6).any(1)
    np.testing.assert_array_equal(got["n_overload"][~tie], ref["n_overload"][~tie])
    assert (gp.unpack_mask(got["overload"], g.n_branch).sum(1) == got["n_overload"]).all()
    np.testing.assert_array_equal(one["theta"][0], got["theta"][0])


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
