"""The inner solves in their two-dimensional Krylov space (complete base-case
factor) on the structures where they differ from the general PCG: parallel
circuits, hubs whose factor rows overflow the padded slots, outages at the
slack, bridges with PV or no generation behind them, no PQ bus at all, and
level schedules with and without a dense tail -- against the oracle and
against the PCG with an incomplete factor, in both precisions.
"""
import numpy as np
import pytest

import gridgen
from oracle import powerflow as pf
from oracle import screen
from cases import grid_from_arrays, random_tree_grid

pytestmark = pytest.mark.gpu


def _meshed(n, seed, taps):
    """Ring with chords, parallel circuits, a hub and two spurs."""
    rng = np.random.default_rng(seed)
    f = [i for i in range(n)] + [0] * 9 + [3, 3, 0]
    t = [(i + 1) % n for i in range(n)] + list(range(4, 22, 2)) + [4, 4, 1]
    f += [5, n, 7]  # a chain of two and a single spur
    t += [n, n + 1, n + 2]
    m, nb = len(f), n + 3
    bt = np.zeros(nb)
    bt[0] = 2
    bt[[2, 9, 15, n + 1]] = 1
    P = rng.uniform(-0.15, 0.0, nb)
    Pg = np.where(bt == 1, 0.4, 0.0)
    P = P + Pg
    x = rng.uniform(0.02, 0.1, m)
    return grid_from_arrays(bt, P, -0.05 * np.ones(nb), Pg, np.where(bt > 0, 1.01, 1.0), f, t,
                            x / 10, x, rng.uniform(0, 0.02, m), rng.uniform(0.1, 0.5, m),
                            rng.uniform(0.97, 1.03, m) if taps else None)


GRIDS = {
    "meshed": lambda: _meshed(30, 1, False),
    "meshed_taps": lambda: _meshed(30, 2, True),
    "tree_no_pq": lambda: random_tree_grid(40, 3)[0],
    "tree": lambda: random_tree_grid(14, 4, lossless=False, all_pv=False)[0],
    "spurs": lambda: gridgen.make_grid(700, 940, 9, spur_frac=0.1, load_scale=0.03),
}


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("tile,tail", [(2, 248), (2, -1), (4, 20), (16, 64)])
@pytest.mark.parametrize("name", list(GRIDS))
def test_reduced_inner_solve(name, tile, tail, precision):
    import paper_1803_03290_gb300 as G
    g = GRIDS[name]()
    th, V, _, st, _ = pf.base_case(g, tol=1e-12, max_outer=200)
    assert st == pf.STATUS_OK
    outages = np.arange(g.n_branch) if g.n_branch < 200 else \
        np.random.default_rng(1).permutation(g.n_branch)[:101]
    ref = screen.n1_screen(g, th, V, outages, tol=1e-11, max_outer=200, processes=1)
    keys = ("theta", "V", "flow", "status", "iters")
    with G.GPCG(g, tol=1e-10, tile=tile, tail_rows=tail, precision=precision,
                max_outer=200) as c:
        c.base_solve()
        got = c.n1_screen(outages, outputs=keys)
        c.set_options(precond=G.PRECOND_IC0)  # the general PCG
        c.base_solve()
        pcg = c.n1_screen(outages, outputs=keys)
    rst = np.asarray(ref["status"])
    np.testing.assert_array_equal(got["status"], rst)
    np.testing.assert_array_equal(pcg["status"], rst)
    ok = (rst == 0) | (rst == 3)
    assert ok.sum() >= 6
    # states at a mismatch of 1e-10 p.u.: the bound of the other parity tests
    for k in ("theta", "V"):
        assert np.abs(got[k][ok] - np.asarray(ref[k])[ok]).max() < 1e-6
        assert np.abs(got[k][ok] - pcg[k][ok]).max() < 1e-6
    # two vectors span the Krylov space: no more than two iterations a solve
    # (a third where rounding leaves one)
    it = got["iters"][ok]
    assert (it[:, 1] <= 3 * it[:, 0]).all() and (it[:, 2] <= 3 * it[:, 0]).all()
