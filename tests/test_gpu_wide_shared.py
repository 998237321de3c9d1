"""Wide launches at the sizes where the solves' vector just fits the CTA's shared
memory or just does not (FP64: 12,789 rows beside the kernel's own arrays of 27.8
KB), against the narrow launch of the same outages."""
import numpy as np
import pytest

import gridgen
import paper_1803_03290_gb300 as gp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,n_bus", [(2, n) for n in (
    5600, 5700, 6500, 12780, 12789, 12790, 12800, 12801, 14530)] + [(1, 27000), (1, 29100)])
def test_vector_at_the_edge_of_shared_memory(n_bus, precision):
    g = gridgen.make_grid(n_bus, int(1.4 * n_bus), 4, load_scale=0.3 * (120.0 / n_bus) ** 0.5)
    keys = ("theta", "V", "flow", "status", "iters", "n_overload")
    out = np.random.default_rng(1).permutation(g.n_branch)[:400].astype(np.int32)
    tol = 1e-10
    with gp.GPCG(g, tol=tol, precision=precision) as wide, \
            gp.GPCG(g, tol=tol, precision=precision, tile=2) as narrow:
        wide.base_solve()
        narrow.base_solve()
        # one scenario a tile, two a tile, 512 threads
        for s in (3, 200, 400):
            got = wide.n1_screen(out[:s], outputs=keys)
            ref = narrow.n1_screen(out[:s], outputs=keys)
            np.testing.assert_array_equal(got["status"], ref["status"])
            ok = np.isin(ref["status"], (0, 3))
            assert ok.mean() > 0.9
            for k in ("theta", "V", "flow"):  # the bound of the other wide-launch tests
                assert np.abs(got[k] - ref[k])[ok].max() < 1e-6
