"""The autotuner and wide launches: what is probed, kept and reported is the
launch that the call takes, on both sides of the rule within one power of two of
the scenario count, and a context that was tuned for a short list has kept nothing
that a long one would take over."""
import numpy as np
import pytest

import paper_1803_03290_gb300 as gp
from gpu_common import grid

pytestmark = pytest.mark.gpu


def test_knobs_of_the_launch():
    g = grid("grid2k")
    keys = ("theta", "V", "status")
    with gp.GPCG(g, tol=1e-10, max_outer=100) as c, \
            gp.GPCG(g, tol=1e-10, max_outer=100, tile=2) as narrow:
        c.base_solve()
        narrow.base_solve()
        sms = c.info()["num_sms"]
        out = np.random.default_rng(4).integers(0, g.n_branch, 8 * sms + 2).astype(np.int32)
        ref = narrow.n1_screen(out, outputs=keys)
        ok = ref["status"] == 0
        most = None
        # (count, tiles per SM of the launch: CTAs of 1,024 and 512 threads)
        for s, per_sm in ((64, 1), (2 * sms, 1), (8 * sms, 2), (8 * sms + 2, None), (64, 1),
                          (8 * sms, 2), (8 * sms + 1, None)):
            got = c.n1_screen(out[:s], outputs=keys)
            i = c.info()
            assert i["tuned"] in (1, 2)
            if per_sm:
                assert i["tile"] == 2 and i["ctas_per_sm"] == per_sm, s
            elif most:  # tuned once, then taken from the cache
                assert (i["tile"], i["ctas_per_sm"]) == most and i["tuned"] == 2
            else:
                most = (i["tile"], i["ctas_per_sm"])
                assert most[0] in (2, 4, 8) and most[1] >= 1
            np.testing.assert_array_equal(got["status"], ref["status"][:s])
            for k in ("theta", "V"):
                assert np.abs(got[k] - ref[k][:s])[ok[:s]].max() < 1e-6
