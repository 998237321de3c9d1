"""Wide launches against really narrow ones (a context with a fixed tile never
takes a wide launch): counts at every edge of the rule -- one and two scenarios
per SM, eight per SM and one more -- both precisions, grids with fewer and more
rows than threads, overload counts, and the entry point without allocations."""
import numpy as np
import pytest

import gridgen
import paper_1803_03290_gb300 as gp

pytestmark = pytest.mark.gpu

F64 = ("theta", "V", "flow", "max_loading")
I32 = ("status", "label", "n_overload", "overload")


def _device(c, call, out, g):
    import torch
    s = len(out)
    shape = dict(flow=(s, g.n_branch), max_loading=(s,), status=(s,), n_overload=(s,),
                 overload=(s, gp.mask_words(g.n_branch)))
    dev = {k: torch.zeros(shape.get(k, (s, g.n_bus)), device="cuda",
                          dtype=torch.float64 if k in F64 else torch.int32) for k in F64 + I32}
    getattr(c, call)(torch.from_numpy(out).cuda(), dev)
    torch.cuda.synchronize()
    return {k: v.cpu().numpy().view(np.uint32 if k == "overload" else v.cpu().numpy().dtype)
            for k, v in dev.items()}


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("n_bus", [300, 700, 1500])
def test_wide_against_narrow(n_bus, precision):
    g = gridgen.make_grid(n_bus, int(1.4 * n_bus), 11, spur_frac=0.05, load_scale=0.03)
    o = dict(tol=1e-10, max_outer=100, precision=precision)
    with gp.GPCG(g, **o) as c:
        flow = np.abs(c.base_solve()["flow"])
    g.rating = np.maximum(flow * np.random.default_rng(5).uniform(0.8, 1.6, g.n_branch), 1e-3)
    with gp.GPCG(g, **o) as c, gp.GPCG(g, tile=2, tail_rows=248, **o) as narrow:
        c.base_solve()
        narrow.base_solve()
        sms = c.info()["num_sms"]
        out = np.random.default_rng(2).integers(0, g.n_branch, 8 * sms + 1).astype(np.int32)
        ref = narrow.n1_screen(out, outputs=F64 + I32)
        ok = np.isin(ref["status"], (0, 3))
        assert ok.mean() > 0.9 and (ref["n_overload"] > 0).any()
        # (loading of the from end: near enough to a tie to be left out)
        tie = np.abs(np.abs(ref["flow"]) / g.rating - 1.0) < 1e-3
        bits = gp.unpack_mask(ref["overload"], g.n_branch)
        for s in (1, 2, sms, sms + 1, 2 * sms, 2 * sms + 1, 8 * sms, 8 * sms + 1):
            got = c.n1_screen(out[:s], outputs=F64 + I32)
            for k in ("status", "label"):
                np.testing.assert_array_equal(got[k], ref[k][:s])
            # the launches differ in the rounding of the inner solve only
            for k in F64:
                d = np.abs(got[k] - ref[k][:s])[ok[:s]]
                assert d.size == 0 or d.max() < 1e-6
            mask = gp.unpack_mask(got["overload"], g.n_branch)
            use = ~tie[:s] & ok[:s, None]
            np.testing.assert_array_equal(mask[use], bits[:s][use])
            np.testing.assert_array_equal(got["n_overload"], mask.sum(1))
            # the same launch, hence the same bits, without allocations
            dev = _device(c, "n1_screen_noalloc_device", out[:s], g)
            for k in F64 + I32:
                np.testing.assert_array_equal(dev[k], got[k], err_msg=f"{k}, {s} scenarios")
