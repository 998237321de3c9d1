"""Verdicts of the screen at the default options (FP32 inner solves, 1e-4 p.u.)
against recorded ones (tests/golden/make_verdicts.py), bit for bit: which kernel
a screen takes may not decide whether a branch near its rating is overloaded, nor
where a scenario that does not converge ends."""
import json

import numpy as np
import pytest

import paper_1803_03290_gb300 as gp
from golden import make_verdicts as mv

pytestmark = pytest.mark.gpu

with open(mv.FILE) as fh:
    GOLDEN = json.load(fh)


@pytest.mark.parametrize("case", GOLDEN, ids=lambda c: c["workload"])
def test_recorded_verdicts(case):
    g = mv.workload(case["workload"], gp)
    for run in case["runs"]:
        got = mv.verdicts(gp, g, case["outages"], run["tile"], run["tail_rows"])
        bad = [(l, a, b) for l, a, b in zip(case["outages"], got, run["rows"]) if a != b]
        assert not bad, f"{len(bad)} of {len(got)} rows, first {bad[0]}"


def test_tolerance_on_a_live_context():
    """set_options moves a context over the tolerance below which FP32 screens
    take reduced inner solves, and back: host, device and scratch-array calls give
    what a fresh context gives there."""
    import torch
    g = mv.workload("grid2k", gp)
    out = np.random.default_rng(3).permutation(g.n_branch)[:301].astype(np.int32)
    keys = ("theta", "V", "flow", "status", "iters", "n_overload", "overload", "max_loading")
    knobs = dict(tile=2, ctas_per_sm=4, tail_rows=64)

    def fresh(tol):
        with gp.GPCG(g, tol=tol, **knobs) as c:
            c.base_solve()
            return c.n1_screen(out, outputs=keys)
    want = {tol: fresh(tol) for tol in (1e-4, 1e-9)}
    assert (want[1e-4]["iters"] != want[1e-9]["iters"]).any()
    dt = dict(status=torch.int32, iters=torch.int32, n_overload=torch.int32,
              overload=torch.int32)
    with gp.GPCG(g, tol=1e-4, **knobs) as c:
        c.base_solve()
        names = torch.from_numpy(out).cuda()
        for tol in (1e-4, 1e-9, 1e-4):
            c.set_options(tol=tol)
            host = c.n1_screen(out, outputs=keys)
            for call in (c.n1_screen_device, c.n1_screen_noalloc_device):
                dev = {k: torch.zeros(host[k].shape, dtype=dt.get(k, torch.float64),
                                      device="cuda") for k in keys}
                call(names, dev)
                torch.cuda.synchronize()
                for k in keys:
                    np.testing.assert_array_equal(
                        dev[k].cpu().numpy().view(want[tol][k].dtype), want[tol][k], err_msg=k)
            for k in keys:
                np.testing.assert_array_equal(host[k], want[tol][k], err_msg=k)
