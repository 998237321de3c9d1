"""A call that failed for want of memory leaves nothing behind that the next call
would report: a screen whose work buffer exceeds the device, then a small one, a
new context, and the screen without allocations."""
import numpy as np
import pytest

import paper_1803_03290_gb300 as gp
from gpu_common import grid

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("then", ["screen", "create", "noalloc"])
def test_call_after_out_of_memory(then):
    import torch
    g = grid("grid50k")
    out = np.arange(5, dtype=np.int32)
    knobs = dict(ctas_per_sm=64, tail_rows=64)
    with gp.GPCG(g, tile=32, **knobs) as c, gp.GPCG(g, tile=2, **knobs) as small:
        c.base_solve()
        small.base_solve()
        want = c.n1_screen(out, outputs=("status",))["status"]
        # 83 MB for a slot of 32 scenarios: 0.8 TB in one allocation, which the runtime
        # refuses as a whole
        many = np.zeros(32 * 64 * c.info()["num_sms"], np.int32)
        with pytest.raises(gp.GPCGError, match="(?i)memory"):
            c.n1_screen(many, outputs=("status",))
        if then == "screen":
            got = c.n1_screen(out, outputs=("status",))["status"]
        elif then == "create":
            with gp.GPCG(g) as d:
                d.base_solve()
                got = d.n1_screen(out, outputs=("status",))["status"]
        else:
            st = torch.zeros(5, dtype=torch.int32, device="cuda")
            small.n1_screen_noalloc_device(torch.from_numpy(out).cuda(), dict(status=st))
            torch.cuda.synchronize()
            got = st.cpu().numpy()
    np.testing.assert_array_equal(got, want)
