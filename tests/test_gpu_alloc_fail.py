"""Every device allocation of gpcg_create and of the adjoint's first call fails
once, by a fake of cudaMalloc linked into a copy of the library: the call reports
GPCG_ERR_OOM and leaks nothing, or, where the allocation belonged to the columns
of the reduced inner solves, succeeds without them and the screens take the
PCG."""
import json
import os
import subprocess
import sys

import pytest

from paper_1803_03290_gb300 import _build

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
SCRIPT = r"""
import json, sys
import numpy as np
sys.path.insert(0, sys.argv[1])
from paper_1803_03290_gb300 import _build, binding
_build.LIB, _build.up_to_date = sys.argv[2], lambda: True
import paper_1803_03290_gb300 as gp
import gridgen
g = gridgen.make_grid(300, 420, 11, spur_frac=0.05, load_scale=0.03)
lib = binding.load()
out = np.arange(0, g.n_branch, 37, dtype=np.int32)
pv = np.flatnonzero(g.bus_type == 1)[:5]
o = dict(tol=1e-10, max_outer=100, precision=gp.BATCHED_FP64, tile=2)

def results(c):
    c.base_solve()
    a, b = c.n1_screen(out, outputs=("theta", "status")), c.n1_gen_screen(pv, outputs=("V", "status"))
    return a["theta"], a["status"], b["V"], b["status"], c.n1_adjoint(out)[2]

lib.fake_arm(-1)
with gp.GPCG(g, **o) as c:
    n_create = lib.fake_count()
    want = results(c)
made, refused, off, leaks = [], [], 0.0, 0
for k in range(n_create):
    lib.fake_arm(k)
    try:
        c = gp.GPCG(g, **o)
    except gp.GPCGError as e:
        assert "OOM" in str(e) or "memory" in str(e), e
        refused.append(k)
    else:
        lib.fake_arm(-1)
        got = results(c)
        c.close()
        off = max([off] + [float(np.abs(x - y).max()) for x, y in zip(got, want)])
        made.append(k)
    leaks = max(leaks, abs(lib.fake_live()))
adj = []
with gp.GPCG(g, **o) as c:
    lib.fake_arm(-1)
    c.n1_adjoint(out)
    n_adj = lib.fake_count()
for k in range(n_adj):
    with gp.GPCG(g, **o) as c:
        lib.fake_arm(k)
        try:
            c.n1_adjoint(out)
            adj.append(k)
        except gp.GPCGError as e:
            assert "OOM" in str(e) or "memory" in str(e), e
        lib.fake_arm(-1)
        off = max(off, float(np.abs(c.n1_adjoint(out)[2] - want[4]).max()))
    leaks = max(leaks, abs(lib.fake_live()))
print(json.dumps(dict(n_create=n_create, made=made, refused=len(refused), n_adj=n_adj, adj=adj,
                      off=off, leaks=leaks)))
"""


def test_each_allocation_fails_once(tmp_path):
    _build.build(force=not os.path.isdir(_build.BUILD))
    shim, lib = str(tmp_path / "fake.o"), str(tmp_path / "libgpcg_fake.so")
    subprocess.run(["gcc", "-O1", "-fPIC", "-c", os.path.join(HERE, "cuda", "malloc_fake.c"),
                    "-o", shim], check=True)
    objs = [os.path.join(_build.BUILD, os.path.basename(s) + ".o") for s in _build.sources()]
    subprocess.run([_build._nvcc(), *_build.ARCH, "-shared", "-cudart", "static", "-Xlinker",
                    "--wrap=cudaMalloc,--wrap=cudaFree", "-o", lib, *objs, shim], check=True)
    r = subprocess.run([sys.executable, "-c", SCRIPT, os.path.dirname(HERE), lib],
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    got = json.loads(r.stdout.splitlines()[-1])
    # six allocations of each matrix's columns, four of the PV buses'; three of the
    # adjoint's own columns
    assert len(got["made"]) == 16 and got["refused"] == got["n_create"] - 16, got
    assert len(got["adj"]) == 3, got
    # solves to 1e-10 p.u.; the adjoint's to 1e-12
    assert got["off"] < 1e-6, got
    assert got["leaks"] == 0, got
