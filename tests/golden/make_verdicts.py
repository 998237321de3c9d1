"""Record verdicts of the default screen (FP32 inner solves, 1e-4 p.u.) as the
general PCG computes them (test fixture).

Per workload every outage is screened once; the file keeps the scenarios that do
not converge, which amplify any rounding, and a sample of the others: status,
iterations, overload count, digest of the overload mask and the bits of the
maximum loading.  Run on a GPU:

    python tests/golden/make_verdicts.py [ROOT]

with the library built under ROOT (default: this repository).  The fixture was
recorded from commit 394ccb4, before the reduced inner solves, with the barrier
between clearing and setting mask bits made uniform.
"""
import hashlib
import json
import os
import sys

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
FILE = os.path.join(HERE, "verdicts.json")
# workload, sampled outages, (tile, tail_rows) of each recording
CASES = [("grid2k_limits", 60, [(2, 248), (8, 64)]), ("grid10k", 60, [(2, 248), (4, 64)]),
         ("grid50k", 20, [(2, 248), (2, 64)])]


def workload(name, gp):
    """The grid, its ratings near the flows of its loading."""
    from gridgen import config_grid
    g = config_grid(name.split("_")[0]).copy()
    g.rating = g.rating * 0.4
    if name.endswith("_limits"):
        with gp.GPCG(g) as c:
            b = c.base_solve()
        v = b["V"] * np.exp(1j * b["theta"])
        y = 1.0 / (g.r + 1j * g.x)
        ysh = y + 0.5j * g.b_sh
        i = np.zeros(g.n_bus, dtype=complex)
        np.add.at(i, g.f, ysh * v[g.f] - y * v[g.t])
        np.add.at(i, g.t, ysh * v[g.t] - y * v[g.f])
        q = (v * i.conj()).imag - g.Q_sched
        # (rounded: the limits are the same for a base case that differs in its last bits)
        g.Q_max = np.round(q + 0.03 + 0.1 * np.abs(q), 6)
        g.Q_min = np.round(q - 0.03 - 0.1 * np.abs(q), 6)
    return g


def verdicts(gp, g, outages, tile, tail):
    """One row per outage: status, outer and inner iterations, overloaded
    branches, mask digest, maximum loading."""
    keys = ("status", "iters", "n_overload", "overload", "max_loading")
    with gp.GPCG(g, tile=tile, tail_rows=tail) as c:
        c.base_solve()
        r = c.n1_screen(np.asarray(outages, np.int32), outputs=keys)
    return [[int(r["status"][s]), *(int(v) for v in r["iters"][s]), int(r["n_overload"][s]),
             hashlib.sha256(r["overload"][s].tobytes()).hexdigest()[:16],
             float(r["max_loading"][s]).hex()] for s in range(len(outages))]


def main(root):
    sys.path.insert(0, os.path.abspath(root))
    import paper_1803_03290_gb300 as gp
    out = []
    for name, sample, knobs in CASES:
        g = workload(name, gp)
        with gp.GPCG(g, tile=2, tail_rows=248) as c:
            c.base_solve()
            st = c.n1_screen(np.arange(g.n_branch), outputs=("status",))["status"]
        bad = np.flatnonzero((st != 0) & (st != 3))
        rest = np.random.default_rng(8).permutation(np.setdiff1d(np.arange(g.n_branch), bad))
        names = [int(k) for k in np.concatenate([bad, rest[:sample]])]
        out.append(dict(workload=name, outages=names,
                        runs=[dict(tile=t, tail_rows=r, rows=verdicts(gp, g, names, t, r))
                              for t, r in knobs]))
        print(name, len(bad), "not converged of", g.n_branch)
    with open(FILE, "w") as fh:
        json.dump(out, fh, separators=(",", ":"))
        fh.write("\n")


if __name__ == "__main__":
    main(sys.argv[1] if len(sys.argv) > 1 else os.path.dirname(os.path.dirname(HERE)))
