"""Workloads of the N-1 contingency screen, each one call through the public
Python API on a seeded synthetic grid.

Grids are the named configurations of `gridgen` (120, 2,000, 10,000 and
50,000 buses) or, for drawn cases, random grids of the same recipe.  The seed
draws the operating point (every load within 3 % of its nominal value, the
generation following), the order of the contingency list and which of its
entries are taken; the topology belongs to the case.

Two kinds of result are asked for, as callers do:

* the state of every scenario (angles, voltages, flows, loading), from solves
  to 1e-10 p.u. with FP32 inner solves, or with FP64 inner solves at the
  default tolerance;
* the verdict alone (status, number and bit mask of overloaded branches), from
  the default options (1e-4 p.u., FP32 inner solves).

Iteration counts are returned with FP64 inner solves only: with FP32 ones they
depend on the rounding of the inner solve, that is, on which of its equivalent
kernel shapes the autotuner picks (0.2 % of them at 1e-4 p.u., 2 to 6 % at
1e-10 p.u.).
"""
import numpy as np
import torch

import paper_1803_03290_gb300 as gpcg
from gridgen import CONFIGS, make_grid

DEVICE = "cuda"


# --------------------------------------------------------------------- cases
def listed():
    """The work of a day with the screen, small to large.

    `grid`: a configuration of gridgen; `outages`: entries of the contingency
    list (0: all); `load`: the loads over the configuration's; `skip`: the
    share of the branches, the most heavily loaded ones, that is left out of
    the contingency list (corridors whose loss has no solution nearby and is
    studied by other means).
    """
    return [
        # the base-case power flow of the full-size grid from a flat start:
        # what every new operating point begins with
        dict(name="base_10k", kind="base", grid="grid10k", load=1.0),
        # a distribution-size grid screened in a control loop: host arrays in
        # and out, every result of the call
        dict(name="screen_120", kind="screen", grid="grid120", load=0.6, outages=0, skip=0.0,
             tol=1e-10, precision="fp32", results="state", memory="host"),
        # a short watch list on a regional grid, far fewer scenarios than the
        # GPU has lanes: latency of one scenario
        dict(name="watch_2k", kind="screen", grid="grid2k", load=0.6, outages=97, skip=0.0,
             tol=1e-10, precision="fp32", results="state", memory="device"),
        # every outage of a regional grid with transformers
        dict(name="xfmr_2k", kind="screen", grid="grid2k", load=0.6, outages=0, skip=0.0,
             tol=1e-10, precision="fp32", results="state", memory="device", xfmr=0.1),
        # the regional grid with reactive limits on its generators
        dict(name="limits_2k", kind="screen", grid="grid2k", load=0.6, outages=0, skip=0.0,
             tol=1e-4, precision="fp32", results="verdict", memory="device", limits=True),
        # the security check of the full-size grid with the default options:
        # which outages overload which branches
        dict(name="verdict_10k", kind="screen", grid="grid10k", load=1.0, outages=0, skip=0.0,
             tol=1e-4, precision="fp32", results="verdict", memory="device"),
        # part of the list solved tightly for planning, full states
        dict(name="tight_10k", kind="screen", grid="grid10k", load=1.0, outages=3001, skip=0.02,
             tol=1e-10, precision="fp32", results="state", memory="device"),
        # every outage with FP64 inner solves, full states
        dict(name="fp64_10k", kind="screen", grid="grid10k", load=1.0, outages=0, skip=0.0,
             tol=1e-4, precision="fp64", results="state", memory="device"),
        # a chunk of the largest grid's list
        dict(name="verdict_50k", kind="screen", grid="grid50k", load=1.0, outages=2047, skip=0.0,
             tol=1e-4, precision="fp32", results="verdict", memory="device"),
        # the loss of every generator, solved tightly
        dict(name="gens_10k", kind="gens", grid="grid10k", load=1.0, outages=0, tol=1e-10,
             max_outer=100),
        # the DC quick screen, full angles and flows, for new injections
        dict(name="dc_10k", kind="dc", grid="grid10k", load=1.0, outages=0),
        # loss and gradients of the overload penalty, one training step's call
        dict(name="adjoint_2k", kind="adjoint", grid="grid2k", load=1.0, outages=0),
    ]


def draw(rng):
    """One more case of these ranges: grid sizes between the smallest and the
    full-size configuration, lists from a few outages to all of them."""
    kind = rng.choice(["base", "state", "state", "fp64", "verdict", "verdict", "limits", "gens",
                       "dc", "adjoint"])
    top = 2000 if kind in ("limits", "adjoint") else 10000
    n = int(round(120 * (top / 120) ** rng.random()))
    m = int(n * rng.uniform(1.3, 1.5))
    c = dict(kind="screen", grid="random", n_bus=n, n_branch=m, topology=rng.randrange(1 << 30),
             spurs=rng.choice([0.0, 0.05]), load=rng.uniform(0.35, 0.5),
             outages=int(round(5 * (m / 5) ** rng.uniform(0.3, 1.0))))
    if kind in ("base", "dc", "adjoint"):
        c["kind"] = kind
        return c
    if kind == "gens":
        c.update(kind="gens", tol=1e-10, max_outer=100, outages=max(1, min(c["outages"], n // 6)))
        return c
    c.update(skip=0.05, tol=1e-4, precision="fp32", results="verdict",
             memory=rng.choice(["device", "device", "host"]))
    if kind == "limits":
        c["limits"] = True
    elif kind == "state":
        c.update(tol=1e-10, results="state", xfmr=rng.choice([0.0, 0.1]),
                 outages=min(c["outages"], 3001))
    elif kind == "fp64":
        c.update(precision="fp64", results="state")
    c["outages"] = min(c["outages"], int(0.95 * m) - 1)
    return c


# -------------------------------------------------------------------- inputs
def _grid(case, seed, attempt=0):
    """The case's grid at the seed's operating point (attempt: the how manieth
    random topology)."""
    more = dict(xfmr_frac=case.get("xfmr", 0.0))
    if case["grid"] == "random":
        n = case["n_bus"]
        # the loading falls with the size as it does over the configurations
        g = make_grid(n, case["n_branch"], case["topology"] + attempt, spur_frac=case["spurs"],
                      load_scale=0.3 * (120.0 / n) ** 0.4, **more)
    else:
        g = make_grid(**CONFIGS[case["grid"]], **more)
    rng = np.random.default_rng(seed)
    u = case["load"] * rng.uniform(0.97, 1.03, g.n_bus)
    load = (g.P_gen - g.P_sched) * u
    g.P_gen = g.P_gen * (load.sum() / g.P_gen.sum())
    g.P_sched = g.P_gen - load
    g.Q_sched = g.Q_sched * u
    # ratings near the flows of this loading, so that some branches exceed them
    g.rating = g.rating * 0.4 * case["load"]
    return g, rng


def _limits(g, base):
    """Reactive limits around each generator's output in the base case."""
    v = base["V"] * np.exp(1j * base["theta"])
    y = 1.0 / (g.r + 1j * g.x)
    ysh = y + 0.5j * g.b_sh
    i = np.zeros(g.n_bus, dtype=complex)
    np.add.at(i, g.f, ysh * v[g.f] - y * v[g.t])
    np.add.at(i, g.t, ysh * v[g.t] - y * v[g.f])
    q = (v * i.conj()).imag - g.Q_sched
    g = g.copy()
    g.Q_max = q + 0.05 + 0.1 * np.abs(q)
    g.Q_min = q - 0.05 - 0.1 * np.abs(q)
    return g


def _solver(case, seed):
    """The grid, its solver with the base case solved, the contingency list.
    A random topology whose base case has no solution from a flat start is
    passed over."""
    for attempt in range(8 if case["grid"] == "random" else 1):
        try:
            return _try_solver(case, seed, attempt)
        except gpcg.GPCGError as e:
            error = e
    raise error


def _try_solver(case, seed, attempt):
    g, rng = _grid(case, seed, attempt)
    options = {k: case[k] for k in ("tol", "max_outer") if k in case}
    if case["kind"] == "dc" or case.get("precision") == "fp64":
        options["precision"] = gpcg.BATCHED_FP64
    solver = gpcg.GPCG(g, **options)
    base = None
    if case["kind"] in ("screen", "gens") or case["grid"] == "random":
        base = solver.base_solve()
    if case.get("limits"):
        solver.close()
        g = _limits(g, base)
        solver = gpcg.GPCG(g, **options)
        base = solver.base_solve()
    if case["kind"] == "gens":
        names = np.flatnonzero(g.bus_type == 1)
    else:
        names = np.arange(g.n_branch)
        skip = int(round(case.get("skip", 0.0) * g.n_branch))
        if skip:
            names = np.argsort(np.abs(base["flow"]), kind="stable")[:g.n_branch - skip]
    names = rng.permutation(names).astype(np.int32)
    if case.get("outages"):
        names = names[:case["outages"]]
    return g, solver, names


def _results(case):
    if case["kind"] == "gens":
        return ("theta", "V", "flow", "status", "max_loading", "n_overload")
    if case["results"] == "verdict":
        return ("status", "n_overload", "overload")
    keys = ("theta", "V", "flow", "label", "status", "max_loading", "n_overload")
    return keys + ("iters",) if case["precision"] == "fp64" else keys


def prepare(case, seed):
    g, solver, names = _solver(case, seed)
    state = dict(kind=case["kind"], solver=solver)
    if case["kind"] == "base":
        return state
    n, m, s = g.n_bus, g.n_branch, len(names)
    host = case.get("memory") == "host"
    state["memory"] = "host" if host else "device"
    state["outages"] = names if host else torch.from_numpy(names).to(DEVICE)
    f64 = dict(dtype=torch.float64, device=DEVICE)
    if case["kind"] in ("dc", "adjoint"):
        state["P"] = torch.from_numpy(g.P_sched).to(DEVICE)
    if case["kind"] == "adjoint":
        state["b"] = torch.from_numpy(1.0 / g.x).to(DEVICE)
        state["out"] = dict(loss=torch.zeros(1, **f64), dP=torch.zeros(n, **f64),
                            db=torch.zeros(m, **f64))
        return state
    i32 = dict(dtype=torch.int32, device=DEVICE)
    make = dict(theta=lambda: torch.zeros((s, n), **f64), V=lambda: torch.zeros((s, n), **f64),
                flow=lambda: torch.zeros((s, m), **f64),
                max_loading=lambda: torch.zeros(s, **f64),
                label=lambda: torch.zeros((s, n), **i32), iters=lambda: torch.zeros((s, 3), **i32),
                status=lambda: torch.zeros(s, **i32), n_overload=lambda: torch.zeros(s, **i32),
                overload=lambda: torch.zeros((s, gpcg.mask_words(m)), **i32))
    keys = (("theta", "flow", "status", "max_loading", "n_overload") if case["kind"] == "dc"
            else _results(case))
    state["results"] = keys
    if not host:
        state["out"] = {k: make[k]() for k in keys}
    return state


# ----------------------------------------------------------------- the calls
def run(state):
    solver, kind = state["solver"], state["kind"]
    if kind == "base":
        r = solver.base_solve()
        return {k: r[k] for k in ("theta", "V", "flow", "iters")}
    if state["memory"] == "host":
        return solver.n1_screen(state["outages"], outputs=state["results"])
    out = state["out"]
    if kind == "screen":
        solver.n1_screen_device(state["outages"], out)
    elif kind == "gens":
        solver.n1_gen_screen_device(state["outages"], out)
    elif kind == "dc":
        solver.n1_dc_screen_device(state["outages"], out, P=state["P"])
    else:
        solver.n1_adjoint_device(state["outages"], state["P"], state["b"], out["loss"], out["dP"],
                                 out["db"])
    return out


def work(case):
    """Bytes of the grid and the outputs, and the arithmetic of the method:
    per scenario and half-step one mismatch evaluation (8 flops per branch end
    and about 30 per bus) and one pair of triangular solves with a factor of
    about three entries a row; half-step pairs as the tolerance needs them."""
    if case["grid"] == "random":
        n, m = case["n_bus"], case["n_branch"]
    else:
        n, m = CONFIGS[case["grid"]]["n_bus"], CONFIGS[case["grid"]]["n_branch"]
    kind = case["kind"]
    s = case.get("outages") or (n // 5 - 1 if kind == "gens" else m)
    grid = 41 * n + 48 * m
    solve, mismatch = 12 * n, 16 * m + 30 * n
    if kind == "base":
        return dict(bytes=grid + 16 * n + 8 * m, flops=18 * 2 * (solve + mismatch))
    if kind == "dc":
        return dict(bytes=grid + s * (16 + 8 * n + 8 * m + 4), flops=s * (2 * solve + 4 * m))
    if kind == "adjoint":
        return dict(bytes=grid + 4 * s + 8 * (1 + n + m), flops=s * (4 * solve + 60 * m))
    pairs = 2.4 if case["tol"] == 1e-4 else 8.0
    if kind == "screen" and case["results"] == "verdict":
        out = 8 + 4 * ((m + 31) // 32)
    else:
        out = 16 * n + 8 * m + 16 + (4 * n if kind == "screen" else 0)
    return dict(bytes=grid + s * (4 + out), flops=s * (pairs * 2 * (solve + mismatch) + 20 * m))


# ------------------------------------------------- the same in plain 64 bits
def _islands(g):
    """Per branch the buses its outage cuts off from the slack (bridges only):
    depth-first preorder, and [lo, hi) of the preorder per bridge."""
    n, m = g.n_bus, g.n_branch
    adj = [[] for _ in range(n)]
    for k in range(m):
        adj[int(g.f[k])].append((int(g.t[k]), k))
        adj[int(g.t[k])].append((int(g.f[k]), k))
    pre, low, size = [-1] * n, [0] * n, [1] * n
    lo, hi = np.zeros(m, dtype=np.int64), np.zeros(m, dtype=np.int64)
    root = int(np.flatnonzero(g.bus_type == 2)[0])
    pre[root] = low[root] = 0
    count, stack = 1, [(root, -1, iter(adj[root]))]
    while stack:
        u, via, it = stack[-1]
        for v, k in it:
            if k == via:
                continue
            if pre[v] < 0:
                pre[v] = low[v] = count
                count += 1
                stack.append((v, k, iter(adj[v])))
                break
            low[u] = min(low[u], pre[v])
        else:
            stack.pop()
            if stack:
                p = stack[-1][0]
                low[p] = min(low[p], low[u])
                size[p] += size[u]
                if low[u] > pre[p]:
                    lo[via], hi[via] = pre[u], pre[u] + size[u]
    return np.array(pre), lo, hi


class _Dense:
    """Dense 64-bit tensors of a grid and of an outage list."""

    def __init__(self, g, names):
        def t(a, kind=torch.float64):
            return torch.as_tensor(np.asarray(a), dtype=kind, device=DEVICE)
        self.n, self.m = g.n_bus, g.n_branch
        n, m = self.n, self.m
        self.f, self.t = t(g.f, torch.int64), t(g.t, torch.int64)
        self.x, self.rating = t(g.x), t(g.rating)
        d = t(g.r) ** 2 + self.x ** 2
        self.g, self.b, self.bsh = t(g.r) / d, -self.x / d, t(g.b_sh)
        self.c = torch.ones(m, dtype=torch.float64, device=DEVICE) if g.tap is None else 1 / t(g.tap)
        self.type = t(g.bus_type, torch.int64)
        self.P, self.Q, self.Vset = t(g.P_sched), t(g.Q_sched), t(g.V_set)
        self.pg = torch.where((self.type == 1) & (t(g.P_gen) > 0), t(g.P_gen), 0.0)
        self.out = t(names, torch.int64)
        pre, lo, hi = _islands(g)
        pre, lo, hi = t(pre, torch.int64), t(lo, torch.int64)[self.out], t(hi, torch.int64)[self.out]
        self.main = ~((pre >= lo[:, None]) & (pre < hi[:, None]))  # [S, n]
        self.bridge = hi > lo
        # the island's injection goes to the main island's generators in
        # proportion to theirs (with none there the slack takes it)
        pg = (self.main * self.pg).sum(1)
        self.share = torch.where(self.bridge & (pg > 0), 1 / pg.clamp_min(1e-300), 0.0)
        self.coef = self.share * ((~self.main) * self.P).sum(1)

    def matrix(self, w, c, keep):
        """Sum of w v v^T, v = c e_from - e_to, the identity off `keep`."""
        a = torch.zeros((self.n, self.n), dtype=torch.float64, device=DEVICE)
        for i, j, v in ((self.f, self.f, w * c * c), (self.t, self.t, w), (self.f, self.t, -w * c),
                        (self.t, self.f, -w * c)):
            a = a.index_put((i, j), v, accumulate=True)
        k = keep.to(torch.float64)
        return a * k[:, None] * k[None, :] + torch.diag(1 - k)


def _inverse(a):
    """Inverse of a positive definite matrix, by blocks."""
    n = len(a)
    if n <= 256:
        return torch.from_numpy(np.linalg.inv(a.cpu().numpy())).to(a.device)
    h = n // 2
    p = _inverse(a[:h, :h])
    pb = p @ a[:h, h:]
    q = _inverse(a[h:, h:] - a[h:, :h] @ pb)
    pbq = pb @ q
    return torch.cat([torch.cat([p + pbq @ pb.T, -pbq], 1), torch.cat([-pbq.T, q], 1)])


def _corrected(inv, rhs, w, c, keep, d):
    """B_s^-1 rhs per scenario on the main island: the base inverse and the
    outaged branch's rank-one term, the island's end of a bridge left out of
    the column that corrects."""
    k = keep.to(torch.float64)
    x = rhs @ inv
    fo, to, wo, co = d.f[d.out], d.t[d.out], w[d.out], c[d.out]
    at = torch.arange(len(fo), device=DEVICE)
    mf, mt = k[fo] * d.main[at, fo], k[to] * d.main[at, to]
    col = (co * mf)[:, None] * inv[fo] - mt[:, None] * inv[to]
    vx = co * x[at, fo] * k[fo] - x[at, to] * k[to]
    vy = co * col[at, fo] * k[fo] - col[at, to] * k[to]
    return (x + (wo * vx / (1 - wo * vy))[:, None] * col) * (d.main & keep)


def _flows(d, th, v, lines):
    z = v[:, d.f] * v[:, d.t] * d.c
    a = th[:, d.f] - th[:, d.t]
    pf = d.g * d.c ** 2 * v[:, d.f] ** 2 - z * (d.g * torch.cos(a) + d.b * torch.sin(a))
    pt = d.g * v[:, d.t] ** 2 - z * (d.g * torch.cos(a) - d.b * torch.sin(a))
    return pf * lines, torch.maximum(pf.abs(), pt.abs()) * lines / d.rating


def _newton_like(d, base_only):
    """The fast-decoupled iteration to rounding: (theta, V) of the base case
    from a flat start, or of every scenario from there."""
    n, dev = d.n, dict(dtype=torch.float64, device=DEVICE)
    w1, w2, one = 1 / d.x, -d.b, torch.ones(d.m, **dev)
    keep_p, keep_q = d.type != 2, d.type == 0
    inv1, inv2 = _inverse(d.matrix(w1, one, keep_p)), _inverse(d.matrix(w2, d.c, keep_q))
    i = torch.cat([d.f, d.t, d.f, d.t])
    j = torch.cat([d.t, d.f, d.f, d.t])
    yg = torch.cat([-d.c * d.g, -d.c * d.g, d.c ** 2 * d.g, d.g])
    yb = torch.cat([-d.c * d.b, -d.c * d.b, d.c ** 2 * (d.b + d.bsh / 2), d.b + d.bsh / 2])
    ge, be = (torch.sparse_coo_tensor(torch.stack([i, j]), v, (n, n)).coalesce() for v in (yg, yb))

    def mismatch(th, v, out, p):
        e, f = v * torch.cos(th), v * torch.sin(th)
        re = (ge @ e.T - be @ f.T).T.contiguous()
        im = (ge @ f.T + be @ e.T).T.contiguous()
        if out is not None:  # the outaged branch's currents back out
            at = torch.arange(len(out), device=DEVICE)
            fo, to, c, g, b, sh = d.f[out], d.t[out], d.c[out], d.g[out], d.b[out], d.bsh[out]
            vf, vt = torch.complex(e[at, fo], f[at, fo]), torch.complex(e[at, to], f[at, to])
            y = torch.complex(g, b)
            ys = torch.complex(g, b + sh / 2)
            for bus, cur in ((fo, c * c * ys * vf - c * y * vt), (to, ys * vt - c * y * vf)):
                re[at, bus] -= cur.real
                im[at, bus] -= cur.imag
        return p - (e * re + f * im), d.Q - (f * re - e * im)

    th, v, out, p = torch.zeros((1, n), **dev), d.Vset[None, :].clone(), None, d.P[None, :]
    main = torch.ones((1, n), dtype=torch.bool, device=DEVICE)

    def loop(th, v, solve1, solve2, out, p, main, cap):
        best, since = 1e30, 0
        for _ in range(cap):
            dp, _ = mismatch(th, v, out, p)
            th = th + solve1(torch.where(main & keep_p, dp / v.clamp_min(1e-3), 0.0))
            dp, dq = mismatch(th, v, out, p)
            err = max(float((dp * (main & keep_p)).abs().max()),
                      float((dq * (main & keep_q)).abs().max()))
            if err < best:
                best, since = err, 0
            since += 1
            if since > 6:  # at the rounding of the mismatch
                break
            v = v + solve2(torch.where(main & keep_q, dq / v.clamp_min(1e-3), 0.0))
        return (th, v) if best < 1e-11 else None

    got = loop(th, v, lambda r: r @ inv1, lambda r: r @ inv2, out, p, main, 120)
    if got is None or base_only:
        return got
    th, v = (a * d.main for a in got)
    p = d.P + d.coef[:, None] * d.pg
    return loop(th, v, lambda r: _corrected(inv1, r, w1, one, keep_p, d),
                lambda r: _corrected(inv2, r, w2, d.c, keep_q, d), d.out, p, d.main, 80)


def _in_service(d):
    lines = d.main[:, d.f] & d.main[:, d.t]
    lines[torch.arange(len(d.out), device=DEVICE), d.out] = False
    return lines


def exact(case, seed):
    kind = case["kind"]
    if kind == "gens" or case.get("results") == "verdict":
        return None
    if kind == "screen" and (case.get("limits") or case["grid"] in ("grid10k", "grid50k")
                             or case.get("n_bus", 0) > 4000 or case["tol"] > 1e-9):
        return None
    g, solver, names = _solver(case, seed)
    solver.close()
    if kind == "base":
        d = _Dense(g, np.zeros(1, dtype=np.int32))
        got = _newton_like(d, True)
        if got is None:
            return None
        th, v = got
        pf, _ = _flows(d, th, v, torch.ones((1, d.m), dtype=torch.bool, device=DEVICE))
        return dict(theta=th[0], V=v[0], flow=pf[0], iters=None)
    d = _Dense(g, names)
    if kind == "screen":
        got = _newton_like(d, False)
        if got is None:
            return None
        th, v = got
        pf, load = _flows(d, th, v, _in_service(d))
        return dict(theta=th, V=v, flow=pf, label=None, status=None, max_loading=load.amax(1),
                    n_overload=None)
    keep = d.type != 2
    one = torch.ones(d.m, dtype=torch.float64, device=DEVICE)
    if kind == "dc":
        w = 1 / d.x
        p = (d.P + d.coef[:, None] * d.pg) * (d.main & keep)
        th = _corrected(_inverse(d.matrix(w, one, keep)), p, w, one, keep, d)
        fl = w * (th[:, d.f] - th[:, d.t]) * _in_service(d)
        return dict(theta=th, flow=fl, status=None, max_loading=(fl.abs() / d.rating).amax(1),
                    n_overload=None)
    # the penalty as a differentiable function of the injections and the
    # susceptances; the shares of the re-dispatch are constants
    P = d.P.clone().requires_grad_(True)
    b = (1 / d.x).requires_grad_(True)
    p = (P + (d.share * ((~d.main) * P).sum(1))[:, None] * d.pg) * (d.main & keep)
    B = d.matrix(b, one, keep)
    inv = _inverse(B.detach())
    # the inverse and, through this Newton step, its derivative
    th = _corrected(2 * inv - inv @ B @ inv, p, b, one, keep, d)
    fl = b * (th[:, d.f] - th[:, d.t])
    pen = torch.nn.functional.softplus(fl.abs() / d.rating - 1, threshold=1e9) ** 2
    loss = (pen * _in_service(d)).sum()
    loss.backward()
    return dict(loss=loss.detach().reshape(1), dP=P.grad, db=b.grad)
