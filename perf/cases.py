"""What this framework is used for, as cases to be timed: operators set up from node
sets, right-hand sides, time steps, batches and gradients, each through the package's
public calls.  Node sets, fields and time steps are drawn from a seed; every case is a
dict of plain values.

Sizes are those of the package's own workloads (the 64 x 64 order-4 and 512 x 512
order-8 Taylor-Green lattices, the 1.0M-node variable-resolution columns, the 512 x 512
channel, the Lamb-Oseen box at R_c/s = 8, the batch of 2k-64k-node instances) and of
its tests (37 x 29).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import labfm_inputs as li
import paper_2102_02019_gb300 as lb

C, MU = 10.0, 0.005  # sound speed and viscosity of the Taylor-Green runs
H_OVER_S = li.H_OVER_S
DTYPES = {"f32": torch.float32, "f64": torch.float64}
DEV = "cuda"


def listed():
    return [
        # a right-hand side for a caller's own integrator on a ragged little box: one launch
        {"name": "rhs_f64_37x29_m4", "kind": "rhs", "nodes": "lattice", "nx": 37, "ny": 29, "m": 4, "dtype": "f64"},
        # the small Taylor-Green run: a hundred short launches
        {"name": "steps_f32_64_m4", "kind": "steps", "nodes": "lattice", "nx": 64, "ny": 64, "m": 4, "dtype": "f32",
         "steps": 20},
        # the headline run
        {"name": "steps_f32_512_m8", "kind": "steps", "nodes": "lattice", "nx": 512, "ny": 512, "m": 8, "dtype": "f32",
         "steps": 4},
        # the same run in double precision, in which the method is validated
        {"name": "steps_f64_512_m8", "kind": "steps", "nodes": "lattice", "nx": 512, "ny": 512, "m": 8, "dtype": "f64",
         "steps": 1},
        # the Lamb-Oseen vortex between an inflow and an outflow, double precision as in the study
        {"name": "steps_f64_lamb_oseen_200_m6", "kind": "steps", "nodes": "open_box", "nx": 200, "ny": 200, "m": 6,
         "dtype": "f64", "steps": 4},
        # a channel between walls
        {"name": "steps_f32_channel_512_m6", "kind": "steps", "nodes": "channel", "nx": 512, "ny": 512, "m": 6,
         "dtype": "f32", "steps": 4},
        # the widest stencils: 1.0M nodes of varying resolution at order 10
        {"name": "rhs_f32_varres_1m_m10", "kind": "rhs", "nodes": "varres", "s0": 6.654e-4, "m": 10, "dtype": "f32"},
        # many instances of mixed orders advanced together, one graph launch per step
        {"name": "graph_f32_batch_48", "kind": "graph", "count": 48, "n_min": 2048, "n_max": 65536, "dtype": "f32",
         "steps": 2},
        # a gradient through a rollout (forward, recomputed segment and reverse sweep)
        {"name": "gradient_f32_256_m8", "kind": "gradient", "nodes": "lattice", "nx": 256, "ny": 256, "m": 8,
         "dtype": "f32", "steps": 20, "every": 10},
        # from a node set to a ready plan and its first right-hand side, as after every remeshing
        {"name": "setup_f32_256_m8", "kind": "setup", "nodes": "lattice", "nx": 256, "ny": 256, "m": 8, "dtype": "f32"},
        # the neighbour search alone, on stencils of varying size
        {"name": "stencils_varres_1m", "kind": "stencils", "nodes": "varres", "s0": 6.654e-4, "m": 10},
        # nodes that move every step: neighbours, weight polynomials and a matrix-free right-hand side
        {"name": "matrix_free_f64_128_m6", "kind": "matrix_free", "nodes": "lattice", "nx": 128, "ny": 128, "m": 6},
    ]


def _side(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rhs", "filter", "steps", "steps", "steps", "graph", "gradient", "setup", "stencils", "matrix_free"])
    if kind == "graph":
        return {"kind": kind, "count": rng.randint(4, 40), "n_min": 2048, "n_max": _side(rng, 4096, 65536),
                "dtype": rng.choice(["f32", "f32", "f64"]), "steps": rng.randint(1, 3)}
    nodes = rng.choice(["lattice", "lattice", "channel", "open_box"]) if kind in ("rhs", "steps") else "lattice"
    if kind == "stencils" and rng.random() < 0.5:
        return {"kind": kind, "nodes": "varres", "s0": math.exp(rng.uniform(math.log(8e-4), math.log(2e-2))), "m": 10}
    m = 6 if nodes in ("channel", "open_box") else rng.choice([4, 6, 8] if kind != "rhs" else [4, 6, 8, 10])
    top = {"gradient": 200, "setup": 250, "matrix_free": 160}.get(kind, 500 if m < 10 else 350)
    nx = _side(rng, 24, top)
    ny = max(24, min(top, int(round(nx * rng.uniform(0.7, 1.4)))))
    case = {"kind": kind, "nodes": nodes, "nx": nx, "ny": ny, "m": m}
    if kind not in ("stencils", "matrix_free"):
        case["dtype"] = rng.choice(["f32", "f64"])
    if kind in ("steps", "gradient"):
        case["steps"] = rng.randint(1, 4 if nx * ny > 65536 else 20)
    if kind == "gradient":
        case["every"] = rng.randint(2, 10)
    return case


# ---------------------------------------------------------------- node sets and fields

def _strips(nx, ny, m, seed):
    """A channel periodic in x between walls at y = 0 and y = ny s (s = 1/nx): five uniform
    rows along each wall, a jittered lattice between them, the rows next to a wall with
    h = 2.2 s.  Returns the node set, the wall nodes' columns and their normals."""
    s, rng = 1.0 / nx, li.rng_for(20, seed)
    H = ny * s
    x = (np.arange(nx) + 0.5) * s
    rows = [(x, np.full(nx, q * s), q) for q in range(5)] + [(x, np.full(nx, H - q * s), q) for q in range(5)]
    for iy in range(5, ny - 4):
        d = rng.uniform(-0.05, 0.05, size=(2, nx))
        rows.append(((x + d[0] * s) % 1.0, (iy + d[1]) * s, 5))
    xy = np.stack([np.concatenate([r[0] for r in rows]), np.concatenate([r[1] for r in rows])], axis=1)
    near = np.concatenate([np.full(nx, r[2] in (1, 2)) for r in rows])
    cols = np.concatenate([np.arange(nx)[:, None] + nx * np.arange(5)[None, :] + 5 * nx * w for w in (0, 1)])
    normals = np.repeat(np.array([[0.0, 1.0], [0.0, -1.0]]), nx, axis=0)
    ns = li.NodeSet(xy, np.full(len(xy), s), np.where(near, 2.2 * s, H_OVER_S[m] * s), 1.0, H, m)
    return ns, cols.astype(np.int32), normals


def _rearranged(ns, seed):
    """The node set mirrored and renumbered from another start: as many stencil entries for
    every seed, so that outputs of that length have one shape."""
    g = np.random.default_rng([seed, 11])
    xy = ns.xy.copy()
    for axis, L in enumerate((ns.Lx, ns.Ly)):
        if g.integers(2):
            xy[:, axis] = np.where(xy[:, axis] > 0, L - xy[:, axis], 0.0)
    k = int(g.integers(1, ns.N))
    return li.NodeSet(np.roll(xy, k, axis=0), np.roll(ns.s, k), np.roll(ns.h, k), ns.Lx, ns.Ly, ns.m)


def _node_set(case, seed):
    if case["kind"] in ("setup", "stencils", "matrix_free"):
        return _rearranged(_drawn_nodes(case, 0)[0], seed), None, None
    return _drawn_nodes(case, seed)


def _drawn_nodes(case, seed):
    """(node set, wall columns, wall normals); the last two are None without boundaries."""
    kind, m = case["nodes"], case["m"]
    if kind == "lattice":
        return li.tgv_lattice(case["nx"], case["ny"], m=m, jitter=0.05, seed=seed), None, None
    if kind == "varres":
        return li.varres_columns(case["s0"], m=m, jitter=0.05, seed=seed), None, None
    if kind == "channel":
        return _strips(case["nx"], case["ny"], m, seed)
    ns, cols, normals = _strips(case["ny"], case["nx"], m, seed)  # the channel turned by 90 degrees
    return li.NodeSet(ns.xy[:, ::-1].copy(), ns.s, ns.h, ns.Ly, ns.Lx, m), cols, normals[:, ::-1].copy()


def _dev(a, dtype=torch.float64):
    return torch.tensor(np.ascontiguousarray(a), dtype=dtype, device=DEV)


def _fields(ns, seed, kind="lattice"):
    """(ln rho, u, v): a Taylor-Green state with seeded phases and a few seeded long waves
    (lattices, columns), a Poiseuille profile with waves that vanish at the walls, or the
    Lamb-Oseen vortex at a seeded centre."""
    g = np.random.default_rng([seed, 77])
    if kind == "open_box":
        ctr = (ns.Lx * (0.5 + 0.1 * g.uniform(-1, 1)), ns.Ly * (0.5 + 0.1 * g.uniform(-1, 1)))
        return _dev(li.lamb_oseen_fields(ns.xy, 1.0 / li.LAMB_OSEEN_MACH, H=ns.Ly, centre=ctr))
    xy = _dev(ns.xy)
    x, y = 2 * math.pi * xy[:, 0] / ns.Lx, 2 * math.pi * xy[:, 1] / ns.Ly
    a, b = g.uniform(0, 2 * math.pi, 2)
    waves = []
    for _ in range(3):
        kx, ky = (int(v) for v in g.integers(1, 5, 2))
        amp, ph = g.uniform(0.01, 0.05), g.uniform(0, 2 * math.pi)
        waves.append(amp * torch.sin(kx * x + ky * y + ph))
    if kind == "channel":
        t = xy[:, 1] / ns.Ly
        edge = torch.where((t <= 0) | (t >= 1), 0.0, torch.sin(math.pi * t))
        return torch.stack([0.01 * waves[0], 4 * t * (1 - t) + edge * waves[1], edge * waves[2]]).contiguous()
    rho = 1.0 - 0.25 / C ** 2 * (torch.cos(2 * (x + a)) + torch.cos(2 * (y + b)))
    return torch.stack([torch.log(rho) + 0.1 * waves[0], -torch.cos(x + a) * torch.sin(y + b) + waves[1],
                        torch.sin(x + a) * torch.cos(y + b) + waves[2]]).contiguous()


def _phys(case, ns):
    if case.get("nodes") == "channel":  # Re = 10, Ma = 0.05
        mu = ns.Ly / 10.0
        return lb.Phys(400.0, mu, 8 * mu / ns.Ly ** 2, 0.0)
    if case.get("nodes") == "open_box":
        c = 1.0 / li.LAMB_OSEEN_MACH
        return lb.Phys(c * c, li.LAMB_OSEEN_RC_OVER_H * ns.Ly / li.LAMB_OSEEN_RE)
    return lb.Phys(C * C, MU)


def _operator(ns, residual=False):
    xy, h, s = _dev(ns.xy), _dev(ns.h), _dev(ns.s)
    rp, col = lb.build_stencils(xy, h, ns.Lx, ns.Ly)
    wb = lb.build_weights(xy, h, s, ns.Lx, ns.Ly, rp, col, ns.m, residual=residual)
    return {"row_ptr": rp, "col": col, "w": wb["w"], "kappa": wb["kappa"], "s": s}


def _plan(case, ns, cols, normals):
    dtype = DTYPES[case["dtype"]]
    if cols is None:
        o = _operator(ns)
        return lb.Plan(o["row_ptr"], o["col"], o["w"], o["kappa"], o["s"], dtype=dtype), o["s"]
    s, nrm = _dev(ns.s), _dev(normals)
    periodic = (True, False) if case["nodes"] == "channel" else (False, True)
    o = lb.build_wall_operator(_dev(ns.xy), _dev(ns.h), s, ns.Lx, ns.Ly, ns.m, 4, _dev(cols, torch.int32), nrm, 1.7,
                               periodic=periodic, check=True)
    plan = lb.Plan(o["row_ptr"], o["col"], o["w"], o["kappa"], s, dtype=dtype)
    wall = _dev(cols[:, 0], torch.int32)
    if case["nodes"] == "channel":
        plan.set_walls(wall, nrm)
    else:
        n = len(cols) // 2
        target = np.zeros((2 * n, 2))
        target[:n, 0], target[n:, 0] = 1.0, _phys(case, ns).c2
        plan.set_boundaries(wall, nrm, _dev([lb.INFLOW] * n + [lb.OUTFLOW] * n, torch.int32), _dev(target), L=ns.Lx,
                            mach=li.LAMB_OSEEN_MACH)
    return plan, s


def _instances(case, seed):
    """The batch's lattices, grouped by order as a caller lays them out."""
    rng = li.rng_for(3, seed)
    sides = np.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"]), case["count"]) / 2)
    orders = [4, 6, 8] * (case["count"] // 3 + 1)
    sides = _spread(sides, case)
    return [li.tgv_lattice(n, n, m=m, jitter=0.05, seed=seed * 1000 + k)
            for k, (n, m) in enumerate(sorted(zip(sides, orders), key=lambda t: t[1]))]


def _spread(sides, case):
    """Log-uniform sides whose total does not depend on the seed: the quantiles of the
    distribution, in the drawn order."""
    q = (np.arange(case["count"]) + 0.5) / case["count"]
    even = np.exp((math.log(case["n_min"]) + q * math.log(case["n_max"] / case["n_min"])) / 2)
    return [max(8, int(round(even[k]))) for k in np.argsort(np.argsort(sides))]


# ---------------------------------------------------------------- a pass

def prepare(case, seed):
    kind = case["kind"]
    if kind == "graph":
        sets = _instances(case, seed)
        plan = lb.Plan.batched([_operator(ns) for ns in sets], dtype=DTYPES[case["dtype"]])
        q = torch.cat([_fields(ns, seed + k) for k, ns in enumerate(sets)], dim=1).to(DTYPES[case["dtype"]]).contiguous()
        s = torch.cat([_dev(ns.s) for ns in sets])
        plan.set_dt(plan.stable_dt_instances(q, s, C, MU).cpu().tolist())
        return {"kind": kind, "plan": plan, "q": q, "steps": case["steps"], "graph": lb.StepGraph(plan, 0.0, lb.Phys(C * C, MU))}
    ns, cols, normals = _node_set(case, seed)
    st = {"kind": kind, "ns": (ns.Lx, ns.Ly, ns.m), "xy": _dev(ns.xy), "h": _dev(ns.h), "s": _dev(ns.s),
          "phys": _phys(case, ns), "dtype": DTYPES.get(case.get("dtype")), "steps": case.get("steps"),
          "every": case.get("every")}
    if kind == "stencils":
        return st
    q = _fields(ns, seed, case["nodes"])
    if kind == "matrix_free":
        return {**st, "q": q}
    st["q"] = q.to(st["dtype"]).contiguous()
    if kind == "setup":
        return st
    plan, s = _plan(case, ns, cols, normals)
    ph = st["phys"]
    st |= {"plan": plan, "work": lb.workspace(plan), "dt": float(lb.stable_dt(plan, st["q"], s, math.sqrt(ph.c2), ph.mu).item())}
    if kind == "gradient":
        lb.enable_adjoint(plan)
    return st


def run(state):
    kind = state["kind"]
    if kind == "rhs":
        return lb.rhs(state["plan"], state["q"], state["phys"])
    if kind == "filter":
        return lb.filter(state["plan"], state["q"])
    if kind == "steps":
        return lb.rk_step(state["plan"], state["q"].clone(), state["dt"], state["steps"], state["phys"], work=state["work"])
    if kind == "graph":
        return state["graph"].run(state["q"].clone(), state["steps"])
    if kind == "gradient":
        q0 = state["q"].clone().requires_grad_(True)
        q = lb.rollout(state["plan"], q0, state["dt"], state["steps"], state["phys"], checkpoint_every=state["every"])
        e = lb.domain_kinetic_energy(q, state["s"])
        e.backward(torch.ones_like(e))
        return {"state": q.detach(), "energy": e.detach(), "gradient": q0.grad}
    Lx, Ly, m = state["ns"]
    xy, h, s = state["xy"], state["h"], state["s"]
    rp, col = lb.build_stencils(xy, h, Lx, Ly)
    if kind == "stencils":
        return {"row_ptr": rp, "col": col}
    if kind == "matrix_free":
        wc = lb.weight_coefficients(xy, h, s, Lx, Ly, rp, col, m)
        r = lb.rhs_matrix_free(xy, h, Lx, Ly, rp, col, m, wc["coef"], state["q"], state["phys"])
        return {"row_ptr": rp, "col": col, "kappa": wc["kappa"], "status": wc["status"], "rhs": r}
    wb = lb.build_weights(xy, h, s, Lx, Ly, rp, col, m, residual=False)
    plan = lb.Plan(rp, col, wb["w"], wb["kappa"], s, dtype=state["dtype"])
    r = lb.rhs(plan, state["q"], state["phys"])
    plan.close()
    return {"row_ptr": rp, "col": col, "w": wb["w"], "kappa": wb["kappa"], "status": wb["status"], "rhs": r}


# ---------------------------------------------------------------- what a pass cannot do without

def _counts(case):
    """(nodes, stencil entries), from the node sets' construction."""
    if case["kind"] == "graph":
        lo, hi = case["n_min"], case["n_max"]
        N = case["count"] * (hi - lo) / math.log(hi / lo) if hi > lo else case["count"] * lo
        return N, N * 4 * math.pi * (1.7 ** 2 + 2.2 ** 2 + 2.8 ** 2) / 3
    hs = H_OVER_S[case["m"]]
    if case["nodes"] == "varres":  # columns of spacing s(x): the integral of 1/s^2; E[M^2] = 1.116
        N = 0.445 / case["s0"] ** 2
        return N, N * (1.116 * 4 * math.pi * hs * hs - 1)
    N = case["nx"] * case["ny"]
    return N, N * (4 * math.pi * hs * hs - 1)


def work(case):
    """Bytes: the operator (five weights and a column per entry; filter one and a column)
    once per right-hand side that reads it, node state and results once.  Flops: 27 per
    entry and right-hand side, 9 per entry and filter; the weight build's linear algebra."""
    N, nnz = _counts(case)
    b = {"f32": 4, "f64": 8, None: 8}[case.get("dtype")]
    rhs_b, rhs_f = nnz * (4 + 5 * b) + 6 * b * N, 27 * nnz + 45 * N
    fil_b, fil_f = nnz * (4 + b) + 6 * b * N, 9 * nnz
    kind, steps = case["kind"], case.get("steps", 1)
    if kind == "rhs":
        return {"bytes": rhs_b, "flops": rhs_f}
    if kind == "filter":
        return {"bytes": fil_b, "flops": fil_f}
    if kind in ("steps", "graph"):
        return {"bytes": steps * (4 * rhs_b + fil_b), "flops": steps * (4 * rhs_f + fil_f)}
    if kind == "gradient":  # forward, the segments recomputed (all but the last), and the reverse sweep
        again = max(0, (steps - 1) // case["every"] * case["every"])
        n = 2 * steps + again
        return {"bytes": n * (4 * rhs_b + fil_b), "flops": n * (4 * rhs_f + fil_f)}
    if kind == "stencils":
        return {"bytes": 24 * N + 4 * nnz + 4 * N, "flops": 8 * nnz}
    m = case["m"]
    n = (m * m + 3 * m) // 2
    build = N * (2 * n ** 3 / 3 + 12 * n * n) + nnz * (2 * (2 * m + 1) * (m + 1) + 12 * (m + 1) * (m + 2) / 2)
    if kind == "matrix_free":
        return {"bytes": 80 * N + 8 * nnz, "flops": build + nnz * (5 * (m + 1) * (m + 2) + 27)}
    return {"bytes": 40 * N + nnz * (4 + 48 + 4 + 5 * b + 4 + b) + rhs_b, "flops": build + rhs_f}


# ---------------------------------------------------------------- the same in plain torch, 64 bits

def _image(d, L):
    d = torch.where(d > 0.5 * L, d - L, d)
    return torch.where(d < -0.5 * L, d + L, d)


class _Exact:
    """The method on a doubly periodic node set, written from its definitions: stencils
    |r_ji| <= 2 h_i, weights from dense solves, difference-form operators."""

    def __init__(self, ns, weights=True):
        self.ns, self.N = ns, ns.N
        xy, h, s = _dev(ns.xy), _dev(ns.h), _dev(ns.s)
        self.s = s
        rows = max(1, (1 << 27) // ns.N)
        parts = []
        for r in range(0, ns.N, rows):
            e = min(ns.N, r + rows)
            dx = _image(xy[None, :, 0] - xy[r:e, None, 0], ns.Lx)
            dy = _image(xy[None, :, 1] - xy[r:e, None, 1], ns.Ly)
            near = dx * dx + dy * dy <= ((2.0 * h[r:e]) * (2.0 * h[r:e]))[:, None]
            near[torch.arange(e - r, device=DEV), torch.arange(r, e, device=DEV)] = False
            i, j = near.nonzero(as_tuple=True)
            parts.append((i + r, j))
        i, j = torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts])
        cnt = torch.bincount(i, minlength=ns.N)
        self.row_ptr = torch.cat([cnt.new_zeros(1), cnt.cumsum(0)])
        self.col = j
        K = int(cnt.max())
        at = torch.arange(len(j), device=DEV) - self.row_ptr[i]
        self.flat = (i, at)
        self.nb = torch.arange(ns.N, device=DEV)[:, None].repeat(1, K)
        self.nb[i, at] = j
        self.mask = torch.zeros((ns.N, K), dtype=torch.bool, device=DEV)
        self.mask[i, at] = True
        if weights:
            self._weights(xy, h, s)

    def _weights(self, xy, h, s):
        m = self.ns.m
        ex = [(k - b, b) for k in range(1, m + 1) for b in range(k + 1)]
        self.w = torch.zeros((6,) + tuple(self.nb.shape), dtype=torch.float64, device=DEV)
        self.kappa = torch.zeros(self.N, dtype=torch.float64, device=DEV)
        sel = torch.zeros((len(ex), 6), dtype=torch.float64, device=DEV)
        for q, e in enumerate(ex):
            for d, t in enumerate([(1, 0), (0, 1), (2, 0), (1, 1), (0, 2)]):
                sel[q, d] = float(e == t)
            if sum(e) == m and e[0] % 2 == 0:
                sel[q, 5] = math.comb(m // 2, e[0] // 2)
        order = torch.tensor([1, 1, 2, 2, 2, m], dtype=torch.float64, device=DEV)
        step = max(1, (1 << 27) // (len(ex) * self.nb.shape[1]))
        for r in range(0, self.N, step):
            nb, ok, hr = self.nb[r:r + step], self.mask[r:r + step], h[r:r + step, None]
            dx = _image(xy[nb, 0] - xy[r:r + step, None, 0], self.ns.Lx)
            dy = _image(xy[nb, 1] - xy[r:r + step, None, 1], self.ns.Ly)
            X, Y = dx / hr, dy / hr
            z = torch.sqrt(X * X + Y * Y)
            psi = torch.where(ok & (z <= 2), (1 - z / 2) ** 4 * (1 + 2 * z), 0.0)
            px, py = [torch.ones_like(X), X], [torch.ones_like(Y), Y]
            hx, hy = [torch.ones_like(X), X], [torch.ones_like(Y), Y]
            for k in range(1, m):
                px.append(px[-1] * X)
                py.append(py[-1] * Y)
                hx.append(X * hx[-1] - k * hx[-2])
                hy.append(Y * hy[-1] - k * hy[-2])
            mono = torch.stack([px[a] * py[b] / (math.factorial(a) * math.factorial(b)) for a, b in ex], 1)
            abf = torch.stack([psi * hx[a] * hy[b] for a, b in ex], 2)
            psi_d = torch.linalg.solve(mono @ abf, sel.expand(len(nb), -1, -1))
            w = (abf @ psi_d) / hr[:, :, None] ** order
            self.w[:, r:r + step] = w.permute(2, 0, 1)
            kx = 1.5 * math.pi / s[r:r + step, None]
            f0 = ((1 - torch.cos(kx * dx) * torch.cos(kx * dy)) * w[:, :, 5]).sum(1)
            self.kappa[r:r + step] = 2 / (3 * f0)

    def rhs(self, q, ph):
        a, u, v = q
        da, du, dv = (f[self.nb] - f[:, None] for f in q)

        def D(d, k):
            return torch.einsum("nk,nk->n", self.w[k], d)

        ax, ay, ux, uy, vx, vy = D(da, 0), D(da, 1), D(du, 0), D(du, 1), D(dv, 0), D(dv, 1)
        nu = ph.mu * torch.exp(-a)
        Ru = nu * (4 / 3 * D(du, 2) + D(du, 4) + D(dv, 3) / 3) - u * ux - v * uy - ph.c2 * ax + ph.gx
        Rv = nu * (4 / 3 * D(dv, 4) + D(dv, 2) + D(du, 3) / 3) - u * vx - v * vy - ph.c2 * ay + ph.gy
        return torch.stack([-u * ax - v * ay - ux - vy, Ru, Rv])

    def filter(self, q):
        return torch.stack([f + self.kappa * torch.einsum("nk,nk->n", self.w[5], f[self.nb] - f[:, None]) for f in q])

    def step(self, q, dt, ph):
        A = (11847461282814 / 36547543011857, 3943225443063 / 7078155732230, -346793006927 / 4029903576067)
        B = (1017324711453 / 9774461848756, 8237718856693 / 13685301971492, 57731312506979 / 19404895981398,
             -101169746363290 / 37734290219643)
        x = q
        for k in range(4):
            f = self.rhs(x, ph)
            q = q + dt * B[k] * f
            x = q + dt * (A[k] - B[k]) * f if k < 3 else q
        return self.filter(x)

    def dt(self, q, c, mu):
        conv = self.s / (torch.sqrt(q[1] ** 2 + q[2] ** 2) + c)
        return float(torch.minimum(conv, 0.4 * self.s ** 2 * torch.exp(q[0]) / mu).min())


def exact(case, seed):
    kind = case["kind"]
    if kind == "graph":
        out = []
        for k, ns in enumerate(_instances(case, seed)):
            e, q = _Exact(ns), _fields(ns, seed + k).to(DTYPES[case["dtype"]]).double()
            dt = e.dt(q, C, MU)
            for _ in range(case["steps"]):
                q = e.step(q, dt, lb.Phys(C * C, MU))
            out.append(q)
        return torch.cat(out, dim=1)
    # stencils are whole numbers only: equal or not
    if kind == "stencils" or case["nodes"] in ("channel", "open_box") or _counts(case)[0] > 280000:
        return None
    ns, _, _ = _node_set(case, seed)
    e, ph = _Exact(ns), _phys(case, ns)
    q = _fields(ns, seed, case["nodes"])
    q = q.to(DTYPES.get(case.get("dtype"), torch.float64)).double()
    if kind == "rhs":
        return e.rhs(q, ph)
    if kind == "filter":
        return e.filter(q)
    if kind == "matrix_free":
        return {"row_ptr": None, "col": None, "kappa": e.kappa, "status": None, "rhs": e.rhs(q, ph)}
    if kind == "setup":
        return {"row_ptr": None, "col": None, "w": e.w[:, e.flat[0], e.flat[1]], "kappa": e.kappa, "status": None,
                "rhs": e.rhs(q, ph)}
    dt = e.dt(q, math.sqrt(ph.c2), ph.mu)
    if kind == "steps":
        for _ in range(case["steps"]):
            q = e.step(q, dt, ph)
        return q
    q0 = q.requires_grad_(True)
    for _ in range(case["steps"]):
        q = e.step(q, dt, ph)
    ke = (0.5 * torch.exp(q[0]) * (q[1] ** 2 + q[2] ** 2) * e.s ** 2).sum().reshape(1)
    return {"state": q.detach(), "energy": ke.detach(), "gradient": torch.autograd.grad(ke, q0)[0]}
