"""FP64 plans, whose sums run in fixed point: against extended-precision sums of the same
weights and differences, over row lengths, lanes, ranges of magnitude and plans that keep
FP64 weights; infinities and NaN; exact zeros."""
import numpy as np
import pytest

import labfm_inputs as li

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lb():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import __graft_entry__ as g
    g.build()
    import paper_2102_02019_gb300 as lb
    return lb


def _operator(N, lengths, scale, seed):
    """Random rows: weights falling off by five orders along the row, columns at random."""
    rng = np.random.default_rng(seed)
    rp = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    col = np.concatenate([np.sort(rng.choice(N, n, replace=False)) for n in lengths]).astype(np.int32)
    fall = np.concatenate([10.0 ** rng.uniform(-5, 0, n) for n in lengths])
    w = scale * fall * rng.standard_normal((6, len(col)))
    return rp, col, w, rng.uniform(0.5, 1.5, N)


def _plan(lb, rp, col, w, kappa):
    dev = lambda a: torch.tensor(a, device="cuda")  # noqa: E731
    return lb.Plan(dev(rp), dev(col), dev(w), dev(kappa), dev(np.ones(len(rp) - 1)), dtype=torch.float64)


def _sums(rp, col, w, q):
    """Per operator and field sum_j w (q_j - q_i) in extended precision, and the bound
    n 2^-50 max|w| max|d| on the fixed-point error: 2^-57 of the bound of |w| (at most 4
    max|w|) and 2^-57 of the bound of |d| (at most 16 max|d|, shifts included) per term,
    2^-56 for the dropped product, and FP64's n 2^-53 besides."""
    N = len(rp) - 1
    out, tol = np.zeros((len(w), 3, N), np.longdouble), np.zeros((len(w), 3, N))
    for i in range(N):
        s = slice(rp[i], rp[i + 1])
        d = (q[:, col[s]] - q[:, i:i + 1])
        out[:, :, i] = w[:, s].astype(np.longdouble) @ d.astype(np.longdouble).T
        if rp[i + 1] > rp[i]:
            tol[:, :, i] = (rp[i + 1] - rp[i]) * 2.0 ** -50 * np.abs(w[:, s]).max(1)[:, None] * np.abs(d).max(1)[None, :]
    return out, tol


def _check(lb, plan, rp, col, w, kappa, q):
    Q = torch.tensor(q, device="cuda")
    f, tf = _sums(rp, col, kappa[np.repeat(np.arange(len(rp) - 1), np.diff(rp))] * w[5:], q)
    got = lb.filter(plan, Q).cpu().numpy()
    assert np.all(np.abs(got - (q + f[0])) <= tf[0] + 2.0 ** -52 * np.abs(q + f[0]))
    # rho du/dt with c^2 = 0, mu = 0: R_a = -(u a_x + v a_y) - (u_x + v_y), R_u = -(u u_x + v u_y)
    s, t = _sums(rp, col, w[:2], q)
    a, u, v = q
    R = np.stack([-(u * s[0, 0] + v * s[1, 0]) - (s[0, 1] + s[1, 2])] + [-(u * s[0, k] + v * s[1, k]) for k in (1, 2)])
    T = np.stack([np.abs(u) * t[0, 0] + np.abs(v) * t[1, 0] + t[0, 1] + t[1, 2]]
                 + [np.abs(u) * t[0, k] + np.abs(v) * t[1, k] for k in (1, 2)])
    mag = np.stack([np.abs(u * s[0, 0]) + np.abs(v * s[1, 0]) + np.abs(s[0, 1]) + np.abs(s[1, 2])]
                   + [np.abs(u * s[0, k]) + np.abs(v * s[1, k]) for k in (1, 2)])
    with np.errstate(over="ignore", invalid="ignore"):
        R[1:] += 0.0 * np.exp(-a)  # the viscous term: mu / rho = 0, not a number where rho underflows
    got = lb.rhs(plan, Q, lb.Phys(0.0, 0.0)).cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(R))
    ok = ~np.isnan(R)
    assert np.all(np.abs(got - R)[ok] <= (T + 2.0 ** -50 * mag)[ok])


@pytest.mark.parametrize("group", [2, 4, 8, 16, 32])
@pytest.mark.parametrize("scale,spread", [(1.0, 1.0), (1e9, 1e-9), (1e-30, 1e40)])
def test_sums_over_row_lengths(lb, group, scale, spread):
    # empty rows, chunk edges, and rows past the 64 entries a lane sums between carries
    lengths = [0, 1, 3, 4, 5, 15, 16, 17, 63, 64, 65, 127, 128, 129, 255, 256, 257, 600] * 3
    rng = np.random.default_rng(1)
    N = 620
    lengths = np.array(lengths + list(rng.integers(0, 40, N - len(lengths))))
    rp, col, w, kappa = _operator(N, lengths, scale, 2)
    plan = _plan(lb, rp, col, w, kappa)
    plan.set_launch(group, 128)
    _check(lb, plan, rp, col, w, kappa, spread * rng.standard_normal((3, N)))
    plan.close()


@pytest.mark.parametrize("what", ["wide_weights", "tiny_weights", "huge_differences", "tiny_differences"])
def test_magnitudes_out_of_the_fixed_range(lb, what):
    rng = np.random.default_rng(5)
    N = 200
    rp, col, w, kappa = _operator(N, np.full(N, 30), 1.0, 3)
    q = rng.standard_normal((3, N))
    if what == "wide_weights":
        w[:, ::7] *= 1e130  # beyond 2^400: FP64 weights
    if what == "tiny_weights":
        w *= 1e-130
    if what == "huge_differences":
        q[0] *= 1e155  # beyond 2^500: those rows in FP64
    if what == "tiny_differences":
        q[1] *= 1e-160
    plan = _plan(lb, rp, col, w, kappa)
    _check(lb, plan, rp, col, w, kappa, q)
    plan.close()


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("where", ["state", "weight"])
def test_not_finite_values_come_out_as_in_fp64(lb, bad, where):
    rng = np.random.default_rng(6)
    N = 150
    rp, col, w, kappa = _operator(N, np.full(N, 20), 1.0, 4)
    q = rng.standard_normal((3, N))
    if where == "state":
        q[1, 17] = bad
    else:
        w[5, rp[40] + 3] = bad
    plan = _plan(lb, rp, col, w, kappa)
    got = lb.filter(plan, torch.tensor(q, device="cuda")).cpu().numpy()
    with np.errstate(invalid="ignore"):
        ref = np.stack([[q[f, i] + (kappa[i] * w[5, rp[i]:rp[i + 1]] * (q[f, col[rp[i]:rp[i + 1]]] - q[f, i])).sum()
                         for i in range(N)] for f in range(3)])
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    fin = np.isfinite(ref)
    assert np.array_equal(got[~fin & ~np.isnan(ref)], ref[~fin & ~np.isnan(ref)])
    assert np.allclose(got[fin], ref[fin], rtol=1e-12, atol=1e-12)
    plan.close()


def test_uniform_fields_give_exact_zeros(lb):
    rng = np.random.default_rng(7)
    N = 300
    rp, col, w, kappa = _operator(N, np.full(N, 25), 1e6, 8)
    plan = _plan(lb, rp, col, w, kappa)
    q = torch.tensor(np.repeat(rng.standard_normal((3, 1)), N, axis=1), device="cuda")
    q[2] = torch.where(torch.arange(N, device="cuda") % 2 == 0, 0.0, -0.0)  # differences of -0
    assert torch.equal(lb.filter(plan, q), q)
    assert not lb.rhs(plan, q, lb.Phys(100.0, 0.1)).any()
    plan.close()


@pytest.mark.parametrize("N", [70, 1073, 20000])
def test_launches_without_a_gap_read_what_came_before(lb, N):
    # right-hand sides and filters, launched to start as the launch before ends, between
    # kernels that write their inputs: the same bits as with a synchronisation after each
    rng = np.random.default_rng(N)
    rp, col, w, kappa = _operator(N, np.full(N, 24), 1.0, N)
    plan = _plan(lb, rp, col, w, 1e-3 * kappa)
    q0 = torch.tensor(rng.standard_normal((3, N)), device="cuda")
    phys = lb.Phys(1.0, 0.01)
    out = []
    for wait, programmatic in ((False, True), (True, True), (False, False)):
        plan.set_programmatic_launch(programmatic)
        q = q0.clone()
        for _ in range(20):
            r = lb.rhs(plan, q, phys)
            q = lb.filter(plan, torch.tanh(q + 1e-3 * r))
            q = lb.filter(plan, q)
            if wait:
                torch.cuda.synchronize()
        out.append(q)
    assert torch.isfinite(out[0]).all()
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
    plan.close()


@pytest.mark.parametrize("scale", [2.0 ** -940, 2.0 ** -958, 2.0 ** -963, 2.0 ** -990, 2.0 ** -1012])
def test_fields_with_tiny_differences_only(lb, scale):
    # rows whose differences are all below the fixed-point range: the tail of a pulse in
    # fluid at rest.  FP64's own error: n 2^-53 sum |w d|, and half of 2^-1074 per product
    rng = np.random.default_rng(11)
    N = 260
    rp, col, w, kappa = _operator(N, rng.integers(1, 70, N), 1.0, 12)
    q = scale * rng.uniform(1.0, 3.0, (3, N))
    plan = _plan(lb, rp, col, w, kappa)
    got = lb.filter(plan, torch.tensor(q, device="cuda")).cpu().numpy()
    r = lb.rhs(plan, torch.tensor(np.stack([0.0 * q[0], q[1], q[2]]), device="cuda"), lb.Phys(0.0, 0.0)).cpu().numpy()
    for i in range(N):
        s = slice(rp[i], rp[i + 1])
        d = (q[:, col[s]] - q[:, i:i + 1]).astype(np.longdouble)
        n, tiny = rp[i + 1] - rp[i], 2.0 ** -1074
        wf = (kappa[i] * w[5, s]).astype(np.longdouble)
        ref, mag = d @ wf, np.abs(d) @ np.abs(wf)
        assert np.all(np.abs(got[:, i] - (q[:, i] + ref)) <= (n + 2) * (2.0 ** -53 * (mag + np.abs(q[:, i])) + tiny)), i
        # R of ln rho with ln rho = 0: -(u_x + v_y)
        ref = -(w[0, s].astype(np.longdouble) @ d[1] + w[1, s].astype(np.longdouble) @ d[2])
        mag = np.abs(w[0, s]) @ np.abs(d[1]) + np.abs(w[1, s]) @ np.abs(d[2])
        assert abs(r[0, i] - ref) <= (n + 3) * (2.0 ** -53 * mag + 2 * tiny), i
    plan.close()


@pytest.mark.parametrize("spread", [5, 15, 40, 140])
def test_weights_are_held_bit_for_bit(lb, spread):
    # weights over `spread` decades within a row, read back one by one: a field that is zero
    # but at one node gives the weights on that node times a power of two (2^-700: below the
    # fixed-point range, so in FP64), and the adjoint of one output gives its row
    rng = np.random.default_rng(spread)
    N = 90
    lengths = rng.integers(1, 80, N)
    rp, col, w, kappa = _operator(N, lengths, 1.0, 13)
    w *= 10.0 ** rng.uniform(5 - spread, 0, w.shape)
    col = np.concatenate([np.sort(rng.choice([j for j in range(N) if j != i], n, replace=False))
                          for i, n in enumerate(lengths)]).astype(np.int32)
    plan = _plan(lb, rp, col, w, kappa)
    lb.enable_adjoint(plan)
    row = np.repeat(np.arange(N), lengths)
    zero = np.zeros((3, N))
    for j in range(0, N, 7):
        on = col == j
        rows = row[on]
        q = zero.copy()
        q[1, j] = 2.0 ** -700
        out = lb.filter(plan, torch.tensor(q, device="cuda")).cpu().numpy()
        assert np.array_equal(out[1, rows], kappa[rows] * w[5, on] * 2.0 ** -700)
        out = lb.rhs(plan, torch.tensor(q, device="cuda"), lb.Phys(0.0, 0.0)).cpu().numpy()
        assert np.array_equal(out[0, rows], -w[0, on] * 2.0 ** -700)
        # R_a = -(u_x + v_y), R_u = -c^2 a_x at rest
        lam = zero.copy()
        lam[0, j] = 1.0
        g = lb.rhs_adjoint(plan, torch.tensor(zero, device="cuda"), torch.tensor(lam, device="cuda"),
                           lb.Phys(1.0, 0.0)).cpu().numpy()
        on = row == j
        assert np.array_equal(g[1, col[on]], -w[0, on]) and np.array_equal(g[2, col[on]], -w[1, on])
        g = lb.filter_adjoint(plan, torch.tensor(lam, device="cuda")).cpu().numpy()
        assert np.array_equal(g[0, col[on]], kappa[j] * w[5, on])
    plan.close()


def _wide_field(kind, ns, rng):
    x, y = ns.xy.T
    s = ns.s[0]
    if kind == "front":
        return np.stack([0.3 * np.tanh((x - 0.5) / (k * s)) for k in (0.2, 0.5, 2.0)])
    if kind == "pulse":
        return np.stack([np.exp(-((x - 0.5) ** 2 + (y - 0.5) ** 2) / (2 * (k * s) ** 2)) for k in (2, 5, 10)])
    if kind == "impulses":
        return (rng.random((3, ns.N)) < 1 / 60) * rng.standard_normal((3, ns.N))
    if kind == "steep":  # saturates: differences of a rounding beside those of the front
        return np.stack([np.tanh((x - 0.5) / (k * s)) for k in (0.1, 0.3, 0.6)])
    if kind == "on_a_stream":  # a pulse that is small against its background, sparse rounding noise
        g = np.exp(-((x - 0.5) ** 2 + (y - 0.5) ** 2) / (2 * (6 * s) ** 2))
        return np.stack([1 + 1e-13 * g, 1 + 2.0 ** -52 * (rng.random(ns.N) < 0.02), 3 + 1e-9 * g])
    if kind == "jump":  # small differences beside a unit one
        return 1e-9 * rng.standard_normal((3, ns.N)) + (x > 0.5)
    return 1e-6 * np.exp(5 * rng.standard_normal((3, ns.N))).clip(max=1e6)  # log-normal


@pytest.mark.parametrize("m", [4, 6, 8, 10])
@pytest.mark.parametrize("kind", ["front", "steep", "pulse", "impulses", "jump", "on_a_stream", "lognormal"])
def test_fields_of_a_wide_span_within_a_stencil(lb, kind, m):
    # every sum within (24 + n) 2^-53 sum |w d| of the exact one (FP64's own bound for n
    # terms and the lanes' sums), for each operator and field: the bounds of the sums that
    # enter an output, with its coefficients, and a few roundings of its terms
    ns = li.tgv_lattice(30, 28, m=m, jitter=0.3 if m != 4 else 0.05, seed=m)
    xy, h, sp = (torch.tensor(a, device="cuda") for a in (ns.xy, ns.h, ns.s))
    rpd, cold = lb.build_stencils(xy, h, ns.Lx, ns.Ly)
    wb = lb.build_weights(xy, h, sp, ns.Lx, ns.Ly, rpd, cold, m, residual=False)
    plan = lb.Plan(rpd, cold, wb["w"], wb["kappa"], sp, dtype=torch.float64)
    rp, col, w, kappa = (t.cpu().numpy() for t in (rpd, cold, wb["w"], wb["kappa"]))
    q = _wide_field(kind, ns, np.random.default_rng(m))
    Q = torch.tensor(q, device="cuda")
    ph = lb.Phys(3.0, 0.7)
    R, filt = lb.rhs(plan, Q, ph).cpu().numpy(), lb.filter(plan, Q).cpu().numpy()
    L, u = np.longdouble, 2.0 ** -53
    S, B = np.zeros((6, 3, ns.N), L), np.zeros((6, 3, ns.N))
    for i in range(ns.N):
        s = slice(rp[i], rp[i + 1])
        d = (q[:, col[s]] - q[:, i:i + 1]).astype(L)
        wi = w[:, s].copy()
        wi[5] *= kappa[i]
        S[:, :, i] = wi.astype(L) @ d.T
        B[:, :, i] = (24 + rp[i + 1] - rp[i]) * u * (np.abs(wi) @ np.abs(d).T.astype(float))
    a, uu, vv = q
    nu = 0.7 * np.exp(-a.astype(L))
    third = L(1) / 3

    def out(terms):  # [(coefficient, operator, field)]: value and bound
        val = sum(c * S[o, f] for c, o, f in terms)
        tol = sum(np.abs(c) * (B[o, f] + 12 * u * np.abs(S[o, f])) for c, o, f in terms)
        return val, tol
    for k, terms in enumerate([[(-uu, 0, 0), (-vv, 1, 0), (-1, 0, 1), (-1, 1, 2)],
                               [(-uu, 0, 1), (-vv, 1, 1), (-3, 0, 0), (4 * third * nu, 2, 1), (nu, 4, 1), (third * nu, 3, 2)],
                               [(-uu, 0, 2), (-vv, 1, 2), (-3, 1, 0), (4 * third * nu, 4, 2), (nu, 2, 2), (third * nu, 3, 1)]]):
        val, tol = out(terms)
        assert np.all(np.abs(R[k] - val) <= tol), k
    for f in range(3):
        assert np.all(np.abs(filt[f] - (q[f] + S[5, f])) <= B[5, f] + 2 * u * np.abs(filt[f])), f
    # one sum at a time: of a field alone, R of ln rho is -u_x or -v_y
    for f in range(3):
        for op in range(2):
            alone = np.zeros_like(q)
            alone[1 + op] = q[f]
            got = lb.rhs(plan, torch.tensor(alone, device="cuda"), lb.Phys(0.0, 0.0)).cpu().numpy()[0]
            assert np.all(np.abs(got + S[op, f]) <= B[op, f]), (f, op)
    plan.close()


def _lattice_operator(lb, nx, ny, m, seed):
    ns = li.tgv_lattice(nx, ny, m=m, jitter=0.05, seed=seed)
    xy, h, s = (torch.tensor(a, device="cuda") for a in (ns.xy, ns.h, ns.s))
    rp, col = lb.build_stencils(xy, h, ns.Lx, ns.Ly)
    wb = lb.build_weights(xy, h, s, ns.Lx, ns.Ly, rp, col, m, residual=False)
    return ns, {"row_ptr": rp, "col": col, "w": wb["w"], "kappa": wb["kappa"], "s": s}


@pytest.mark.parametrize("weight", [np.nan, np.inf, 1e130, 1e-310])
def test_a_row_out_of_the_fixed_range_changes_no_other_instance(lb, weight):
    # an instance's bits alone and beside one with such a weight in one row (a failed node)
    ns, a = _lattice_operator(lb, 22, 20, 4, 1)
    nb, b = _lattice_operator(lb, 17, 19, 6, 2)
    b["w"] = b["w"].clone()
    b["w"][5, 40] = weight
    alone = lb.Plan.batched([a], dtype=torch.float64)
    both = lb.Plan.batched([b, a], dtype=torch.float64)
    q = torch.tensor(li.tgv_fields(ns.xy, 10.0), device="cuda")
    Q = torch.cat([torch.tensor(li.tgv_fields(nb.xy, 10.0), device="cuda"), q], dim=1).contiguous()
    ph, part = lb.Phys(100.0, 0.005), slice(nb.N, None)
    assert torch.equal(lb.rhs(both, Q, ph)[:, part], lb.rhs(alone, q, ph))
    assert torch.equal(lb.filter(both, Q)[:, part], lb.filter(alone, q))
    dt = float(lb.stable_dt(alone, q, a["s"], 10.0, 0.005).item())
    assert torch.equal(lb.rk_step(both, Q, dt, 3, ph)[:, part], lb.rk_step(alone, q, dt, 3, ph))
    alone.close()
    both.close()


def _plain_rows(op):
    """The operator with one more entry in every row, on a node that is not in it (a column
    stands in a row once), whose weights are subnormal (1e-310): rows that hold plain FP64
    weights, with the same sums."""
    rp, col, w = (op[k].cpu().numpy() for k in ("row_ptr", "col", "w"))
    at = rp[1:]
    N = len(at)
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    return {**op, "row_ptr": dev((rp + np.arange(N + 1)).astype(np.int32)),
            "col": dev(np.insert(col, at, (np.arange(N) + N // 2) % N).astype(np.int32)),
            "w": dev(np.insert(w, at, 1e-310, axis=1))}


def _close(a, b):
    return bool((torch.linalg.vector_norm(a - b, dim=-1) <= 1e-12 * torch.linalg.vector_norm(b, dim=-1)).all())


@pytest.mark.parametrize("group", [2, 4, 8, 16, 32])
def test_plain_fp64_rows_through_every_call(lb, group):
    # right-hand side, filter, steps, recorded steps, ranges and adjoints of a plan whose rows
    # all hold FP64 weights, against the same operator in fixed point: the package's FP64 bar
    ns, op = _lattice_operator(lb, 26, 25, 6, 3)
    ph = lb.Phys(100.0, 0.005)
    q = torch.tensor(li.tgv_fields(ns.xy, 10.0), device="cuda")
    q[0] += 0.01 * torch.sin(torch.arange(ns.N, device="cuda"))
    out = []
    for o in (op, _plain_rows(op)):
        plan = lb.Plan(o["row_ptr"], o["col"], o["w"], o["kappa"], o["s"], dtype=torch.float64)
        plan.set_launch(group, 128)
        lb.enable_adjoint(plan)
        dt = float(lb.stable_dt(plan, q, o["s"], 10.0, 0.005).item())
        r = [lb.rhs(plan, q, ph), lb.filter(plan, q), lb.rk_step(plan, q.clone(), dt, 3, ph)]
        r.append(lb.rhs_adjoint(plan, q, r[0], ph))
        r.append(lb.filter_adjoint(plan, r[0]))
        q0 = q.clone().requires_grad_(True)
        z = lb.rollout(plan, q0, dt, 4, ph, checkpoint_every=2)
        lb.domain_kinetic_energy(z, o["s"]).backward()
        r += [z.detach(), q0.grad]
        plan.set_launch_ranges([0, 300, ns.N], [group, 4], [0, 0])
        r.append(lb.rk_step(plan, q.clone(), dt, 2, ph))
        out.append(r)
        plan.close()
    for a, b in zip(*out):
        assert torch.isfinite(b).all() and _close(b, a)


def test_plain_fp64_rows_beside_walls(lb):
    ns = li.channel(24, 20, m=6, jitter=0.1, seed=4)
    cols, normals = li.channel_walls(ns)
    dev = lambda a, t=torch.float64: torch.tensor(np.ascontiguousarray(a), dtype=t, device="cuda")  # noqa: E731
    xy, h, s = dev(ns.xy), dev(ns.h), dev(ns.s)
    op = lb.build_wall_operator(xy, h, s, ns.Lx, ns.Ly, 6, 4, dev(cols, torch.int32), dev(normals), 1.7,
                                periodic=(True, False), check=True)
    op["s"] = s
    ph = lb.Phys(400.0, ns.Ly / 10.0, 0.8, 0.0)
    t = xy[:, 1] / ns.Ly
    x = 2 * np.pi * xy[:, 0] / ns.Lx
    q = torch.stack([0.01 * torch.sin(x), 4 * t * (1 - t), 0.01 * torch.sin(np.pi * t) * torch.cos(x)]).contiguous()
    q[1:, dev(cols[:, 0], torch.int64)] = 0.0
    out = []
    for o in (op, _plain_rows(op)):
        plan = lb.Plan(o["row_ptr"], o["col"], o["w"], o["kappa"], s, dtype=torch.float64)
        plan.set_walls(dev(cols[:, 0], torch.int32), dev(normals))
        dt = float(lb.stable_dt(plan, q, s, 20.0, ph.mu).item())
        out.append([lb.rhs(plan, q, ph), lb.rk_step(plan, q.clone(), dt, 5, ph)])
        plan.close()
    for a, b in zip(*out):
        assert torch.isfinite(b).all() and _close(b, a)


@pytest.mark.parametrize("n", [32, 64, 128, 256])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_the_largest_low_sums_do_not_overflow(lb, n, sign):
    # digits at their largest and all products of one sign: weights 1 - 2^-53, differences
    # with a high digit of 2^29 - 1 and the largest low digit, rows of 64 entries a lane and more
    N = n + 1
    rp = np.concatenate([[0], np.full(N, n).cumsum()]).astype(np.int32)
    col = np.concatenate([[j for j in range(N) if j != i] for i in range(N)]).astype(np.int32)
    w = np.full((6, len(col)), sign * (1 - 2.0 ** -53))
    q = np.full((3, N), 1 - 2.0 ** -30 - 2.0 ** -50)
    q[0] = 0.0
    q[1:, 0] = 0.0
    plan = _plan(lb, rp, col, w, np.ones(N))
    plan.set_launch(2, 128)
    _check(lb, plan, rp, col, w, np.ones(N), q)
    q[0] = q[1]
    _check(lb, plan, rp, col, w, np.ones(N), q)
    plan.close()


@pytest.mark.parametrize("side", [140, 250])
@pytest.mark.parametrize("walls", [False, True])
def test_same_bits_from_every_form_of_the_kernels(lb, side, walls):
    # a small instance alone (one wave, gathering ahead) and beside one that makes the launch
    # take the 96- and the 128-register form
    if walls:
        ns = li.channel(24, 20, m=6, jitter=0.1, seed=4)
        cols, normals = li.channel_walls(ns)
        dev = lambda a, t=torch.float64: torch.tensor(np.ascontiguousarray(a), dtype=t, device="cuda")  # noqa: E731
        s = dev(ns.s)
        a = lb.build_wall_operator(dev(ns.xy), dev(ns.h), s, ns.Lx, ns.Ly, 6, 4, dev(cols, torch.int32), dev(normals),
                                   1.7, periodic=(True, False), check=True)
        a["s"] = s
    else:
        ns, a = _lattice_operator(lb, 24, 21, 6, 5)
    big, b = _lattice_operator(lb, side, side, 4, 6)
    alone = lb.Plan.batched([a], dtype=torch.float64)
    both = lb.Plan.batched([a, b], dtype=torch.float64)
    rng = np.random.default_rng(side)
    q = torch.tensor(0.1 * rng.standard_normal((3, ns.N)), device="cuda")
    if walls:
        wn = dev(cols[:, 0], torch.int32)
        q[1:, wn.long()] = 0.0
        for p in (alone, both):
            p.set_walls(wn, dev(normals))
    Q = torch.cat([q, torch.tensor(li.tgv_fields(big.xy, 10.0), device="cuda")], dim=1).contiguous()
    ph, part = lb.Phys(100.0, 0.005), slice(0, ns.N)
    assert torch.equal(lb.rhs(both, Q, ph)[:, part], lb.rhs(alone, q, ph))
    assert torch.equal(lb.filter(both, Q)[:, part], lb.filter(alone, q))
    # stage and recording launches; steps short enough for both instances
    assert torch.equal(lb.rk_step(both, Q.clone(), 1e-5, 3, ph)[:, part], lb.rk_step(alone, q.clone(), 1e-5, 3, ph))
    if not walls:
        rec = []
        for p, x in ((both, Q), (alone, q)):
            lb.enable_adjoint(p)
            x = x.clone()
            X = lb.stage_states(p)
            lb.rk_step_record(p, x, X, 1e-5, ph)
            rec.append((x[:, part], lb.rhs_adjoint(p, x, x, ph)[:, part]))
        assert all(torch.equal(x, y) for x, y in zip(*rec))
    alone.close()
    both.close()
