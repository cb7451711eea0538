"""F32 stages and filters that keep several chunks of a row in flight (plans whose warps
fit on the GPU at once): the same bits as the work-queue stage and the grid-stride filter,
which read a row chunk by chunk, on both sides of every line of the rule that picks the
number of chunks, for every number of lanes, over consecutive steps."""
import pytest

import labfm_inputs as li

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

C, MU = 10.0, 0.005


@pytest.fixture(scope="module")
def lb():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import __graft_entry__ as g
    g.build()
    import paper_2102_02019_gb300 as lb
    return lb


# at 4 lanes: 1 warp an SM, and either side of 8, 12, 16 and 56 warps an SM
@pytest.mark.parametrize("nx,ny,m", [(11, 9, 4), (37, 29, 8), (99, 98, 4), (101, 97, 4), (121, 120, 4), (123, 121, 6),
                                     (140, 138, 4), (141, 139, 4), (262, 259, 4), (262, 261, 4)])
def test_same_bits_as_chunk_by_chunk(lb, nx, ny, m):
    ns = li.tgv_lattice(nx, ny, m=m, jitter=0.3, seed=nx + ny)
    xy, h, s = (torch.tensor(a, device="cuda") for a in (ns.xy, ns.h, ns.s))
    rp, col = lb.build_stencils(xy, h, ns.Lx, ns.Ly)
    wb = lb.build_weights(xy, h, s, ns.Lx, ns.Ly, rp, col, m, residual=False)
    plan = lb.Plan(rp, col, wb["w"], wb["kappa"], s, dtype=torch.float32)
    q0 = torch.tensor(li.tgv_fields(ns.xy, C), dtype=torch.float32, device="cuda")
    dt = float(lb.stable_dt(plan, q0, s, C, MU).item())
    for group in (2, 4, 8, 16, 32):
        plan.set_launch(group, 128)
        plan.set_staging(0)
        out = []
        for chunked in (True, False):
            plan.set_persistent(chunked)
            plan.set_filter_launch(0, chunked)
            Q = q0.clone()
            lb.rk_step(plan, Q, dt, 3, lb.Phys(C * C, MU))
            assert plan.device_status() == 0
            out.append(Q)
        assert torch.isfinite(out[0]).all()
        assert torch.equal(out[0], out[1]), group
    plan.close()


def _lattice(lb, nx, ny, m, seed):
    ns = li.tgv_lattice(nx, ny, m=m, jitter=0.1, seed=seed)
    xy, h, s = (torch.tensor(a, device="cuda") for a in (ns.xy, ns.h, ns.s))
    rp, col = lb.build_stencils(xy, h, ns.Lx, ns.Ly)
    wb = lb.build_weights(xy, h, s, ns.Lx, ns.Ly, rp, col, m, residual=False)
    return ns, {"row_ptr": rp, "col": col, "w": wb["w"], "kappa": wb["kappa"], "s": s}


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("side", [15, 60])
def test_recording_and_walls_same_bits_as_past_the_line(lb, walls, side):
    # an instance alone (chunks ahead) and beside a lattice of 70,200 nodes, with which the
    # launches read chunk by chunk: steps with and without walls, and recorded steps with the
    # reverse sweep over what they recorded
    if walls:
        ns = li.channel(side + 5, side, m=6, jitter=0.1, seed=4)
        cols, normals = li.channel_walls(ns)
        dev = lambda a, t=torch.float64: torch.tensor(a.copy(), dtype=t, device="cuda")  # noqa: E731
        s = dev(ns.s)
        a = lb.build_wall_operator(dev(ns.xy), dev(ns.h), s, ns.Lx, ns.Ly, 6, 4, dev(cols, torch.int32), dev(normals),
                                   1.7, periodic=(True, False), check=True)
        a["s"] = s
    else:
        ns, a = _lattice(lb, side, side + 3, 6, 5)
    big, b = _lattice(lb, 270, 260, 4, 6)
    alone = lb.Plan.batched([a], dtype=torch.float32)
    both = lb.Plan.batched([a, b], dtype=torch.float32)
    g = torch.Generator().manual_seed(side)
    q = (0.1 * torch.randn((3, ns.N), generator=g)).cuda()
    if walls:
        wn = dev(cols[:, 0], torch.int32)
        q[1:, wn.long()] = 0.0
        for p in (alone, both):
            p.set_walls(wn, dev(normals))
    Q = torch.cat([q, torch.tensor(li.tgv_fields(big.xy, C), dtype=torch.float32, device="cuda")], dim=1).contiguous()
    ph, dt = lb.Phys(C * C, MU), 1e-5
    assert torch.equal(lb.rk_step(both, Q.clone(), dt, 3, ph)[:, :ns.N], lb.rk_step(alone, q.clone(), dt, 3, ph))
    if not walls:
        out = []
        for p, x in ((both, Q), (alone, q)):
            lb.enable_adjoint(p)
            z = x.clone()
            X = lb.stage_states(p)
            lb.rk_step_record(p, z, X, dt, ph)
            lam = x.clone()
            lb.rk_step_adjoint_recorded(p, X, lam, dt, ph)
            out.append((z[:, :ns.N], lam[:, :ns.N]))
        assert torch.isfinite(out[0][1]).all()
        assert all(torch.equal(x, y) for x, y in zip(*out))
    alone.close()
    both.close()
