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
