"""The objectives' sums over the nodes, at the edges of their grids."""
import pytest

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


@pytest.mark.parametrize("N", [1, 31, 1024, 1025, 8192, 8193, 16384, 16385, 100003])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_objective_sums_at_every_grid_size(lb, N, dtype):
    # one to sixteen blocks, a ragged last pass; terms of one sign, so that the sum of N
    # terms is within N u of the exact one, u = 2^-53, and exp within 2 u
    g = torch.Generator().manual_seed(N)
    q = (torch.rand((3, N), generator=g, dtype=torch.float64) + 0.1).to(dtype).cuda()
    s, px, py = (torch.rand(N, generator=g, dtype=torch.float64).cuda() + 0.1 for _ in range(3))
    rho, u, v = torch.exp(q[0].double()), q[1].double(), q[2].double()
    for got, ref in ((lb.kinetic_energy(q, s), (0.5 * rho * (u * u + v * v) * s * s).sum()),
                     (lb.probe_momentum(q, px, py), (rho * (px * u + py * v)).sum())):
        assert abs(float(got) - float(ref)) <= (2 * N + 16) * 2.0 ** -53 * float(ref)
    assert torch.equal(lb.kinetic_energy(q, s), lb.kinetic_energy(q, s))
