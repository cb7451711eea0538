"""The neighbour search against the definition (every pair tested in FP64), at the
edges of its row sort, of its cell list and of its FP32 pre-test."""
import numpy as np
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


def _brute(xy, h, Lx, Ly, periodic):
    """Rows of |r_ji|^2 <= (2 h_i)^2 with separately rounded products and sums (numpy)."""
    rows = []
    for i in range(len(xy)):
        d = xy - xy[i]
        for a, L in ((0, Lx), (1, Ly)):
            if periodic[a]:
                v = d[:, a]
                d[:, a] = np.where(v > 0.5 * L, v - L, np.where(v < -0.5 * L, v + L, v))
        near = d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1] <= (2.0 * h[i]) * (2.0 * h[i])
        near[i] = False
        rows.append(np.nonzero(near)[0])
    return np.concatenate([[0], np.cumsum([len(r) for r in rows])]), np.concatenate(rows)


def _cases():
    rng = np.random.default_rng(9)
    lat = lambda n, L: (np.stack(np.meshgrid(np.arange(n), np.arange(n)), -1).reshape(-1, 2) + 0.5) * (L / n)  # noqa: E731
    u = rng.uniform(size=(700, 2))
    both, none = (True, True), (False, False)
    yield "radius_on_the_lattice", lat(24, 1.0), np.full(576, 1.0 / 24), 1.0, 1.0, both
    # rows of 57 .. 513 entries: every size class of the row sort, and past the last one
    for n in (64, 65, 128, 129, 256, 257, 512, 513, 514):
        yield f"rows_of_{n - 1}", u[:n], np.full(n, 2.0), 1.0, 1.0, none
    yield "rows_of_mixed_length", u, rng.uniform(0.02, 0.6, 700), 1.0, 1.0, both
    yield "mixed_h_bounded", u, np.exp(rng.uniform(-7, -1, 700)), 1.0, 1.0, (True, False)
    yield "narrow_box", u * [1e-3, 50.0], np.full(700, 0.1), 1e-3, 50.0, both
    yield "flat_box", u * [300.0, 1e-2], np.full(700, 0.5), 300.0, 1e-2, (False, True)
    yield "cluster_in_a_huge_box", 0.5e9 + u, np.full(700, 0.05), 1e9, 1e9, both
    yield "on_the_walls", np.concatenate([u[:200], [[0, 0], [1, 1], [0, 1], [1, 0], [1, 0.5]]]), np.full(205, 0.1), 1.0, 1.0, none
    yield "tiny_scale", u * 1e-20, np.full(700, 3e-22), 1e-20, 1e-20, both
    yield "huge_h", u[:50], np.full(50, 1e200), 1.0, 1.0, none
    yield "two_nodes", u[:2], np.full(2, 0.3), 1.0, 1.0, both


@pytest.mark.parametrize("case", list(_cases()), ids=lambda c: c[0])
def test_rows_are_the_definition(lb, case):
    _, xy, h, Lx, Ly, periodic = case
    rp, col = _brute(np.array(xy, dtype=np.float64), h, Lx, Ly, periodic)
    # one double off the 16-byte boundary as well: the search reads scalars
    for off in (0, 1):
        buf = torch.empty(2 * len(xy) + off, dtype=torch.float64, device="cuda")
        t = buf[off:].view(-1, 2)
        t.copy_(torch.tensor(np.ascontiguousarray(xy)))
        got_rp, got = lb.build_stencils(t, torch.tensor(h, device="cuda"), Lx, Ly, periodic=periodic)
        assert np.array_equal(got_rp.cpu().numpy(), rp)
        assert np.array_equal(got.cpu().numpy(), col)


def test_search_on_another_stream(lb):
    rng = np.random.default_rng(3)
    xy, h = rng.uniform(size=(5000, 2)), np.full(5000, 0.03)
    t, ht = torch.tensor(xy, device="cuda"), torch.tensor(h, device="cuda")
    torch.cuda.synchronize()
    rp, col = lb.build_stencils(t, ht, 1.0, 1.0)
    s = torch.cuda.Stream()
    for _ in range(3):
        rp2, col2 = lb.build_stencils(t, ht, 1.0, 1.0, stream=s)
        s.synchronize()
        assert torch.equal(rp, rp2) and torch.equal(col, col2)


def test_search_on_another_stream_beside_work_on_freed_blocks(lb):
    # blocks of the search's sizes, freed with a write of the current stream still to come: the
    # search on the other stream takes none of them, for its cell list or for its results
    rng = np.random.default_rng(4)
    N = 5000
    t, ht = torch.tensor(rng.uniform(size=(N, 2)), device="cuda"), torch.tensor(np.full(N, 0.03), device="cuda")
    rp, col = lb.build_stencils(t, ht, 1.0, 1.0)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(3):
        blocks = [torch.empty(n, dtype=torch.uint8, device="cuda")
                  for n in (int(lb.lib.labfm_stencil_work_bytes(N)), 4 * (N + 1), 4 * len(col))]
        torch.cuda._sleep(20_000_000)
        for b in blocks:
            b.fill_(255)
        del b, blocks
        rp2, col2 = lb.build_stencils(t, ht, 1.0, 1.0, stream=s)
        torch.cuda.synchronize()
        assert torch.equal(rp, rp2) and torch.equal(col, col2)
