"""What the library and the binding hold on to between calls."""
import numpy as np
import pytest

from meshgen import box_graph

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

import paper_2606_14659_gb300 as R  # noqa: E402


def _hexes(nx, ny, nz):
    e = torch.arange(nx * ny * nz, device="cuda")
    i, j, k = e % nx, (e // nx) % ny, e // (nx * ny)
    corner = [(i + a) + (nx + 1) * ((j + b) + (ny + 1) * (k + c))
              for c in (0, 1) for b in (0, 1) for a in (0, 1)]
    return torch.stack(corner, 1).contiguous()


@pytest.mark.parametrize("dims", [(2, 1, 1), (30, 20, 1), (41, 33, 23), (64, 64, 64), (500, 400, 1)])
def test_dual_graph_views_hold_little_more(dims):
    n, rp, col, w = R.rsb.rsb_dual_graph(_hexes(*dims))
    for t in (col, w):
        held = t.untyped_storage().nbytes() // 4
        assert held - t.numel() <= max(t.numel() // 8, 1 << 16)


def test_a_partition_takes_the_dual_graphs_room():
    """With little memory left, a partition gets what the gather-scatter calls keep."""
    g = box_graph(128, 96, 64)
    G = R.graph(g)
    opts = R.options(precision="mixed", degenerate_policy="none", max_restarts=3, polish_cycles=1)

    def free():
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        return torch.cuda.mem_get_info()[0]

    R.rsb_partition(R.graph(box_graph(9, 5, 3)), 2, opts)  # the context itself
    R.rsb_release()
    before = free()
    ref = R.rsb_partition(G, 2, opts)[0]
    need = before - free()
    R.rsb_release()
    before = free()
    R.rsb.rsb_dual_graph(_hexes(200, 160, 128))
    held = before - free()
    left = need // 4
    assert held > need, "the test's sizes: the held room has to be what the partition takes"
    hog = torch.empty(free() - left, dtype=torch.uint8, device="cuda")
    try:
        got = R.rsb_partition(G, 2, opts)[0]
        assert torch.equal(got, ref)
        ev = _hexes(8, 4, 4)
        n, rp, col, w = R.rsb.rsb_dual_graph(ev)  # and the next of those calls is as usual
        assert int(rp[-1]) == len(col)
    finally:
        del hog
        torch.cuda.empty_cache()
        R.rsb_release()
    assert np.array_equal(np.bincount(ref.cpu().numpy()), [g.n // 2, g.n - g.n // 2])


def test_dual_graph_on_the_host_without_the_large_room(monkeypatch):
    """The host allocator's refusal is a plain RuntimeError; the exact room is taken then."""
    ev = _hexes(6, 5, 4)
    want = R.rsb.rsb_dual_graph(ev.cpu().numpy(), device="host")
    empty = torch.empty

    def small(n, **kw):
        if n >= 26 * len(ev):
            raise RuntimeError("DefaultCPUAllocator: can't allocate memory")
        return empty(n, **kw)

    monkeypatch.setattr(torch, "empty", small)
    got = R.rsb.rsb_dual_graph(ev.cpu().numpy(), device="host")
    assert got[0] == want[0] and all(torch.equal(a, b) for a, b in zip(got[1:], want[1:]))
