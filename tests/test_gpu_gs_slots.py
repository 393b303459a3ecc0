"""The slot table of the gather-scatter kernels against brute force and the bucket path.

A mesh whose vertices have at most eight elements, whose elements have at most 32
neighbours and whose ids lie below 2 ne + 4096 is answered from the slot table; the
others from the sorted buckets.  Both sum a vertex's elements in ascending order, so a
mesh gives the same bits whether its ids fit the table or (shifted by 2^20) do not.  The
dual graph is integer work and must equal brute force entry for entry.
"""
import numpy as np
import pytest

from meshgen import box_graph, box_graph_deleted

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

import paper_2606_14659_gb300 as R  # noqa: E402


def _random(ne, nv, nvert, seed):
    rng = np.random.default_rng(seed)
    return np.stack([rng.choice(nvert, nv, replace=False) for _ in range(ne)]).astype(np.int64)


def _grid(nx, ny, nv):  # nv = 2: the edges of a path, 4: quads
    if nv == 2:
        return np.array([[i, i + 1] for i in range(nx)], dtype=np.int64)
    q = [[i + (nx + 1) * j, i + 1 + (nx + 1) * j, i + (nx + 1) * (j + 1), i + 1 + (nx + 1) * (j + 1)]
         for j in range(ny) for i in range(nx)]
    return np.array(q, dtype=np.int64)


MESHES = {
    "one": np.arange(8, dtype=np.int64).reshape(1, 8),
    "hex33": box_graph(33, 1, 1).hex_vertices(),
    "hex": box_graph(9, 7, 5).hex_vertices(),
    "hexdel": box_graph_deleted(17, 13, 9, 0.2, 3, "vertex").hex_vertices(),
    "path": _grid(300, 1, 2),
    "quads": _grid(17, 16, 4),
    "fan8": np.array([[0, 1 + 2 * i, 2 + 2 * i] for i in range(8)], dtype=np.int64),
    "fan9": np.array([[0, 1 + 2 * i, 2 + 2 * i] for i in range(9)], dtype=np.int64),
    "nv1": np.arange(40, dtype=np.int64).reshape(40, 1) // 3,
    "nv7": _random(60, 7, 400, 1),
    "many": _random(64, 8, 80, 2),  # more than 32 neighbours, vertices of few elements
    "twice": np.array([[0, 1, 1, 2], [1, 2, 3, 4], [4, 5, 6, 6]], dtype=np.int64),
}


def _brute(ev):
    ne = len(ev)
    m = np.zeros((ne, int(ev.max()) + 1), dtype=np.int64)
    np.add.at(m, (np.arange(ne)[:, None], ev), 1)
    a = m @ m.T
    np.fill_diagonal(a, 0)
    return a


@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("shift", [0, 1 << 20])
@pytest.mark.parametrize("where", ["cuda", "odd", "host"])
def test_dual_graph_against_brute_force(name, shift, where):
    ev = MESHES[name]
    a = _brute(ev)
    arg = ev + shift
    if where == "odd":  # ids that start 8 bytes off a 16-byte boundary
        buf = torch.empty(ev.size + 1, dtype=torch.int64, device="cuda")
        buf[1:] = torch.from_numpy(arg).reshape(-1)
        arg = buf[1:].view(ev.shape)
        assert arg.data_ptr() % 16 == 8
    if a.max() > 7:
        with pytest.raises(R.RSBError):
            R.rsb.rsb_dual_graph(arg, device="host" if where == "host" else "cuda")
        return
    n, rp, col, w = R.rsb.rsb_dual_graph(arg, device="host" if where == "host" else "cuda")
    rp, col, w = rp.cpu().numpy(), col.cpu().numpy(), w.cpu().numpy()
    assert n == len(ev) and rp[0] == 0 and rp[-1] == len(col) == len(w)
    for e in range(n):
        nb = np.nonzero(a[e])[0]
        assert np.array_equal(col[rp[e]:rp[e + 1]], nb), e
        assert np.array_equal(w[rp[e]:rp[e + 1]], a[e][nb]), e


@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("f32", [False, True])
def test_laplacian_slots_equal_buckets(name, f32):
    ev = torch.from_numpy(MESHES[name]).cuda()
    rng = np.random.default_rng(4)
    x = rng.standard_normal(len(ev))
    xt = torch.from_numpy(x).cuda()
    xt = xt.float() if f32 else xt
    y = R.rsb.rsb_laplacian_apply_gs(ev, xt)
    assert torch.equal(y, R.rsb.rsb_laplacian_apply_gs(ev + (1 << 20), xt))
    a = _brute(MESHES[name]).astype(np.float64)
    xr = xt.double().cpu().numpy()
    ref = a.sum(1) * xr - a @ xr
    # vertex sums of up to nv x 9 terms, nv vertex terms: 2 (9 + nv) roundings of d max|x|
    eps = 2.0 ** -24 if f32 else 2.0 ** -53
    d = (a.sum(1) + np.asarray((MESHES[name] >= 0).sum(1))).max()
    assert np.abs(y.double().cpu().numpy() - ref).max() <= 2 * 17 * eps * 2 * d * np.abs(xr).max()


def test_bad_ids_are_refused_by_both_paths():
    for bad in (-1, 1 << 31):
        ev = torch.from_numpy(MESHES["hex"].copy()).cuda()
        ev[3, 2] = bad
        for call in (lambda: R.rsb.rsb_dual_graph(ev),
                     lambda: R.rsb.rsb_laplacian_apply_gs(ev, torch.ones(len(ev), device="cuda"))):
            with pytest.raises(R.RSBError) as err:
                call()
            assert err.value.code == R.rsb.RSB_EINVAL


@pytest.mark.parametrize("name", ["hex", "fan9", "many"])  # fits; nine at a vertex; many neighbours
@pytest.mark.parametrize("shift", [0, 1 << 20])
def test_laplacian_in_place(name, shift):
    ev = torch.from_numpy(MESHES[name] + shift).cuda()
    x = torch.linspace(-1, 1, len(ev), dtype=torch.float64, device="cuda")
    y = R.rsb.rsb_laplacian_apply_gs(ev, x)
    z = x.clone()
    R.rsb.rsb_laplacian_apply_gs(ev, z, z)
    assert torch.equal(z, y)
    ev[0, 0] = -1  # refused: the vector stays
    z = x.clone()
    with pytest.raises(R.RSBError):
        R.rsb.rsb_laplacian_apply_gs(ev, z, z)
    assert torch.equal(z, x)


@pytest.mark.parametrize("who", ["torch", "library"])
def test_dual_graph_without_the_large_room(who, monkeypatch):
    """Room for 26 neighbours an element refused: the exact room is taken."""
    ev = MESHES["quads"]
    want = R.rsb.rsb_dual_graph(ev)
    if who == "torch":
        empty = torch.empty

        def small(n, **kw):
            if n >= 26 * len(ev):
                raise torch.OutOfMemoryError("no room")
            return empty(n, **kw)

        monkeypatch.setattr(torch, "empty", small)
    else:
        class Lib:
            calls = 0

            def rsb_dual_graph(self, *a):
                Lib.calls += 1
                return R.rsb.RSB_ENOMEM if Lib.calls == 1 else lib.rsb_dual_graph(*a)

        lib = R.rsb.load()
        monkeypatch.setattr(R.rsb, "load", lambda: Lib())
    got = R.rsb.rsb_dual_graph(ev)
    assert got[0] == want[0] and all(torch.equal(a, b) for a, b in zip(got[1:], want[1:]))
