"""Meshes that the slot table does not hold, and rows too long for the merged buffer.

The buckets take over from what the table's pass over the ids left (its counts, or the
largest id); an element of 33 to 56 neighbours is merged straight into CSR.  References:
the dense product of the element-vertex incidence, small integers throughout, so graphs
agree exactly; the Laplacian of integer-valued vectors is exact too.
"""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

import paper_2606_14659_gb300 as R  # noqa: E402

RNG = np.random.default_rng(11)


def _cap(ne):
    return 2 * ne + 4096  # ids the table is laid out for


def _dealt(ne, nv, share):
    """Every vertex column deals the elements to vertices of `share` elements."""
    per = (ne + share - 1) // share
    return np.stack([RNG.permutation(ne) // share + c * per for c in range(nv)], 1)


def _with(ev, e, a, vid):
    ev = ev.copy()
    ev[e, a] = vid
    return ev


BASE = _dealt(300, 4, 5)
MESHES = {
    "valence8": _dealt(200, 5, 8),
    "valence9": _dealt(200, 5, 9),
    "valence24": _dealt(1000, 4, 24),
    "valence9_at_the_last_id": np.concatenate([BASE, np.column_stack(
        [np.full(9, _cap(309) - 1), 2000 + np.arange(27).reshape(9, 3)])]),
    "id_below_cap": _with(BASE, 7, 1, _cap(300) - 1),
    "id_at_cap": _with(BASE, 7, 1, _cap(300)),
    "id_far": _with(BASE, 299, 3, 1 << 24),
    "ids_far": BASE + (1 << 22),
    "valence9_and_far": _with(_dealt(200, 5, 9), 3, 0, 1 << 21),
    "rows33": _dealt(400, 5, 8),
    "rows56": _dealt(900, 8, 8),
    "rows56_one": np.concatenate([np.arange(8 * 300).reshape(300, 8) + 8,
                                  _dealt(64, 8, 8) + 3000]),
}


def _brute(ev):
    _, inv = np.unique(ev, return_inverse=True)
    q = np.zeros((len(ev), inv.max() + 1), np.int64)
    np.add.at(q, (np.arange(len(ev)).repeat(ev.shape[1]), inv.reshape(-1)), 1)
    return q


@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("odd", [False, True])
def test_dual_graph(name, odd):
    ev = MESHES[name].astype(np.int64)
    q = _brute(ev)
    a = (q @ q.T)
    np.fill_diagonal(a, 0)
    buf = torch.empty(ev.size + 1, dtype=torch.int64, device="cuda")
    buf[odd:odd + ev.size] = torch.from_numpy(ev).reshape(-1)
    arg = buf[odd:odd + ev.size].view(ev.shape)
    lib = R.rsb.load()
    ne, nv = ev.shape
    rp = torch.empty(ne + 1, dtype=torch.int64, device="cuda")
    nnz = C.c_int64(0)
    code = lib.rsb_dual_graph(ne, nv, arg.data_ptr(), rp.data_ptr(), None, None, 0, C.byref(nnz), None)
    if a.max() > 7:
        assert code == R.rsb.RSB_EINVAL
        with pytest.raises(R.RSBError):
            R.rsb.rsb_dual_graph(arg)
        return
    assert code == 0 and nnz.value == np.count_nonzero(a)
    counted = rp.clone()
    n, rp, col, w = R.rsb.rsb_dual_graph(arg)
    assert torch.equal(rp, counted)
    rows, cols = np.nonzero(a)
    assert np.array_equal(rp.cpu().numpy(), np.concatenate([[0], np.cumsum((a > 0).sum(1))]))
    assert np.array_equal(col.cpu().numpy(), cols)
    assert np.array_equal(w.cpu().numpy(), a[rows, cols])


@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_laplacian_of_integers(name, dtype):
    ev = MESHES[name].astype(np.int64)
    q = _brute(ev)
    x = RNG.integers(-50, 50, len(ev))
    want = (q * q.sum(0)).sum(1) * x - q @ (q.T @ x)
    y = R.rsb.rsb_laplacian_apply_gs(torch.from_numpy(ev).cuda(), torch.from_numpy(x).cuda().to(dtype))
    assert np.array_equal(y.double().cpu().numpy(), want)
