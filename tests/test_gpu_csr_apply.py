"""y = L x straight from CSR against the sliced-ELL path.

rsb_laplacian_apply sums every row in entry order from the caller's CSR; the
allocation-free entry point builds the sliced form and sums it in the same order, so
FP64 results must be equal bit for bit.  FP32 is held to the oracle: each of the d_r
products and sums of a row rounds once, so |error| <= 2 (K + 2) eps32 d_r max|x|.
Sizes: around a warp (32 rows), a CTA (256 rows) and the 1024 entries a warp stages at
a time; empty rows; weights given and not.
"""
import numpy as np
import pytest

import oracle as O
from meshgen import DualGraph, box_graph, box_graph_deleted

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

import paper_2606_14659_gb300 as R  # noqa: E402


def _edges(n, edges, w):
    a = np.array([(u, v, x) for (u, v), x in zip(edges, w)] +
                 [(v, u, x) for (u, v), x in zip(edges, w)], dtype=np.int64).reshape(-1, 3)
    a = a[np.lexsort((a[:, 1], a[:, 0]))]
    rp = np.zeros(n + 1, dtype=np.int64)
    np.add.at(rp, a[:, 0] + 1, 1)
    return DualGraph(n, np.cumsum(rp), a[:, 1].astype(np.int32), a[:, 2].astype(np.int32),
                     np.arange(n, dtype=np.int64))


def _star(n):
    return _edges(n, [(0, i) for i in range(1, n)], [1 + i % 7 for i in range(1, n)])


GRAPHS = [_edges(1, [], []), _edges(40, [(3, 35)], [5]), box_graph(31, 1, 1), box_graph(32, 1, 1),
          box_graph(33, 1, 1), box_graph(257, 1, 1), box_graph(16, 16, 1), box_graph(17, 5, 3),
          box_graph_deleted(13, 11, 7, 0.3, 5, "vertex"), _star(1024), _star(1026), _star(3000)]


@pytest.mark.parametrize("g", GRAPHS, ids=lambda g: f"{g.n}-{g.nnz}")
@pytest.mark.parametrize("where", ["cuda", "host"])
def test_csr_apply_equals_sliced_form(g, where):
    rng = np.random.default_rng(g.n)
    x = rng.standard_normal(g.n)
    G = R.graph(g, device=where)
    xt = torch.from_numpy(x).cuda() if where == "cuda" else x
    y = R.rsb_laplacian_apply(G, xt)
    y = y.cpu().numpy() if where == "cuda" else y
    xd = torch.from_numpy(x).cuda()
    ref = torch.empty_like(xd)
    assert R.rsb.rsb_laplacian_apply_noalloc(R.graph(g), xd, ref) == 0
    assert np.array_equal(y, ref.cpu().numpy())
    y32 = R.rsb_laplacian_apply(R.graph(g), xd.float()).cpu().numpy()
    x32 = x.astype(np.float32).astype(np.float64)
    deg = O.degree(g)
    k = np.diff(g.row_ptr)
    bound = 2 * (k + 2) * 2.0 ** -24 * deg * max(np.abs(x32).max(), 1e-30)
    assert np.all(np.abs(y32 - O.laplacian_apply(g, x32)) <= bound)


def test_unit_weights_when_weight_is_null():
    g = box_graph(17, 5, 3)
    G = R.graph(g)
    H = R.Graph(G.n, G.row_ptr, G.col, None, None, "cuda")
    x = torch.randn(g.n, dtype=torch.float64, device="cuda")
    assert torch.equal(R.rsb_laplacian_apply(G, x), R.rsb_laplacian_apply(H, x))


@pytest.mark.parametrize("what", ["column", "self", "weight0", "weight8", "row_ptr", "row_ptr0"])
def test_malformed_graphs_are_refused(what):
    G = R.graph(box_graph(17, 5, 3))
    x = torch.randn(G.n, dtype=torch.float64, device="cuda")
    if what == "column":
        G.col[5] = G.n
    elif what == "self":
        G.col[int(G.row_ptr[9])] = 9
    elif what == "weight0":
        G.weight[100] = 0
    elif what == "weight8":
        G.weight[-1] = 8
    elif what == "row_ptr":
        G.row_ptr[40] = G.row_ptr[39] - 1
    else:
        G.row_ptr[0] = 1
    for xx in (x, x.float()):
        with pytest.raises(R.RSBError) as err:
            R.rsb_laplacian_apply(G, xx)
        assert err.value.code == R.rsb.RSB_EINVAL
    ok = R.graph(box_graph(17, 5, 3))  # the next call is clean
    assert torch.isfinite(R.rsb_laplacian_apply(ok, x)).all()


def test_refused_graph_leaves_a_host_vector():
    g = box_graph(17, 5, 3)
    G = R.graph(g, device="host")
    G.weight[100] = 0
    y = np.full(g.n, 3.5)
    with pytest.raises(R.RSBError):
        R.rsb_laplacian_apply(G, np.ones(g.n), y)
    assert np.all(y == 3.5)
