"""Connected components, validation and coordinate bisection without the graph.

Components start from every row's first neighbour and are flattened by pointer jumping
before the edges are hooked, so the cases are long chains in an unfavourable order, many
components of every size around a warp and a CTA, and isolated rows.  The contrast
vector of a disconnected graph shows the component of the smallest gid exactly.
Malformed graphs are refused by every method; the check reads coalesced entries whose
rows it finds by their starts, so the fault is put at the edges of warps and CTAs.
"""
import numpy as np
import pytest

from meshgen import DualGraph, box_graph

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

import paper_2606_14659_gb300 as R  # noqa: E402


def _paths(sizes, seed, order):
    """Disjoint paths; rows in path order, reversed or shuffled; random gids."""
    n = int(sum(sizes))
    rng = np.random.default_rng(seed)
    rows = {"path": np.arange(n), "reversed": np.arange(n)[::-1], "shuffled": rng.permutation(n)}[order]
    nb = [[] for _ in range(n)]
    comp = np.empty(n, dtype=np.int64)
    at = 0
    for c, s in enumerate(sizes):
        for i in range(s):
            comp[rows[at + i]] = c
            if i:
                u, v = int(rows[at + i]), int(rows[at + i - 1])
                nb[u].append(v)
                nb[v].append(u)
        at += s
    col = np.array([c for r in nb for c in sorted(r)], dtype=np.int32)
    rp = np.concatenate([[0], np.cumsum([len(r) for r in nb])]).astype(np.int64)
    gid = rng.choice(1 << 40, n, replace=False).astype(np.int64)
    return DualGraph(n, rp, col, np.ones(len(col), np.int32), gid), comp


@pytest.mark.parametrize("order", ["path", "reversed", "shuffled"])
@pytest.mark.parametrize("sizes", [[2], [255, 1], [256, 256, 3], [5000, 1], [1] * 600,
                                   [300, 1, 31, 32, 33, 700, 2]], ids=str)
def test_components(sizes, order):
    g, comp = _paths(sizes, len(sizes), order)
    lam, v, res, code = R.rsb_fiedler(R.graph(g), R.options(max_restarts=1))
    if len(sizes) == 1:
        assert code != R.rsb.RSB_EDISCONNECTED
        return
    if sizes == [1] * 600:
        g.col = np.zeros(1, np.int32)[:0]
    assert code == R.rsb.RSB_EDISCONNECTED and lam == 0.0
    inside = comp == comp[np.argmin(g.gid)]
    v = v.cpu().numpy()
    # one value on the component, one of the other sign everywhere else
    assert len(np.unique(v[inside])) == 1 and len(np.unique(v[~inside])) == 1
    assert v[inside][0] * v[~inside][0] < 0


@pytest.mark.parametrize("row", [0, 31, 32, 255, 256, 300])
@pytest.mark.parametrize("what", ["column", "negative", "self", "weight0", "weight8", "row_ptr"])
@pytest.mark.parametrize("method", ["lanczos", "rcb"])
def test_malformed_graphs_are_refused(row, what, method):
    g = box_graph(43, 7, 1, "vertex")  # 301 rows
    G = R.graph(g)
    p = int(g.row_ptr[row])
    last = int(g.row_ptr[row + 1]) - 1
    if what == "column":
        G.col[last] = g.n
    elif what == "negative":
        G.col[p] = -1
    elif what == "self":
        G.col[last] = row
    elif what == "weight0":
        G.weight[p] = 0
    elif what == "weight8":
        G.weight[last] = 8
    else:
        G.row_ptr[row] = -1 if row == 0 else int(g.row_ptr[row - 1]) - 1
    with pytest.raises(R.RSBError) as err:
        R.rsb_partition(G, 2, R.options(method=method))
    assert err.value.code == R.rsb.RSB_EINVAL
