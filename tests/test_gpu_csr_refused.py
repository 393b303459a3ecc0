"""A malformed graph leaves y as it was, wherever y lies and whichever rows are at fault."""
import pytest

from meshgen import box_graph

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

import paper_2606_14659_gb300 as R  # noqa: E402


def _spoil(G, what, row):
    at = int(G.row_ptr[row])
    if what == "column":
        G.col[at] = G.n + 7
    elif what == "self":
        G.col[at] = row
    elif what == "weight":
        G.weight[at] = 0
    else:  # the rows of its warp are not looked at
        G.row_ptr[row + 1] = at - 1


@pytest.mark.parametrize("what", ["column", "self", "weight", "row_ptr"])
@pytest.mark.parametrize("dims,row", [((5, 1, 1), 2), ((17, 5, 3), 0), ((17, 5, 3), 253),
                                      ((40, 32, 9), 6000)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_refused_graph_leaves_a_device_vector(what, dims, row, dtype):
    G = R.graph(box_graph(*dims))
    x = torch.randn(G.n, dtype=dtype, device="cuda")
    y = torch.randn(G.n, dtype=dtype, device="cuda")
    y[0] = float("nan")
    was, xwas = y.clone(), x.clone()
    good = R.rsb_laplacian_apply(G, x)
    _spoil(G, what, row)
    with pytest.raises(R.RSBError) as err:
        R.rsb_laplacian_apply(G, x, y)
    assert err.value.code == R.rsb.RSB_EINVAL
    assert torch.equal(y[1:], was[1:]) and bool(y[0].isnan())
    with pytest.raises(R.RSBError):
        R.rsb_laplacian_apply(G, x, x)  # in place
    assert torch.equal(x, xwas)
    H = R.graph(box_graph(*dims))
    R.rsb_laplacian_apply(H, x, y)
    assert torch.equal(y, good)
