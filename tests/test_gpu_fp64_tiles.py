"""FP64 Fiedler pairs at the edges of the one-row tiles: from more than one tile of two rows
to as many tiles of one row as the chip has SMs.  The launch modes share the tiles and give
the same bits; the residual is the solver's tolerance and the rounding of the check."""
import numpy as np
import pytest

import oracle as O
from meshgen import box_graph

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

import paper_2606_14659_gb300 as R  # noqa: E402


@pytest.mark.parametrize("dims", [(8, 8, 8), (27, 19, 1), (64, 38, 16), (109, 51, 7)],
                         ids=["512", "513", "38912", "38913"])
def test_fp64_pair_at_the_edges_of_one_row_tiles(dims):
    g = box_graph(*dims)
    G = R.graph(g)
    got = [R.rsb_fiedler(G, R.options(precision="fp64", use_graph=m)) for m in (0, 1, 3)]
    for lam, v, _, code in got:
        assert code == 0 and lam == got[0][0] and torch.equal(v, got[0][1])
    lam, v = got[0][0], got[0][1].cpu().numpy()
    dmax = O.degree(g).max()
    assert np.linalg.norm(O.laplacian_apply(g, v) - lam * v) <= (1e-10 + 1e-13) * dmax
