"""Ritz vectors and the thick-restart basis for every number of kept vectors.

The kernel that forms y = Q s_0 and the kept vectors sums a basis vector into 1, 9
or 17 outputs at a time, several rows per thread; the sizes below leave rows and
outputs over at each of them.  In FP64 the returned pair must meet the solver's own
stopping test when the oracle's Laplacian is applied to it (1e-10 d_max, plus the
rounding of that product, below 1e-13 d_max); in mixed precision the resident
launch, the per-cycle graphs and the plain launches must agree bit for bit.
"""
import numpy as np
import pytest

import oracle as O
from meshgen import box_graph_deleted

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

import paper_2606_14659_gb300 as R  # noqa: E402

MESHES = [box_graph_deleted(7, 5, 4, 0.05, 3, "vertex"),
          box_graph_deleted(13, 9, 7, 0.1, 5, "vertex"),
          box_graph_deleted(19, 11, 7, 0.1, 7, "vertex")]


@pytest.mark.parametrize("g", MESHES, ids=lambda g: str(g.n))
@pytest.mark.parametrize("keep,krylov", [(0, 40), (1, 9), (7, 40), (8, 23), (9, 40), (16, 40)])
def test_ritz_vectors_for_every_keep(g, keep, krylov):
    G = R.graph(g)
    for mode in (0, 2, 3):
        # restarts of few steps converge slowly: the cap is not what is tested here
        o = R.options(keep=keep, krylov_dim=krylov, use_graph=mode, max_restarts=2000)
        lam, v, _, code = R.rsb_fiedler(G, o)
        assert code == 0
        v = v.cpu().numpy()
        dmax = O.degree(g).max()
        assert np.linalg.norm(O.laplacian_apply(g, v) - lam * v) <= (1e-10 + 1e-13) * dmax


@pytest.mark.parametrize("g", MESHES, ids=lambda g: str(g.n))
@pytest.mark.parametrize("keep,krylov", [(0, 40), (7, 40), (8, 23), (16, 40)])
def test_launch_modes_agree_for_every_keep(g, keep, krylov):
    G = R.graph(g)
    got = []
    for mode in (0, 1, 3):
        o = R.options(precision="mixed", keep=keep, krylov_dim=krylov, use_graph=mode)
        lam, v, _, _ = R.rsb_fiedler(G, o)
        got.append((lam, v))
    for lam, v in got[1:]:
        assert lam == got[0][0] and torch.equal(v, got[0][1])
