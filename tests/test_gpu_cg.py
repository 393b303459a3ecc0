"""Inverse iteration: the resident CG launch against the launches per iteration.

Both sum the same rows in the same order, so the launch modes must agree bit for bit:
units of one tile and of several, several units of different sizes at once, parts of a
segment that fell apart, with and without deflation vectors, in both precisions.  The
pair must meet the stopping test with the oracle's Laplacian (FP64: 1e-10 d_max plus
the product's rounding).
"""
import numpy as np
import pytest

import oracle as O
from meshgen import box_graph, box_graph_deleted

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

import paper_2606_14659_gb300 as R  # noqa: E402

MESHES = [box_graph(3, 2, 1), box_graph(16, 8, 1), box_graph(43, 4, 3),
          box_graph_deleted(9, 8, 8, 0.05, 1, "vertex"),
          box_graph_deleted(41, 23, 17, 0.1, 3, "vertex")]


@pytest.mark.parametrize("g", MESHES, ids=lambda g: str(g.n))
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_fiedler_modes_agree(g, prec):
    G = R.graph(g)
    got = [R.rsb_fiedler(G, R.options(method="inverse", precision=prec, use_graph=m))
           for m in (0, 1, 3)]
    for lam, v, res, code in got[1:]:
        assert lam == got[0][0] and res == got[0][2] and code == got[0][3]
        assert torch.equal(v, got[0][1])
    lam, v, _, code = got[0]
    if code == 0 and prec == "fp64":
        v = v.cpu().numpy()
        dmax = O.degree(g).max()
        assert np.linalg.norm(O.laplacian_apply(g, v) - lam * v) <= (1e-10 + 1e-13) * dmax


@pytest.mark.parametrize("g,parts", [(box_graph(24, 17, 6), 8),
                                     (box_graph_deleted(30, 21, 9, 0.45, 8, "face"), 7),
                                     (box_graph_deleted(48, 33, 21, 0.1, 9, "vertex"), 16)],
                         ids=["box", "fallen", "vertex"])
@pytest.mark.parametrize("policy", ["none", "resolve"])
def test_partition_modes_agree(g, parts, policy):
    G = R.graph(g)
    got = [R.rsb_partition(G, parts, R.options(method="inverse", precision="mixed",
                                               degenerate_policy=policy, use_graph=m,
                                               max_outer=12, cg_maxit=400))
           for m in (0, 1, 3)]
    for part, st, _ in got[1:]:
        assert torch.equal(part, got[0][0])
        assert st["inner"] == got[0][1]["inner"] and st["cycles"] == got[0][1]["cycles"]
