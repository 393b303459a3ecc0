"""The FP32 Lanczos steps at the sizes where their splits leave something over.

Step D1 loads 13 entries of a row at a time (rows narrower, as wide, wider), step D2
gives a warp two coefficients and 128 rows, step D3 a CTA 512 rows and four basis
vectors, and the closing kernel takes one CTA, one per 32 or one per four coefficients
by the number of tiles of a unit.  The streaming launches (plain and as a graph) and
the resident launch share only their arithmetic, so they must agree bit for bit; the
vector must meet the stopping test with the oracle's Laplacian: the FP32 stage stops at
1e-6 d_max and the FP64 polish can only lower the residual (1.01e-6: the rounding of
the FP64 products is far below 1 %).
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

# face (6 entries a row) and vertex (26) graphs; 2 to 118000 rows: one tile, some
# tiles, above 32 and above 192 tiles of one unit
MESHES = [box_graph(2, 1, 1), box_graph(3, 2, 1), box_graph(33, 1, 1), box_graph(16, 8, 1),
          box_graph(43, 4, 3), box_graph_deleted(9, 8, 8, 0.05, 1, "vertex"),
          box_graph_deleted(17, 11, 7, 0.1, 2, "vertex"),
          box_graph_deleted(41, 33, 17, 0.1, 3, "vertex"),
          box_graph_deleted(71, 53, 35, 0.1, 4, "vertex")]


@pytest.mark.parametrize("g", MESHES, ids=lambda g: str(g.n))
@pytest.mark.parametrize("krylov", [2, 5, 40])
def test_steps_streaming_equals_resident_and_oracle(g, krylov):
    G = R.graph(g)
    got = []
    for mode in (0, 1, 3):
        lam, v, _, code = R.rsb_fiedler(G, R.options(precision="mixed", use_graph=mode,
                                                     krylov_dim=krylov, max_restarts=400,
                                                     keep=min(8, krylov - 1)))
        got.append((lam, v, code))
    for lam, v, code in got[1:]:
        assert lam == got[0][0] and code == got[0][2] and torch.equal(v, got[0][1])
    if got[0][2] == 0:
        lam, v = got[0][0], got[0][1].cpu().numpy()
        dmax = O.degree(g).max()
        assert np.linalg.norm(O.laplacian_apply(g, v) - lam * v) <= 1.01e-6 * dmax
    else:  # only a two- or five-step Krylov space may reach the cap
        assert krylov < 40


@pytest.mark.parametrize("rows", [2, 5])
def test_deflated_steps_streaming_equals_resident(rows):
    """RESOLVE: one and two FP64 deflation vectors in the basis, several units at once."""
    g = box_graph(24, 24, 12)
    G = R.graph(g)
    parts = [R.rsb_partition(G, 8, R.options(precision="mixed", use_graph=mode,
                                             tile_rows=rows))[0] for mode in (0, 1, 3)]
    assert torch.equal(parts[0], parts[1]) and torch.equal(parts[0], parts[2])


def test_many_short_tiles_equal_the_mesh_alone():
    """Step D3 runs CTAs of 128 threads once a level has more than 1216 tiles: 1300
    one-tile units of 4 to 88 rows, each bit-equal to its mesh solved alone."""
    meshes = [box_graph(2 + i % 3, 2, 1 + i % 11) for i in range(1300)]
    o = R.options(precision="mixed", use_graph=1, krylov_dim=12, keep=4, max_restarts=6)
    parts, _, _ = R.rsb_partition_batch([R.graph(g) for g in meshes], [4] * len(meshes), o)
    for i in list(range(0, 33)) + [1299]:
        alone, _, _ = R.rsb_partition(R.graph(meshes[i]), 4, o)
        assert torch.equal(torch.as_tensor(parts[i]), torch.as_tensor(alone)), i


# FP64 tiles have one row a thread in units above 1024 rows of meshes up to 31000
FP64 = [box_graph(16, 16, 4), box_graph(41, 5, 5), box_graph(31, 25, 40), box_graph(52, 71, 9)]


@pytest.mark.parametrize("g", FP64, ids=lambda g: str(g.n))
def test_fp64_tiles_at_the_edges_of_their_rule(g):
    G = R.graph(g)
    got = [R.rsb_fiedler(G, R.options(precision="fp64", use_graph=m)) for m in (0, 1, 3)]
    for lam, v, _, code in got[1:]:
        assert lam == got[0][0] and code == got[0][3] and torch.equal(v, got[0][1])
    assert got[0][3] == 0
    lam, v = got[0][0], got[0][1].cpu().numpy()
    dmax = O.degree(g).max()
    assert np.linalg.norm(O.laplacian_apply(g, v) - lam * v) <= (1e-10 + 1e-13) * dmax
