"""Ritz pairs of the projected matrix for every parity and size of the Krylov space.

A cycle whose Krylov space is the whole of 1-perp ends with the exact eigenpairs of
the graph's Laplacian, so the dense eigenvalues are the reference: lambda_2 of a path
or small box from a space of n - 1 dimensions, n - 1 = 1 .. 40 (odd sizes pad the
rotation pairs).  FP64: eigenvalues of a symmetric matrix computed to rounding agree
to 1e-13 of its norm.  The launch modes share the routine and must agree bit for bit.
"""
import numpy as np
import pytest

from meshgen import box_graph

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

import paper_2606_14659_gb300 as R  # noqa: E402


def _dense(g):
    a = np.zeros((g.n, g.n))
    a[g.rows(), g.col] = g.w
    return np.diag(a.sum(1)) - a


@pytest.mark.parametrize("dims", [(2, 1, 1), (3, 1, 1), (4, 1, 1), (5, 1, 1), (3, 2, 1), (7, 1, 1),
                                  (17, 1, 1), (18, 1, 1), (33, 1, 1), (40, 1, 1), (41, 1, 1),
                                  (5, 4, 2), (13, 3, 1)])
def test_lambda2_from_the_whole_space(dims):
    g = box_graph(*dims)
    lap = _dense(g)
    ev = np.linalg.eigvalsh(lap)
    got = []
    for mode in (0, 2, 3):
        lam, v, _, code = R.rsb_fiedler(R.graph(g), R.options(use_graph=mode, max_restarts=400))
        assert code == 0
        assert abs(lam - ev[1]) <= 1e-13 * ev[-1]
        got.append((lam, v))
    assert got[0][0] == got[2][0] or abs(got[0][0] - got[2][0]) <= 1e-13 * ev[-1]
    for prec in ("mixed",):
        a = [R.rsb_fiedler(R.graph(g), R.options(use_graph=m, precision=prec)) for m in (0, 1, 3)]
        assert a[0][0] == a[1][0] == a[2][0]
        assert torch.equal(a[0][1], a[1][1]) and torch.equal(a[0][1], a[2][1])
        assert abs(a[0][0] - ev[1]) <= 1e-9 * ev[-1]
