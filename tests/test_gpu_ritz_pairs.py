"""Eigenpairs of a cycle's projected matrix, close pairs among them.

FP64 pairs come from the FP32 ones by refinement, or by FP64 rotations where an eigenvalue
gap is too small for FP32 vectors.  Matrices with known eigenvalues, one gap from 0 to 0.1
of the norm among the kept ones; whatever the route, the pairs have FP64's residual and
orthogonality.  Bound: a pair is the result of products of K terms (the last refinement) or
of at most 8 sweeps of K - 1 rotations a column, four roundings each: 32 K u ||S||.  Pairs
left at FP32's accuracy miss it by a factor of 10^5.
"""
import numpy as np
import pytest

from meshgen import box_graph

torch = pytest.importorskip("torch")
needs_gpu = pytest.mark.skipif(not torch.cuda.is_available(), reason="no GPU")

U = 2.0 ** -53
SIZES = [(2, 1), (3, 2), (16, 8), (17, 16), (40, 8), (40, 16)]
GAPS = [0.0, 1e-16, 1e-13, 1e-10, 1e-8, 1e-7, 1e-5, 1e-4, 1e-3, 0.1]


def _matrix(K, gap, where, seed):
    rng = np.random.default_rng(seed)
    lam = np.sort(rng.uniform(0.05, 1.0, K)) + np.arange(K) * 0.2
    at = 0 if where == "first" else min(K - 2, 6)
    lam[at + 1] = lam[at] + gap * lam[-1]
    q = np.linalg.qr(rng.standard_normal((K, K)))[0]
    s = (q * lam) @ q.T
    return (s + s.T) / 2, lam


def _first_correction(s):
    """The largest correction that the refinement takes from FP32 eigenvectors."""
    x = np.linalg.eigh(s.astype(np.float32))[1].astype(np.float64)
    r, b = np.eye(len(s)) - x.T @ x, x.T @ s @ x
    lam = np.diag(b) / (1 - np.diag(r))
    with np.errstate(divide="ignore", invalid="ignore"):
        e = np.abs((b + lam * r) / (lam - lam[:, None]))
    np.fill_diagonal(e, 0)
    return (e + e.T).max()


def test_matrices_lie_on_both_sides_of_the_refinement():
    """A correction above 1e-2 sends the FP64 solve to the rotations."""
    close = [_first_correction(_matrix(40, g, w, 1)[0]) for g in (1e-13, 1e-10, 1e-8)
             for w in ("first", "inner")]
    wide = [_first_correction(_matrix(40, g, w, 1)[0]) for g in (1e-3, 0.1)
            for w in ("first", "inner")]
    assert min(close) > 1e-2 > max(wide)


@needs_gpu
@pytest.mark.gpu
@pytest.mark.parametrize("K,keep", SIZES)
@pytest.mark.parametrize("where", ["first", "inner"])
def test_fp64_pairs(K, keep, where):
    import paper_2606_14659_gb300 as R

    for gap in GAPS:
        for seed in range(3):
            s, _ = _matrix(K, gap, where, seed)
            ev = np.linalg.eigvalsh(s)
            theta, y = R.rsb.rsb_probe_ritz(s, keep)
            norm = np.linalg.norm(s)
            bound = 32 * K * U
            assert np.abs(s @ y - y * theta).max() <= bound * norm, (gap, seed)
            assert np.abs(y.T @ y - np.eye(keep + 1)).max() <= bound, (gap, seed)
            assert np.abs(theta - ev[:keep + 1]).max() <= bound * norm, (gap, seed)
            assert np.all(np.diff(theta) >= 0)


@needs_gpu
@pytest.mark.gpu
@pytest.mark.parametrize("diagonal", [True, False])
def test_fp64_pairs_of_special_matrices(diagonal):
    import paper_2606_14659_gb300 as R

    if diagonal:  # nothing to rotate, several equal values
        s = np.diag([3.0, 1.0, 1.0, 2.0, 0.0, 1.0, 5.0])
    else:  # all of the eigenvalues but one equal
        v = np.arange(1.0, 10.0)
        s = 2 * np.eye(9) - np.outer(v, v) / (v @ v)
    K = len(s)
    theta, y = R.rsb.rsb_probe_ritz(s, K - 1)
    bound = 32 * K * U
    assert np.abs(theta - np.linalg.eigvalsh(s)).max() <= bound * np.linalg.norm(s)
    assert np.abs(s @ y - y * theta).max() <= bound * np.linalg.norm(s)
    assert np.abs(y.T @ y - np.eye(K)).max() <= bound


@needs_gpu
@pytest.mark.gpu
@pytest.mark.parametrize("dims", [(2, 1, 1), (3, 1, 1), (5, 1, 1), (17, 1, 1), (18, 1, 1),
                                  (41, 1, 1), (5, 4, 2), (13, 3, 1)])
def test_fp64_modes_agree_bit_for_bit(dims):
    import paper_2606_14659_gb300 as R

    G = R.graph(box_graph(*dims))
    a = [R.rsb_fiedler(G, R.options(use_graph=m, max_restarts=400)) for m in (0, 1, 3)]
    for lam, v, _, _ in a[1:]:
        assert lam == a[0][0] and torch.equal(v, a[0][1])
