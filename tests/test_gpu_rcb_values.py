"""Coordinate bisection of coordinates that are not all finite.

Every part has its size whatever the coordinates hold: NaNs of either sign sort behind
every number, an infinite extent makes every number of a segment a tie, an extent that is
no number (tie_rel = 0) leaves the exact ties.  The reference states that rule in numpy,
comparisons only, so parts agree exactly; on finite coordinates it is the oracle's.  The
cooperative split (few meshes) and the split step by step (20,000 copies in a batch) take
the same decisions.
"""
import numpy as np
import pytest

import oracle as O
from meshgen import box_graph

torch = pytest.importorskip("torch")
needs_gpu = pytest.mark.skipif(not torch.cuda.is_available(), reason="no GPU")

COPIES = 20000  # tiles (one each): above 32 x 4 x 152, the cooperative launch's limit


def _split(v, gid, k, tie_rel):
    num = v[~np.isnan(v)]
    vk = np.sort(v)[k - 1]  # (numpy sorts NaNs last)
    with np.errstate(invalid="ignore", over="ignore"):
        if np.isnan(vk):
            below, tie = ~np.isnan(v), np.isnan(v)
        else:
            tau = tie_rel * (max(-1e300, num.max()) - min(1e300, num.min()))
            if np.isnan(tau):
                tau = 0.0
            below = v < (-np.inf if np.isinf(tau) else vk - tau)
            tie = ~below & ((v <= vk) | (v - vk <= tau))
    t = np.nonzero(tie)[0]
    t = t[np.argsort(gid[t], kind="stable")]
    left = below.copy()
    left[t[:k - int(below.sum())]] = True
    return left


def _extent(c):
    num = c[~np.isnan(c)]
    with np.errstate(over="ignore"):
        return (max(-1e300, num.max()) if len(num) else -1e300) + \
            (max(-1e300, (-num).max()) if len(num) else -1e300)


def _rcb(coords, gid, P, tie_rel):
    n = len(coords)
    part = np.full(n, -1, np.int32)
    stack = [(np.arange(n), 0, P)]
    while stack:
        idx, p0, p1 = stack.pop()
        if p1 - p0 == 1:
            part[idx] = p0
            continue
        pm = p0 + (p1 - p0) // 2
        k = (pm * n) // P - (p0 * n) // P
        ext = [_extent(coords[idx, a]) for a in range(3)]
        axis = max(range(3), key=lambda a: (ext[a], -a))
        left = _split(coords[idx, axis], gid[idx], k, tie_rel)
        stack.append((idx[~left], pm, p1))
        stack.append((idx[left], p0, pm))
    return part


def _sizes(n, P):
    return [O.seg_size(p, p + 1, n, P) for p in range(P)]


# (share of the rows, value) put in the x column, others in y
KINDS = {
    "nan": [(0.02, np.nan)],
    "negative_nan": [(0.1, -np.nan)],
    "both_nan": [(0.1, np.nan), (0.1, -np.nan)],
    "most_nan": [(0.6, np.nan)],
    "all_nan": [(1.0, np.nan)],
    "every_nan": [(1.0, np.nan)],
    "inf": [(0.05, np.inf)],
    "most_inf": [(0.7, np.inf)],
    "most_minus_inf": [(0.7, -np.inf)],
    "both_inf": [(0.3, np.inf), (0.3, -np.inf)],
    "inf_and_nan": [(0.2, np.inf), (0.2, np.nan), (0.2, -np.inf)],
    "huge": [(0.3, 1.7e308), (0.3, -1.7e308)],
}


def _case(kind, n, seed):
    rng = np.random.default_rng(seed)
    xyz = rng.standard_normal((n, 3)) * [9.0, 2.0, 1.0]
    xyz[:, 0] = np.round(xyz[:, 0])  # ties, also at zero of either sign
    order = rng.permutation(n)
    at = 0
    for share, value in KINDS.get(kind, []):
        m = max(1, int(share * n))
        xyz[order[at:at + m], 0] = value
        if kind != "nan":
            xyz[order[at:at + m // 2], 1] = value
        at += m
    if kind == "every_nan":
        xyz[:] = np.nan
    return xyz


def test_reference_is_the_oracle_on_finite_coordinates():
    for seed in range(5):
        xyz = _case("finite", 200, seed)
        gid = np.random.default_rng(seed).permutation(200).astype(np.int64)
        for P in (2, 7, 32):
            assert np.array_equal(_rcb(xyz, gid, P, 1e-5), O.rcb_partition(xyz, gid, P))


@pytest.mark.parametrize("kind", list(KINDS))
def test_reference_keeps_the_sizes(kind):
    xyz = _case(kind, 100, 3)
    for tie_rel in (0.0, 1e-5, 1.0):
        part = _rcb(xyz, np.arange(100), 7, tie_rel)
        assert np.array_equal(np.bincount(part, minlength=7), _sizes(100, 7))


@needs_gpu
@pytest.mark.gpu
@pytest.mark.parametrize("kind", list(KINDS))
@pytest.mark.parametrize("dims", [(25, 2, 2), (40, 20, 3)])
def test_rcb_of_values_that_are_not_finite(kind, dims):
    import paper_2606_14659_gb300 as R

    g = box_graph(*dims)
    g.gid = np.random.default_rng(8).permutation(g.n).astype(np.int64) + 17
    xyz = _case(kind, g.n, 4)
    G = R.graph(g, coords=xyz)
    for P, tie_rel in ((2, 1e-5), (7, 1e-5), (7, 0.0), (16, 1.0)):
        opts = R.options(method="rcb", tie_rel=tie_rel)
        ref = _rcb(xyz, g.gid, P, tie_rel)
        assert np.array_equal(np.bincount(ref, minlength=P), _sizes(g.n, P))
        part, _, code = R.rsb_partition(G, P, opts)
        assert code == 0
        assert np.array_equal(part.cpu().numpy(), ref), (P, tie_rel)


@needs_gpu
@pytest.mark.gpu
@pytest.mark.parametrize("kind", list(KINDS))
def test_the_steps_decide_alike(kind):
    import paper_2606_14659_gb300 as R

    g = box_graph(13, 2, 2)
    xyz = _case(kind, g.n, 5)
    G = R.graph(g, coords=xyz)
    for P, tie_rel in ((2, 1e-5), (5, 0.0)):
        ref = _rcb(xyz, g.gid, P, tie_rel)
        many, _, code = R.rsb_partition_batch([G] * COPIES, [P] * COPIES,
                                              R.options(method="rcb", tie_rel=tie_rel))
        assert code == 0
        for p in (many[0], many[777], many[COPIES - 1]):
            assert np.array_equal(p.cpu().numpy(), ref), (P, tie_rel)


@needs_gpu
@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["nan", "most_nan", "inf_and_nan"])
def test_reorder_by_such_coordinates(kind):
    import paper_2606_14659_gb300 as R

    g = box_graph(32, 16, 8)
    xyz = _case(kind, g.n, 6)
    G = R.graph(g, coords=xyz)
    part, _, code = R.rsb_partition(G, 16, R.options(reorder=1))
    assert code == 0  # the order of the rows does not change the partition
    assert np.array_equal(part.cpu().numpy(), O.box_partition_closed_form(32, 16, 8, 16))
