"""The split of a level in one cooperative launch against the split step by step.

A level of more than 32 tiles for every co-resident CTA takes the steps one by one, so
20,000 copies of a small mesh in one batch are split by the general path and a few
copies by the cooperative launch; a mesh gives the same parts in any batch.  The meshes
have every kind of tie (boxes: whole slabs), odd and single-element splits, halves that
fall apart, gids that are large, sparse and in no order, and values of either sign.
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

COPIES = 20000  # tiles (one each): above 32 x 4 x 152


def _gids(n, seed):
    rng = np.random.default_rng(seed)
    return rng.choice(1 << 50, n, replace=False).astype(np.int64)


MESHES = {
    "two": (box_graph(2, 1, 1), None),
    "cube": (box_graph(3, 3, 3), None),
    "slab": (box_graph(4, 4, 2), 11),
    "path": (box_graph(13, 1, 1), 12),
    "fallen": (box_graph_deleted(5, 4, 3, 0.4, 6, "face"), 13),
    "vertex": (box_graph_deleted(4, 4, 4, 0.2, 7, "vertex"), 14),
}


@pytest.mark.parametrize("name", list(MESHES))
@pytest.mark.parametrize("method", ["rcb", "lanczos"])
def test_cooperative_split_equals_the_steps(name, method):
    g, seed = MESHES[name]
    rng = np.random.default_rng(3)
    xyz = g.centroids()
    if seed:  # rotated: coordinates of either sign, few of them equal
        g.gid = _gids(g.n, seed)
        if method == "rcb" and seed % 2:
            xyz = (xyz - xyz.mean(0)) @ np.linalg.qr(rng.standard_normal((3, 3)))[0]
    G = R.graph(g, coords=xyz)
    for parts in sorted({2, min(7, g.n)}):
        opts = R.options(method=method, degenerate_policy="none" if method == "rcb" else "resolve")
        many, _, _ = R.rsb_partition_batch([G] * COPIES, [parts] * COPIES, opts)
        few, _, _ = R.rsb_partition_batch([G] * 3, [parts] * 3, opts)
        one, _, _ = R.rsb_partition(G, parts, opts)
        for p in (many[0], many[COPIES - 1], many[777], few[0], few[2]):
            assert torch.equal(p, one)
        sizes = np.bincount(one.cpu().numpy(), minlength=parts)
        assert np.array_equal(sizes, [O.seg_size(p, p + 1, g.n, parts) for p in range(parts)])


@pytest.mark.parametrize("dims", [(31, 1, 1), (40, 32, 16), (64, 64, 48)])
@pytest.mark.parametrize("parts", [2, 5, 64])
def test_rcb_of_tied_boxes_against_the_oracle(dims, parts):
    g = box_graph(*dims)
    if parts > g.n:
        pytest.skip("more parts than elements")
    part, _, code = R.rsb_partition(R.graph(g), parts, R.options(method="rcb"))
    assert code == 0
    assert np.array_equal(part.cpu().numpy(), O.rcb_partition(g.centroids(), g.gid, parts))
