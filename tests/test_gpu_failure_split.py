"""A level's cooperative split whose barrier wait runs out.

The hook starts the barrier's arrivals out of reach, so the kernel gives up (after 4 s)
and leaves its side bits unfinished.  The levels that follow must then cut every segment by
row number, so that nothing lands outside its segment; the call returns RSB_ETIMEOUT, and
the next call is as usual.  No GPU fault is involved: every wait is bounded.
"""
import time

import pytest

from meshgen import box_graph, box_graph_deleted

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

import paper_2606_14659_gb300 as R  # noqa: E402

# launch mode 1 keeps the solves free of barriers, so that the split is what gives up
CASES = [
    ("rcb_one_tile", box_graph(8, 4, 4), 2, dict(method="rcb")),
    ("rcb_levels", box_graph(40, 32, 24), 37, dict(method="rcb")),
    ("lanczos_candidates", box_graph(16, 16, 16), 8, dict(use_graph=1, precision="mixed")),
    ("lanczos_pieces", box_graph_deleted(24, 16, 9, 0.45, 5, "face"), 16,
     dict(use_graph=1, degenerate_policy="none", precision="mixed")),
    ("reorder", box_graph(32, 16, 8), 4, dict(use_graph=1, reorder=1)),
]


@pytest.mark.parametrize("name,g,parts,kw", CASES, ids=[c[0] for c in CASES])
def test_split_timeout_returns_error_then_recovers(name, g, parts, kw):
    G = R.graph(g)
    opts = R.options(**kw)
    ref = R.rsb_partition(G, parts, opts)[0]
    R.rsb.rsb_test_poison_barrier(True)
    try:
        t0 = time.time()
        with pytest.raises(R.RSBError) as err:
            R.rsb_partition(G, parts, opts)
        assert err.value.code == R.rsb.RSB_ETIMEOUT
        assert time.time() - t0 < 30
    finally:
        R.rsb.rsb_test_poison_barrier(False)
    for _ in range(2):
        assert torch.equal(R.rsb_partition(G, parts, opts)[0], ref)
