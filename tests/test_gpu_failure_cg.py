"""A resident CG solve whose unit barrier runs out.

The hook starts the arrivals out of reach: k_cg_res gives up (after 4 s) before it writes a
solution, the call returns RSB_ETIMEOUT and the next one is as usual.  No GPU fault is
involved: every wait is bounded.
"""
import time

import pytest

from meshgen import box_graph

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

import paper_2606_14659_gb300 as R  # noqa: E402


@pytest.mark.parametrize("dims", [(7, 5, 3), (40, 24, 16)])  # one tile, many
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_cg_timeout_returns_error_then_recovers(dims, precision):
    G = R.graph(box_graph(*dims))
    opts = R.options(method="inverse", precision=precision, use_graph=3)
    ref = R.rsb_fiedler(G, opts)
    R.rsb.rsb_test_poison_barrier(True)
    try:
        t0 = time.time()
        with pytest.raises(R.RSBError) as err:
            R.rsb_fiedler(G, opts)
        assert err.value.code == R.rsb.RSB_ETIMEOUT
        assert time.time() - t0 < 30
    finally:
        R.rsb.rsb_test_poison_barrier(False)
    again = R.rsb_fiedler(G, opts)
    assert again[0] == ref[0] and again[3] == ref[3]
    assert torch.equal(again[1], ref[1])
