"""Step D3 in CTAs of 128 and of 256 threads: the same mesh, alone and in batches that put
the level on either side of the rule (one wave of 1216 CTAs, two waves, short tiles), gives
the same parts."""
import pytest

from meshgen import box_graph

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

import paper_2606_14659_gb300 as R  # noqa: E402


@pytest.mark.parametrize("dims,counts", [
    ((8, 8, 8), (1, 1216, 1217, 2432, 2433)),    # full tiles of 512 rows
    ((13, 9, 9), (2, 500, 811, 1300)),           # 512 + 512 + 29
    ((6, 5, 4), (1, 1300, 3000)),                # 120 rows
])
def test_batches_equal_the_mesh_alone(dims, counts):
    G = R.graph(box_graph(*dims))
    o = R.options(precision="mixed", use_graph=1, krylov_dim=12, keep=4, max_restarts=4,
                  polish_cycles=1, degenerate_policy="none")
    alone = R.rsb_partition(G, 4, o)[0]
    for n in counts:
        parts = R.rsb_partition_batch([G] * n, [4] * n, o)[0]
        for i in (0, n // 2, n - 1):
            assert torch.equal(parts[i], alone), (n, i)
