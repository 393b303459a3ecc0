"""The gather-scatter benchmark times the kernels that a call on the mesh runs: it counts the
bytes of the slot table's path for hexes, of the buckets' for ids beyond the table."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

import paper_2606_14659_gb300 as R  # noqa: E402


@pytest.mark.parametrize("f32", [True, False])
def test_bytes_of_the_path_that_runs(f32):
    nx = 24
    e = torch.arange(nx ** 3, device="cuda")
    i, j, k = e % nx, (e // nx) % nx, e // nx ** 2
    ev = torch.stack([(i + a) + (nx + 1) * ((j + b) + (nx + 1) * (k + c))
                      for c in (0, 1) for b in (0, 1) for a in (0, 1)], 1).contiguous()
    ne, V, es = nx ** 3, (nx + 1) ** 3, 4 if f32 else 8
    ms, by = R.rsb.rsb_laplacian_bench_gs(ev, f32, 5)
    assert ms > 0 and by == 4 * V + 96 * ne + 3 * es * ne + 4 * es * V
    shift = 1 << 20
    ms, by = R.rsb.rsb_laplacian_bench_gs(ev + shift, f32, 5)
    V += shift
    assert ms > 0 and by == 16 * (V + 1) + 64 * ne + 3 * es * ne + 2 * es * V
    with pytest.raises(R.RSBError):
        R.rsb.rsb_laplacian_bench_gs(ev - 1, f32, 5)
