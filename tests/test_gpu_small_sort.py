"""The one-block sort of small clouds on either side of its largest size, with one,
two and three digits of cells, shuffled: lists and cell order equal the oracle's
and the generator's."""
import numpy as np
import pytest

from paper_2405_13165_gb300 import clouds as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_13165_gb300 import mafp as M  # noqa: E402


@pytest.mark.parametrize("dtype", [M.F32_REFINED, M.F64])
@pytest.mark.parametrize("n", [2, 1023, 1025, 8192, 8193])
@pytest.mark.parametrize("h", [0.6, 0.12, 0.01])     # about 4, 600 and 10^6 cells
def test_shuffled_small_clouds(orc, n, h, dtype):
    rng = np.random.default_rng(n)
    pos = np.concatenate([rng.uniform(0, 1, (n, 3)), np.full((n, 1), h)], 1).astype(np.float32)
    rp, col = orc.neighbours(pos)
    if (np.diff(rp) > 2048).any():
        pytest.skip("rows longer than the row sort takes")
    ctx = M.Context(n, cap_cells=1 << 21)
    t = torch.from_numpy(pos).cuda().to(M.real_dtype(dtype))
    grp, gcol, order = M.neighbours(ctx, t, dtype, cap_nnz=int(rp[-1]), order=True)
    np.testing.assert_array_equal(grp.cpu().numpy(), rp)
    np.testing.assert_array_equal(gcol.cpu().numpy(), col)
    np.testing.assert_array_equal(order.cpu().numpy(), C.cell_order(pos))
    ctx.close()
