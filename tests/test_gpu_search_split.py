"""The search on either side of the size up to which it quarters the costly cells (beyond
it halves them): a film with blocks of 3D density, whose cells of more than 24 particles
are the costly ones.  Lists equal the oracle's bit for bit."""
import numpy as np
import pytest

from paper_2405_13165_gb300 import clouds as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_13165_gb300 import mafp as M  # noqa: E402


@pytest.mark.parametrize("dtype", [M.F32_REFINED, M.F64])
@pytest.mark.parametrize("n", [524288, 524289])
def test_lists_equal_the_oracle(orc, n, dtype):
    rng = np.random.default_rng(2)
    dense = 60_000
    h = (8.0 / (np.pi * (n - dense))) ** 0.5
    film = np.concatenate([rng.uniform(0, 1, (n - dense, 2)), np.zeros((n - dense, 1))], 1)
    # about 35 particles per cell
    block = rng.uniform(0, (dense / 35.0) ** (1 / 3) * h, (dense, 3)) + 0.4
    pos = np.concatenate([np.concatenate([film, block]), np.full((n, 1), h)], 1).astype(np.float32)
    pos = pos[C.cell_order(pos)]
    rp, col = orc.neighbours(pos)
    ctx = M.Context(n)
    t = torch.from_numpy(np.ascontiguousarray(pos)).cuda().to(M.real_dtype(dtype))
    grp, gcol, _ = M.neighbours(ctx, t, dtype, cap_nnz=int(rp[-1]) + 8)
    np.testing.assert_array_equal(grp.cpu().numpy(), rp)
    np.testing.assert_array_equal(gcol.cpu().numpy(), col)
    ctx.close()
