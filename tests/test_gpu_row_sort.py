"""Row lengths at the edges of the row sort's register sizes (32, 64, 128, 256,
512) and of its shared-memory one: clusters of exactly that many particles,
each within every other's reach, in a shuffled order.  Lists equal the
oracle's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_13165_gb300 import mafp as M  # noqa: E402

SIZES = [1, 2, 31, 32, 33, 64, 65, 127, 128, 129, 256, 257, 511, 512, 513, 1025]


@pytest.mark.parametrize("dtype", [M.F32_REFINED, M.F64])
def test_shuffled_clusters_give_sorted_rows(orc, dtype):
    rng = np.random.default_rng(7)
    parts = []
    for k, m in enumerate(SIZES):
        p = rng.uniform(0, 0.5, (m, 4))
        p[:, 0] += 4.0 * k
        p[:, 3] = 1.0
        parts.append(p)
    pos = np.concatenate(parts).astype(np.float32)
    pos = pos[rng.permutation(pos.shape[0])]
    rp, col = orc.neighbours(pos)
    assert sorted(set(np.diff(rp))) == SIZES
    ctx = M.Context(pos.shape[0])
    t = torch.from_numpy(pos).cuda().to(M.real_dtype(dtype))
    grp, gcol, _ = M.neighbours(ctx, t, dtype, cap_nnz=int(rp[-1]))
    assert ctx.status()["cells_identity"] == 0
    np.testing.assert_array_equal(grp.cpu().numpy(), rp)
    np.testing.assert_array_equal(gcol.cpu().numpy(), col)
    ctx.close()
