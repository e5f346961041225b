"""The search's pool of hit words and cells that need far more than their share of it: a
dense patch's cells leave the rest of a cloud to the mask kernel as if they were not
there; the lists are the oracle's."""
import numpy as np
import pytest

from paper_2405_13165_gb300 import clouds as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_13165_gb300 import mafp as M  # noqa: E402


def _film(n, dense, side, seed=3):
    """n film particles of ~40 neighbours and `dense` more in a patch of that side."""
    rng = np.random.default_rng(seed)
    h = np.sqrt(40.0 / (n * np.pi))
    x = np.concatenate([rng.uniform(0, 1, (n, 2)), 0.4 + side * rng.uniform(0, 1, (dense, 2))])
    pos = np.concatenate([x, np.zeros((n + dense, 1)), np.full((n + dense, 1), h)], 1)
    pos = pos.astype(np.float32)
    return np.ascontiguousarray(pos[C.cell_order(pos)])


@pytest.mark.parametrize("dtype", [M.F32_REFINED, M.F64])
@pytest.mark.parametrize("dense,side", [(3000, 0.002), (9000, 0.05), (20000, 0.05)])
def test_lists_equal_the_oracle(orc, dense, side, dtype):
    # one cell beyond its limit; many near it; many beyond the pool
    pos = _film(20_000, dense, side)
    rp, col = orc.neighbours(pos)
    ctx = M.Context(pos.shape[0])
    t = torch.from_numpy(pos).cuda().to(M.real_dtype(dtype))
    grp, gcol, _ = M.neighbours(ctx, t, dtype, cap_nnz=int(rp[-1]) + 8)
    np.testing.assert_array_equal(grp.cpu().numpy(), rp)
    np.testing.assert_array_equal(gcol.cpu().numpy(), col)
    ctx.close()


def test_a_dense_patch_does_not_use_the_pool_up():
    # the patch's ~50 cells of ~2400 particles would need 80M words of a pool of 12.8M.  A
    # few dozen heavy blocks take as long as one: left with the film's thousands of
    # cells beside them, in an order that varies, some shared an SM (584 to 752 ms)
    pos = torch.from_numpy(_film(80_000, 120_000, 0.09)).cuda().double()
    n = pos.shape[0]
    ctx = M.Context(n)
    rp = torch.empty(n + 1, dtype=torch.int64, device="cuda")
    col = torch.empty(830 * 10**6, dtype=torch.int32, device="cuda")
    ms = []
    for _ in range(9):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        M.build_neighbours(ctx, pos, rp, col, None, None, M.F64)
        b.record()
        b.synchronize()
        ms.append(a.elapsed_time(b))
    assert ctx.status()["code"] == 0
    ctx.close()
    assert max(ms[1:]) <= 1.15 * min(ms), ms
