"""The search's hit-mask and fill kernels at the edges of their dispatch: pairs
exactly at the bound (the FP64 definition decides them), cells with more
particles than a work item's counters hold, clouds on either side of the size
up to which cells are split, clouds whose candidates exceed the mask pool, and
coordinates of extreme scale.  Lists equal the oracle's bit for bit."""
import numpy as np
import pytest

from paper_2405_13165_gb300 import clouds as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_13165_gb300 import mafp as M  # noqa: E402


def _lattice(m, h):
    g = np.arange(m, dtype=np.float32)
    x = np.stack([a.ravel() for a in np.meshgrid(g, g, g, indexing="ij")], 1)
    return np.concatenate([x, np.full((x.shape[0], 1), h, np.float32)], 1)


def _random(n, h_lo, h_hi, seed=3):
    rng = np.random.default_rng(seed)
    return np.concatenate([rng.uniform(0, 1, (n, 3)), rng.uniform(h_lo, h_hi, (n, 1))],
                          1).astype(np.float32)


CLOUDS = {
    "lattice at the bound": lambda: _lattice(17, 3.0),
    "one dense cell": lambda: _random(3000, 2.0, 2.0),
    "largest split cloud": lambda: _random(131072, 0.02, 0.03),
    "smallest unsplit cloud": lambda: _random(131073, 0.02, 0.03),
    "beyond the mask pool": lambda: _random(20000, 0.15, 0.2),
    "one particle": lambda: _random(1, 0.1, 0.1),
    "33 particles": lambda: _random(33, 0.5, 1.0),
}


@pytest.mark.parametrize("dtype", [M.F32_REFINED, M.F64])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -50, 3.0e12, 2.0 ** 122])
@pytest.mark.parametrize("name", sorted(CLOUDS))
def test_lists_equal_the_oracle(orc, name, scale, dtype):
    pos = CLOUDS[name]() * np.float32(scale)
    n = pos.shape[0]
    if n > 100_000 and scale != 1.0:
        pytest.skip("extreme scales on the small clouds only")
    pos = pos[C.cell_order(pos)]
    rp, col = orc.neighbours(pos)
    ctx = M.Context(n)
    t = torch.from_numpy(np.ascontiguousarray(pos)).cuda().to(M.real_dtype(dtype))
    grp, gcol, _ = M.neighbours(ctx, t, dtype, cap_nnz=int(rp[-1]) + 8)
    np.testing.assert_array_equal(grp.cpu().numpy(), rp)
    np.testing.assert_array_equal(gcol.cpu().numpy(), col)
    ctx.close()
