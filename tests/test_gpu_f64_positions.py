"""The FP64 search on positions that 32 bits do not hold: it decides in FP32 where that is
certain, so pairs at the bound, coordinates at the cells' faces and whole clouds whose
structure lies below FP32's last bit have to come out as the FP64 definition has them.
Lists and cell order equal the oracle's and the generator's, which take 64 bits."""
import numpy as np
import pytest

from paper_2405_13165_gb300 import clouds as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_13165_gb300 import mafp as M  # noqa: E402


def _noise(rng, shape, bits):
    """0 and +-2^-bits times small whole numbers."""
    return rng.integers(-3, 4, shape) * 2.0 ** -bits


def _pairs_at_the_bound(rng):
    # a lattice of spacing 1 whose pairs at distance 3 are at the bound, off it by bits
    # far below FP32's last
    g = np.arange(13.0)
    x = np.stack([a.ravel() for a in np.meshgrid(g, g, g, indexing="ij")], 1)
    return np.concatenate([x + _noise(rng, x.shape, 46),
                           3.0 + _noise(rng, (x.shape[0], 1), 46)], 1)


def _at_the_faces(rng):
    # every coordinate within a few 2^-48 of a cell's face
    h = 0.25
    c = h * (1.0 + 1e-6)
    q = rng.integers(0, 9, (4000, 3)) * c
    q[0] = 0.0
    p = np.concatenate([q + np.abs(_noise(rng, q.shape, 48)), np.full((4000, 1), h)], 1)
    p[1:, :3] -= 2.0 ** -48 * (p[1:, :3] > c / 2) * rng.integers(0, 4, (3999, 3))
    return p


def _below_the_last_bit(rng):
    # a cloud of extent 2^-13 at 1000: FP32 holds three different coordinates there
    x = 1000.0 + rng.uniform(0, 2.0 ** -13, (6000, 3))
    return np.concatenate([x, np.full((6000, 1), 2.0 ** -13 * 0.14)], 1)


def _wide_h(rng):
    x = rng.uniform(0, 1, (5000, 3))
    return np.concatenate([x, rng.uniform(0.02, 0.16, (5000, 1))], 1)


CLOUDS = {"pairs at the bound": _pairs_at_the_bound, "at the faces": _at_the_faces,
          "below the last bit": _below_the_last_bit, "wide h": _wide_h}


@pytest.mark.parametrize("ordered", [True, False])
@pytest.mark.parametrize("name", sorted(CLOUDS))
def test_lists_and_order(orc, name, ordered):
    rng = np.random.default_rng(11)
    pos = np.ascontiguousarray(CLOUDS[name](rng))
    if name != "wide h":     # the values are not those of 32 bits
        assert (pos != pos.astype(np.float32)).any(1).mean() > 0.5
    pos = pos[C.cell_order(pos) if ordered else rng.permutation(len(pos))]
    n = pos.shape[0]
    rp, col = orc.neighbours(pos)
    ctx = M.Context(n)
    t = torch.from_numpy(np.ascontiguousarray(pos)).cuda()
    grp, gcol, order = M.neighbours(ctx, t, M.F64, cap_nnz=int(rp[-1]) + 8, order=True)
    np.testing.assert_array_equal(grp.cpu().numpy(), rp)
    np.testing.assert_array_equal(gcol.cpu().numpy(), col)
    np.testing.assert_array_equal(order.cpu().numpy(), C.cell_order(pos))
    ctx.close()
