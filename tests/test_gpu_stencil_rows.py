"""The stencil build at the edges of its dispatch: rows longer than the per-lane
cache (long-range supports), clouds on either side of the sizes at which the
lanes per row and the rows per warp change, particle counts that leave a warp's
last look partly past the end, and clouds of one model only.  Coefficients
against the oracle, per row and operator, at the suite's tolerances."""
import numpy as np
import pytest

from paper_2405_13165_gb300 import clouds as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_13165_gb300 import mafp as M  # noqa: E402
from parity_util import TOL, run_gpu, stencil_rowwise_error_vec  # noqa: E402


def _wide(c, factor):
    c = c.take(np.arange(c.n))
    c.pos_h[:, 3] *= np.float32(factor)
    c.h3d[:] = c.pos_h[:, 3]
    return c


def _first(c, n):
    return c.take(np.arange(n))


CLOUDS = {
    "long rows": lambda: _wide(C.config_small(), 1.5),           # up to ~600 / 90 entries
    "film only": lambda: C.flat_film(0.01, 0.5, 0.003),
    "3D only": lambda: C.shallow_layer(0.02, 14, 0.18),
    "16384": lambda: _first(C.cell_sorted(C.flat_film(0.01, 1.3, 0.003)), 16384),
    "16385": lambda: _first(C.cell_sorted(C.flat_film(0.01, 1.3, 0.003)), 16385),
    "65536": lambda: _first(C.cell_sorted(C.jet_on_plate(None, 68_000)), 65536),
    "65537": lambda: _first(C.cell_sorted(C.jet_on_plate(None, 68_000)), 65537),
    "65567": lambda: _first(C.cell_sorted(C.jet_on_plate(None, 68_000)), 65567),
}


@pytest.mark.parametrize("dtype", [M.F32_REFINED, M.F32_PLAIN, M.F64])
@pytest.mark.parametrize("name", sorted(CLOUDS))
def test_coefficients(orc, name, dtype):
    c = CLOUDS[name]()
    rp, col = orc.neighbours(c.pos_h)
    coef, status, _ = orc.stencils(c.pos_h, c.model, rp, col)
    g, *_ = run_gpu(c, dtype, cap_nnz=int(rp[-1]) + 8, stages=("nbr", "cls", "st"))
    assert g["status_block"]["code"] == 0
    np.testing.assert_array_equal(g["col"], col)
    np.testing.assert_array_equal(g["status"] == M.STENCIL_DEFICIENT, status != 0)
    err, _ = stencil_rowwise_error_vec(rp, g["coef"], coef)
    assert np.all(err <= TOL[dtype]), err
    # entries of the other model are exact zeros
    rows = np.repeat(np.arange(c.n), np.diff(rp))
    assert not g["coef"][c.model[rows] != c.model[col]].any()
