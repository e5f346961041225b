"""The lanes per row that a caller asks for are the lanes that the stencil build takes in
clouds of more than 16384 particles (the names of its kernels say them), and on film in
FP32 always, with the oracle's coefficients; the defaults, and smaller clouds, leave them to
the library."""
import numpy as np
import pytest

from paper_2405_13165_gb300 import clouds as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_13165_gb300 import mafp as M  # noqa: E402
from parity_util import TOL, run_gpu, stencil_rowwise_error_vec  # noqa: E402


def _first(cloud, n):
    return C.cell_sorted(cloud).take(np.arange(n))


CLOUDS = {
    "small": lambda: C.config_small(),
    # 3D rows on either side of that size
    "16384": lambda: _first(C.jet_on_plate(None, 17_500), 16384),
    "16385": lambda: _first(C.jet_on_plate(None, 17_500), 16385),
}


def _taken(asked, n, dtype):
    if n <= 16384:
        return 32, 8 if dtype == M.F64 else asked[1]
    return {32: 8}.get(asked[0], asked[0]), 4 if dtype == M.F64 and asked[1] == 8 else asked[1]


ASKED = [(8, 4), (16, 16), (16, 4), (8, 16), (32, 8)]


@pytest.mark.parametrize("dtype", [M.F32_REFINED, M.F32_PLAIN, M.F64])
@pytest.mark.parametrize("name", sorted(CLOUDS))
def test_lanes_asked_for_are_taken(orc, name, dtype):
    c = CLOUDS[name]()
    rp, col = orc.neighbours(c.pos_h)
    coef, status, _ = orc.stencils(c.pos_h, c.model, rp, col)
    for lanes in ASKED:
        ctx = M.Context(c.n)
        ctx.set_tuning(stencil3d_group=lanes[0], stencil2d_group=lanes[1])
        ctx.profile(True)
        g, *_ = run_gpu(c, dtype, ctx=ctx, cap_nnz=int(rp[-1]) + 8, stages=("nbr", "cls", "st"))
        names = ctx.profile_read()
        ctx.profile(False)
        for model, k in zip((10, 6), _taken(lanes, c.n, dtype)):
            assert any(f"k_stencil<" in s and f"M={model},G={k}," in s for s in names), (lanes, names)
        assert g["status_block"]["code"] == 0
        np.testing.assert_array_equal(g["status"] == M.STENCIL_DEFICIENT, status != 0)
        err, _ = stencil_rowwise_error_vec(rp, g["coef"], coef)
        assert np.all(err <= TOL[dtype]), (lanes, err)
        ctx.close()
