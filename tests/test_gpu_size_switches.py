"""One particle more may not cost much more: the stencil build on either side of the
sizes at which the lanes per row or the rows per warp change, for a column of 3D rows in
a wide film (whose 3D rows lie in few warps) and a block of 3D rows on a small film."""
import numpy as np
import pytest

from paper_2405_13165_gb300 import clouds as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_13165_gb300 import mafp as M  # noqa: E402
from paper_2405_13165_gb300.pipeline import Pipeline, cloud_to_device  # noqa: E402


def _build_us(cloud, dtype):
    d = cloud_to_device(cloud, dtype)
    n = d["pos_h"].shape[0]
    ctx = M.Context(n)
    p = Pipeline(ctx, n, 200 * n, dtype)
    p.step(d)
    assert ctx.status()["code"] == 0
    t = []
    for _ in range(15):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        p.stencils(d)
        b.record()
        b.synchronize()
        t.append(a.elapsed_time(b))
    ctx.close()
    return 1e3 * sorted(t)[len(t) // 2]


@pytest.mark.parametrize("dtype", [M.F32_REFINED, M.F64])
@pytest.mark.parametrize("shape", ["jet", "cube"])
@pytest.mark.parametrize("n", [16384, 65536, 163840, 262144])
def test_build_time_has_no_step(n, shape, dtype):
    if dtype == M.F64 and n > 65536:
        pytest.skip("FP64 has no switch there")
    if shape == "jet":
        c = C.cell_sorted(C.jet_on_plate(None, n + n // 20))
    else:
        dx = 1.1 * (0.027 / n) ** (1 / 3)
        while (c := C.cube_on_sheet(dx)).n <= n:
            dx *= 0.95
        c = C.cell_sorted(c)
    below, above = (_build_us(c.take(np.arange(k)), dtype) for k in (n, n + 1))
    # a quarter more is well beyond the runs' own spread (5 %)
    assert above <= 1.25 * below, (below, above)
