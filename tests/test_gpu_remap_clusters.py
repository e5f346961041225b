"""The remap's work lists: no particle flagged, every 3D wall particle flagged (one
compact cluster), a few scattered ones, in clouds whose sizes leave the last warp
of the seeding pass partly filled.  The transition equals the oracle's."""
import numpy as np
import pytest

from paper_2405_13165_gb300 import clouds as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_13165_gb300 import mafp as M  # noqa: E402
from test_gpu_remap import _compare  # noqa: E402


@pytest.mark.parametrize("dtype", [M.F32_REFINED, M.F64])
@pytest.mark.parametrize("share", ["none", "some", "all"])
@pytest.mark.parametrize("drop", [0, 1, 31])
def test_clusters_of_flagged_particles(dtype, share, drop):
    c = C.cell_sorted(C.config_small())
    c = c.take(np.arange(c.n - drop))
    wall = (c.model == C.MODEL_3D) & (c.ptype == C.TYPE_WALL)
    c.user[:] = 0
    if share == "all":
        c.user[wall] = C.USER_TO_2D
    elif share == "some":
        c.user[np.nonzero(wall)[0][::7]] = C.USER_TO_2D
    _compare(c, dtype, 2e-6 if dtype == M.F32_REFINED else 1e-12)
