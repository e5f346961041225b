"""apply_ops over rows of every length around the lanes' strides (0 to 40 entries, 4, 8 and
16 lanes per row), where a lane's second or later entry in flight is past the row's
end: against the sums in 64 bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_13165_gb300 import mafp as M  # noqa: E402


@pytest.mark.parametrize("dtype", [M.F32_REFINED, M.F64])
@pytest.mark.parametrize("lanes", [4, 8, 16])
def test_rows_of_every_length(lanes, dtype):
    rng = np.random.default_rng(lanes)
    lens = np.concatenate([np.arange(41), rng.permutation(41), np.zeros(7, int), [33]])
    n, rp = len(lens), np.concatenate([[0], np.cumsum(lens)])
    col = rng.integers(0, n, rp[-1]).astype(np.int32)
    coef, fld = rng.normal(size=(rp[-1], 4)), rng.normal(size=(n, 4))
    rd = M.real_dtype(dtype)
    coef, fld = (torch.tensor(a, dtype=rd) for a in (coef, fld))
    want, size = np.zeros((n, 4, 4)), np.zeros((n, 4, 4))
    c, f = coef.double().numpy(), fld.double().numpy()
    for i in range(n):
        for e in range(rp[i], rp[i + 1]):
            t = np.outer(f[col[e]] - f[i], c[e])
            want[i] += t
            size[i] += np.abs(t)
    ctx = M.Context(n)
    ctx.set_tuning(apply_group=lanes)
    out = torch.full((n, 4, 4), 7.0, dtype=rd, device="cuda")
    M.apply_ops(ctx, torch.tensor(rp).cuda(), torch.tensor(col).cuda(), coef.cuda(), fld.cuda(), out,
                dtype)
    # a difference, a product and at most 40 additions, each rounded once
    eps = 42 * (2.0 ** -24 if dtype != M.F64 else 2.0 ** -53)
    err = np.abs(out.double().cpu().numpy() - want)
    assert np.all(err <= eps * size), (err / np.maximum(size, 1e-300)).max()
    ctx.close()
