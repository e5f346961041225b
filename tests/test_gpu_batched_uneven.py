"""Batches of very uneven clouds: bounding boxes are reduced by blocks that follow each
cloud's own size, so clouds that end at, just before and just behind a block's share,
empty clouds at either end and in between, and one large cloud among many small ones
give each cloud's own lists, and the large one costs what it costs alone."""
import numpy as np
import pytest

from paper_2405_13165_gb300 import clouds as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_13165_gb300 import mafp as M  # noqa: E402

SIZES = {
    "around a block's share": [2047, 1, 2048, 2049, 4095, 4096, 4097, 3],
    "empty clouds": [0, 0, 50, 0, 5000, 0, 7, 0],
    "one large": [60] * 40 + [9000] + [1] * 40,
}


def _film(n, seed):
    """n film particles in cell order, about 40 neighbours each."""
    rng = np.random.default_rng(seed)
    h = np.sqrt(40.0 / (max(n, 40) * np.pi))
    pos = np.concatenate([rng.uniform(-1 - seed, -seed, (n, 2)), np.zeros((n, 1)),
                          np.full((n, 1), h)], 1).astype(np.float32)
    return pos[C.cell_order(pos)] if n else pos


def _search(pos, sizes, dtype, cap):
    n = pos.shape[0]
    off = torch.tensor(np.concatenate([[0], np.cumsum(sizes)]), dtype=torch.int64).cuda()
    t = torch.from_numpy(pos).cuda().to(M.real_dtype(dtype))
    ctx = M.Context(n)
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    col = torch.zeros(cap, dtype=torch.int32, device="cuda")
    return ctx, rp, col, lambda: M.build_neighbours_batched(ctx, off, t, rp, col, None, None, dtype)


@pytest.mark.parametrize("dtype", [M.F32_REFINED, M.F64])
@pytest.mark.parametrize("name", sorted(SIZES))
def test_lists_are_each_clouds_own(orc, name, dtype):
    sizes = SIZES[name]
    parts = [_film(k, i) for i, k in enumerate(sizes)]
    rps, cols, at = [np.zeros(1, np.int64)], [], 0
    for p in parts:
        if len(p):
            rp, col = orc.neighbours(p)
            rps.append(rp[1:] + rps[-1][-1])
            cols.append(col + at)
        at += len(p)
    rp, col = np.concatenate(rps), np.concatenate(cols)
    ctx, grp, gcol, call = _search(np.concatenate(parts), sizes, dtype, len(col))
    call()
    assert ctx.status()["code"] == 0
    np.testing.assert_array_equal(grp.cpu().numpy(), rp)
    np.testing.assert_array_equal(gcol.cpu().numpy(), col)
    ctx.close()


def _median_ms(call, reps=7):
    t = []
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        call()
        b.record()
        b.synchronize()
        t.append(a.elapsed_time(b))
    return sorted(t)[reps // 2]


def test_a_large_cloud_among_small_ones_costs_what_it_costs_alone():
    n, small = 500_000, [100] * 500
    large, tiny = _film(n, 0), _film(100, 1)
    ms = []
    for pos, sizes in ((large, [n, 0]), (np.concatenate([large] + [tiny] * len(small)), [n] + small)):
        ctx, _, _, call = _search(pos, sizes, M.F32_REFINED, 60 * pos.shape[0])
        call()
        ms.append(_median_ms(call))
        assert ctx.status()["code"] == 0
        ctx.close()
    # 10 % more particles; a factor of two leaves room for the small clouds' own latencies
    assert ms[1] <= 2.0 * ms[0], ms
