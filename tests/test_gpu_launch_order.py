"""The library's kernels overlap their set-up with the kernel before them; what they
compute has to be that of kernels run one after another: calls on fresh inputs
back to back without a wait between them, on the default stream and on another
one, across a memset and torch kernels in between, and replayed from a CUDA
graph, each equal to the same calls with a device synchronisation after each."""
import numpy as np
import pytest

from paper_2405_13165_gb300 import clouds as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_13165_gb300 import mafp as M  # noqa: E402
from paper_2405_13165_gb300.pipeline import Pipeline, cloud_to_device  # noqa: E402

KEYS = ("row_ptr", "col", "flag", "frame", "coef", "status", "out")


def _inputs(k, shuffled):
    c = C.cube_on_sheet(0.02, seed=C.SEED_BASE + 100 + k)
    if shuffled:
        c = c.take(np.random.default_rng(k).permutation(c.n))
    else:
        c = C.cell_sorted(c)
    return cloud_to_device(c)


def _clear(p):
    for k in KEYS:
        getattr(p, k).zero_()


def _calls(p, d, wait):
    for call in (p.neighbours, p.classify, p.stencils, p.apply):
        call(d)
        if wait:
            torch.cuda.synchronize()


@pytest.mark.parametrize("where", ["default", "stream", "graph"])
def test_back_to_back_calls_equal_waited_ones(where):
    ds = [_inputs(k, k % 2 == 1) for k in range(6)]
    n = ds[0]["pos_h"].shape[0]
    ctx = M.Context(n)
    p = Pipeline(ctx, n, 200 * n)
    want = []
    for d in ds:
        _clear(p)
        _calls(p, d, True)
        want.append({k: getattr(p, k).clone() for k in KEYS})
    torch.cuda.synchronize()
    got = [{k: torch.empty_like(v) for k, v in want[0].items()} for _ in ds]

    def one(d, g):
        _clear(p)
        _calls(p, d, False)
        for k in KEYS:
            g[k].copy_(getattr(p, k))

    stream = torch.cuda.Stream() if where != "default" else torch.cuda.current_stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        if where == "graph":
            one(ds[0], got[0])   # (nothing is set up for the first time under capture)
            stream.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=stream):
                for d, o in zip(ds, got):
                    one(d, o)
            for o in got:
                for v in o.values():
                    v.zero_()
            for _ in range(3):
                g.replay()
        else:
            for _ in range(3):
                for d, o in zip(ds, got):
                    one(d, o)
    torch.cuda.synchronize()
    assert ctx.status()["code"] == 0
    for w, o in zip(want, got):
        for k in KEYS:
            assert torch.equal(w[k], o[k]), k
    ctx.close()
