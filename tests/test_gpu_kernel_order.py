"""Inside a call too, what the overlapping kernels compute has to be that of kernels run
one after another: the chains of the whole library -- unordered and batched searches,
detection, transition and cell order into the next search, stencils, application and film
momentum, both adjoints, the buffer zone -- run back to back here and, for the values to
compare with, in a process that waits after every kernel (CUDA_LAUNCH_BLOCKING)."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2405_13165_gb300 import clouds as C

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2405_13165_gb300 import mafp as M  # noqa: E402
from paper_2405_13165_gb300.ghosts import GhostZone, empty_state  # noqa: E402
from paper_2405_13165_gb300.pipeline import Pipeline, cloud_to_device  # noqa: E402

# summed by atomics in an order that varies; everything else comes out bit for bit
BY_ATOMICS = ("gpos", "gscatter", "stress", "flux")


def _zeros_like_state(d, room):
    return {k: torch.zeros((room,) + tuple(d[k].shape[1:]), dtype=d[k].dtype, device="cuda")
            for k in M.STATE_F4 + M.STATE_F1 + M.STATE_U8}


def chains(dtype):
    """{name: tensor} of every chain's results, nothing waited for but particle counts."""
    out = {}
    rng = np.random.default_rng(5)
    # an unordered cloud beyond the one-block sort, then everything on its lists
    c = C.cube_on_sheet(0.016, seed=C.SEED_BASE + 40)
    assert c.n > 8192
    c = c.take(rng.permutation(c.n))
    c.user[:] = 0
    c.user[(c.model == 1) & (c.pos_h[:, 0] < 0.3)] = M.USER_TO_3D
    c.user[(c.model == 0) & (c.pos_h[:, 0] > 0.5)] = M.USER_TO_2D
    n = c.n
    d = cloud_to_device(c, dtype)
    d["type"] = d["ptype"]
    ctx = M.Context(2 * n)
    p = Pipeline(ctx, 2 * n, 400 * n, dtype)
    p.neighbours(d, with_order=True)
    p.classify(d)
    p.stencils(d)
    p.apply(d)
    vp = d["vp"].clone()
    M.film_momentum(ctx, d["model"], vp, d["rho"], d["eta"], d["hfilm"], d["normal"], p.out[:n],
                    (0.3, 0.0, -9.81), 1e-4, dtype)
    stress = torch.zeros(2, dtype=torch.float64, device="cuda")
    M.normal_stress(ctx, d["model"], p.out[:n], d["eta"], d["normal"], stress, dtype)
    flux = torch.zeros(2, dtype=torch.float64, device="cuda")
    moved = d["pos_h"] + torch.tensor([0.05, 0, 0, 0], dtype=d["pos_h"].dtype, device="cuda")
    M.plane_flux(ctx, d["pos_h"], moved, d["mass"], d["rho"], (0.5, 0, 0), (1, 0, 0), flux, dtype)
    rp, col = p.row_ptr[: n + 1], p.col
    tloc = torch.zeros(col.numel(), dtype=torch.int16, device="cuda")
    M.transpose_map(ctx, rp, col, tloc)
    gmap, gscatter, gpos = (torch.zeros_like(d["pos_h"]) for _ in range(3))
    M.apply_ops_backward(ctx, rp, col, tloc, p.coef, p.out[:n], gmap, dtype)
    M.apply_ops_backward(ctx, rp, col, None, p.coef, p.out[:n], gscatter, dtype)
    M.build_stencils_backward(ctx, d["pos_h"], d["model"], p.frame[:n], rp, col, gmap, p.out[:n],
                              gpos, dtype)
    # the transition's cloud sorted and searched
    state = _zeros_like_state(d, 2 * n)
    old2new = torch.zeros(n, dtype=torch.int32, device="cuda")
    n_out = torch.zeros(1, dtype=torch.int64, device="cuda")
    M.remap_switched(ctx, n, d, p.flag, rp, col, state, 2 * n, old2new, n_out, dtype)
    k = int(n_out.item())
    order = torch.zeros(k, dtype=torch.int32, device="cuda")
    q = Pipeline(ctx, 2 * n, 400 * n, dtype)
    M.cell_order(ctx, state["pos_h"][:k], order, dtype)
    q.neighbours({"pos_h": state["pos_h"][:k]})
    out.update(row_ptr=rp, col=col, order=p.order[:n], flag=p.flag[:n], eig=p.eig[:n],
               frame=p.frame[:n], hfilm=p.hfilm[:n], coef=p.coef, status=p.status[:n],
               out=p.out[:n], vp=vp, stress=stress, flux=flux, tloc=tloc, gmap=gmap,
               gscatter=gscatter, gpos=gpos, old2new=old2new, order2=order,
               row_ptr2=q.row_ptr[: k + 1], col2=q.col)
    out.update({"state_" + key: v[:k] for key, v in state.items()})
    # a batch in no order
    parts = [C.random_cloud(m, 7 + m) for m in (3000, 1, 9000, 40)]
    b = C.concat(parts)
    off = np.concatenate([[0], np.cumsum([x.n for x in parts])])
    d = cloud_to_device(b, dtype, cloud_offset=off)
    r = Pipeline(ctx, 2 * n, 400 * n, dtype)
    r.neighbours(d, with_order=True)
    r.classify(d)
    out.update(b_row_ptr=r.row_ptr[: b.n + 1], b_col=r.col, b_order=r.order[: b.n],
               b_eig=r.eig[: b.n])
    # the buffer zone
    c = C.interface_strip(dx=0.02, quadratic=True, columns=True)
    S = empty_state(2 * c.n, dtype)
    for key, v in S.items():
        a = torch.from_numpy(np.asarray(getattr(c, {"type": "ptype"}.get(key, key))))
        v[: c.n] = a.to("cuda", v.dtype)
    zctx = M.Context(2 * c.n)
    z = Pipeline(zctx, 2 * c.n, 400 * c.n, dtype)
    z.neighbours({"pos_h": S["pos_h"][: c.n]})
    rp, col = z.csr(c.n)
    n_all, _, _ = GhostZone(zctx, 2 * c.n, c.n, 4 * c.n, 400 * c.n, dtype).build(S, c.n, rp, col)
    z.neighbours({"pos_h": S["pos_h"][:n_all]})
    out.update({"z_" + key: v[:n_all] for key, v in S.items()}, z_row_ptr=z.row_ptr[: n_all + 1],
               z_col=z.col)
    torch.cuda.synchronize()
    for x in (ctx, zctx):
        assert x.status()["code"] == 0, x.status()
    return {k: v.cpu() for k, v in out.items()}


@pytest.mark.parametrize("dtype", [M.F32_REFINED, M.F64])
def test_overlapping_kernels_equal_waited_ones(dtype, tmp_path):
    here = os.path.dirname(os.path.abspath(__file__))
    path = str(tmp_path / "want.pt")
    code = (f"import sys; sys.path[:0] = [{os.path.dirname(here)!r}, {here!r}]; import torch; "
            f"import test_gpu_kernel_order as t; torch.save(t.chains({int(dtype)}), {path!r})")
    subprocess.run([sys.executable, "-c", code], check=True, timeout=600,
                   env=dict(os.environ, CUDA_LAUNCH_BLOCKING="1"))
    want = torch.load(path)
    for _ in range(4):
        got = chains(dtype)
        assert got.keys() == want.keys()
        for k, w in want.items():
            if k in BY_ATOMICS:
                # sums of up to ~700 terms (or one per particle) in another order
                eps = 2.0 ** -53 if w.dtype == torch.float64 else 2.0 ** -24
                terms = 700 if w.numel() > 2 else 20_000
                assert (got[k] - w).abs().max() <= 2 * terms * eps * w.abs().max(), k
            else:
                assert torch.equal(got[k], w), k
