"""The work that users of the operator pipeline have it do, as measurable cases.

A case names an operation (`op`), a particle cloud (`shape`, about `n` particles,
and for a batch the number of `clouds`), the precision (`f64`) and whether the
launch shapes are the library's defaults or the ones its autotuner picks on the
jet cloud (`tuned`).  The clouds are those of paper_2405_13165_gb300.clouds
(a cube on a film sheet, a jet column on a film disc, a curved film, a tray
with puddles, an unstructured cloud), generated on the device so that preparing
them is quick: lattice spacing dx, h = 3.5 dx, jitter of 0.1 dx, fields that are
sums of sinusoids, particles in cell order as a Lagrangian code keeps them
(except the unstructured cloud, which comes in no order).

  step        neighbours, detection, stencils, apply (Pipeline.step)
  neighbours  build_neighbours with the cell order
  stencils    build_stencils over given lists and frames
  apply       apply_ops over given stencils
  gradient    gfdm_operators and the gradient of the sum of squared Laplacians
              with respect to positions and field values
  transition  detection, remap_switched and cell_order over given lists
"""
import math

import torch

from paper_2405_13165_gb300 import mafp as M
from paper_2405_13165_gb300.autograd import gfdm_operators
from paper_2405_13165_gb300.pipeline import Pipeline

DEV = "cuda"
RHO, ETA = 1000.0, 1.0e-3
ROW_3D, ROW_2D = 165.0, 38.5     # usual row lengths at h = 3.5 dx
# what the autotuner picks on the jet cloud
TUNED = {"stencil3d_group": 8, "stencil2d_group": 4, "apply_group": 4, "grad3d_group": 2,
         "grad2d_group": 2, "classify_group": 1}


def _case(name, op, shape, n, f64=False, tuned=False, clouds=1):
    c = {"op": op, "shape": shape, "n": n, "f64": f64, "tuned": tuned, "clouds": clouds}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest cloud that anyone steps: launches and latency count
        _case("step_small", "step", "cube", 5_650),
        # the cleaning jet, a million particles, with tuned launch shapes
        _case("step_jet", "step", "jet", 1_000_000, tuned=True),
        # the double-precision path, for reference solutions
        _case("step_f64", "step", "jet", 60_000, f64=True),
        # uneven clouds of 2k to 200k particles in one call, as ensembles run
        _case("step_batch", "step", "cube", 1_500_000, tuned=True, clouds=32),
        # the first search over particles in no order, with a varying h
        _case("neighbours_random", "neighbours", "random", 199_999),
        # the search of a time loop over a large tray, particles in cell order
        _case("neighbours_tray", "neighbours", "tray", 3_000_000),
        # coefficients of a mostly 3D cloud, default launch shapes
        _case("stencils_cube", "stencils", "cube", 500_000),
        # repeated application inside a solver's iterations
        _case("apply_jet", "apply", "jet", 1_000_000, tuned=True),
        # differentiation, mostly 3D rows
        _case("gradient_cube", "gradient", "cube", 300_000, tuned=True),
        # differentiation, film rows on a curved surface
        _case("gradient_film", "gradient", "film", 400_000),
        # the model transition of a time loop: detection, remap, re-sort
        _case("transition_tray", "transition", "tray", 1_000_000),
    ]


#: op: (shapes, smallest n, largest n) that the listed cases stand for
RANGES = {
    "step": (("cube", "jet", "film"), 5_000, 1_000_000),
    "batch": (("cube",), 100_000, 1_500_000),
    "step_f64": (("cube", "jet", "film"), 5_000, 60_000),
    "neighbours": (("random", "tray", "jet"), 5_000, 2_000_000),
    "stencils": (("cube", "jet", "film"), 5_000, 600_000),
    "apply": (("cube", "jet", "film"), 5_000, 1_000_000),
    "gradient": (("cube", "jet", "film"), 5_000, 300_000),
    "transition": (("tray", "jet"), 5_000, 1_000_000),
}


def draw(rng):
    kind = rng.choice(sorted(RANGES))
    shapes, lo, hi = RANGES[kind]
    shape = rng.choice(shapes)
    n = int(math.exp(rng.uniform(math.log(lo), math.log(hi))))
    if shape == "random":
        n = min(n, 400_000)
    op = {"batch": "step", "step_f64": "step"}.get(kind, kind)
    return _case(None, op, shape, n, f64=kind == "step_f64", tuned=rng.random() < 0.5,
                 clouds=rng.randint(2, 48) if kind == "batch" else 1)


# ------------------------------------------------------------------ the clouds
def _bisect(count, n):
    """The spacing whose lattice holds about n particles."""
    lo, hi = 1e-5, 0.2
    for _ in range(60):
        dx = math.sqrt(lo * hi)
        lo, hi = (dx, hi) if count(dx) > n else (lo, dx)
    return math.sqrt(lo * hi)


def _cube_edges(m3, m2):
    return max(3, int(round(m3))), max(5, int(round(m2)))


def _grid(*axes):
    return [a.reshape(-1) for a in torch.meshgrid(*axes, indexing="ij")]


def _ar(lo, hi):
    return torch.arange(lo, hi, device=DEV)


def _cube(m, s, dx):
    """A cube of m^3 particles on a film sheet of s^2 sites (dx = 0.02 scaled)."""
    off = (s - m) // 2
    i, j, k = _grid(_ar(0, m), _ar(0, m), _ar(0, m))
    face = (i == 0) | (i == m - 1) | (j == 0) | (j == m - 1) | (k == m - 1)
    t3 = torch.where(k == 0, 2, torch.where(face, 1, 0))
    fi, fj = _grid(_ar(0, s), _ar(0, s))
    keep = ~((fi >= off) & (fi < off + m) & (fj >= off) & (fj < off + m))
    fi, fj = fi[keep], fj[keep]
    x3 = torch.stack([(i + off + 0.5) * dx, (j + off + 0.5) * dx, k * dx], 1).double()
    x2 = torch.stack([(fi + 0.5) * dx, (fj + 0.5) * dx, 0 * fi], 1).double()
    return x3, t3, x2


def _jet(dx):
    """A vertical column (radius 0.05, height 0.5) on a film disc of radius 1."""
    nr, nk, nf = int(0.05 / dx), int(0.5 / dx) + 1, int(1.0 / dx)
    i, j = _grid(_ar(-nr, nr + 1), _ar(-nr, nr + 1))
    r = torch.hypot(i * dx, j * dx)
    i, j, r = (a[r <= 0.05] for a in (i, j, r))
    k = _ar(0, nk).repeat(i.numel())
    ring = (r > 0.05 - dx).repeat_interleave(nk)
    t3 = torch.where(k == 0, 2, torch.where(ring | (k == nk - 1), 1, 0))
    x3 = torch.stack([i.repeat_interleave(nk) * dx + 1, j.repeat_interleave(nk) * dx + 1, k * dx],
                     1).double()
    fi, fj = _grid(_ar(-nf, nf + 1), _ar(-nf, nf + 1))
    fr = torch.hypot(fi * dx, fj * dx)
    keep = (fr <= 1.0) & (fr > 0.05)
    fi, fj = fi[keep], fj[keep]
    x2 = torch.stack([fi * dx + 1, fj * dx + 1, 0 * fi], 1).double()
    return x3, t3, x2


def _tray(dx, gen):
    """A 2 x 1 film sheet with puddles of up to 8 layers under Gaussian bumps (as many
    per lattice site as 256 on the sheet of 16 million particles)."""
    ni, nj = int(2.0 / dx), int(1.0 / dx)
    blobs = max(1, round(256 * (4.565e-4 / dx) ** 2))
    u = torch.rand(blobs, 4, generator=gen, dtype=torch.float64)
    L = torch.zeros(ni, nj, device=DEV)
    for cx, cy, sg, am in u.tolist():
        cx, cy, sg, am = 0.1 + 1.8 * cx, 0.1 + 0.8 * cy, (10 + 30 * sg) * dx, 2 + 6 * am
        i0, i1 = max(0, int((cx - 3 * sg) / dx)), min(ni, int((cx + 3 * sg) / dx) + 1)
        j0, j1 = max(0, int((cy - 3 * sg) / dx)), min(nj, int((cy + 3 * sg) / dx) + 1)
        xs, ys = (_ar(i0, i1) + 0.5) * dx - cx, (_ar(j0, j1) + 0.5) * dx - cy
        b = am * torch.exp(-(xs[:, None] ** 2 + ys[None, :] ** 2) / (2 * sg * sg))
        L[i0:i1, j0:j1] = torch.maximum(L[i0:i1, j0:j1], b)
    L = torch.floor(L + 0.5).long()
    pi, pj = torch.nonzero(L, as_tuple=True)
    top = L[pi, pj]
    first = torch.cumsum(top, 0) - top
    pk = _ar(0, int(top.sum())) - first.repeat_interleave(top)
    pi, pj, top = (a.repeat_interleave(top) for a in (pi, pj, top))
    P = torch.nn.functional.pad(L, (1, 1, 1, 1))
    side = torch.minimum(torch.minimum(P[pi, pj + 1], P[pi + 2, pj + 1]),
                         torch.minimum(P[pi + 1, pj], P[pi + 1, pj + 2]))
    t3 = torch.where(pk == 0, 2, torch.where((pk == top - 1) | (side <= pk), 1, 0))
    x3 = torch.stack([(pi + 0.5) * dx, (pj + 0.5) * dx, pk * dx], 1).double()
    fi, fj = torch.nonzero(L == 0, as_tuple=True)
    x2 = torch.stack([(fi + 0.5) * dx, (fj + 0.5) * dx, 0 * fi], 1).double()
    return x3, t3, x2


def _cell_order(x, h):
    """Stable order by cells of edge just above max h, from the lower corner."""
    lo, c = x.amin(0), float(h.max()) * (1.0 + 1e-6)
    dim = torch.floor((x.amax(0) - lo) / c).long() + 1
    q = torch.minimum(torch.floor((x - lo) * (1.0 / c)).long(), dim - 1)
    return torch.argsort((q[:, 2] * dim[1] + q[:, 1]) * dim[0] + q[:, 0], stable=True)


def _cloud(shape, n, seed, sort=True, edges=None):
    """One cloud's arrays in 32 bits (what a program holds before it calls).  The
    lattice goes by shape and n, what is drawn on it by the seed."""
    cpu = torch.Generator().manual_seed(seed)
    gen = torch.Generator(device=DEV).manual_seed(seed + 1)
    rnd = lambda *s: torch.rand(*s, generator=gen, device=DEV, dtype=torch.float64)
    normal = None
    if shape == "cube":
        # edge 0.3 and sheet 1.0 at the spacing that gives n, or a batch's own edges
        dx = 0.02 if edges else _bisect(lambda d: (0.3 / d) ** 3 + 0.91 / d ** 2, n)
        m, s = edges or _cube_edges(0.3 / dx, 1.0 / dx)
        x3, t3, x2 = _cube(m, s, dx)
    elif shape == "jet":
        dx = _bisect(lambda d: math.pi * (0.00125 / d ** 3 + 0.9975 / d ** 2), n)
        x3, t3, x2 = _jet(dx)
    elif shape == "tray":
        dx = math.sqrt(2.45 / n)
        x3, t3, x2 = _tray(dx, torch.Generator().manual_seed(n))
    elif shape == "film":
        # a spherical cap of radius 1 up to 0.6 of it
        dx = math.sqrt(math.pi * 0.36 / n)
        k = int(0.6 / dx)
        i, j = _grid(_ar(-k, k + 1), _ar(-k, k + 1))
        keep = (i * dx) ** 2 + (j * dx) ** 2 <= 0.6 ** 2
        x2 = torch.stack([i[keep] * dx, j[keep] * dx, 0 * i[keep]], 1).double()
        x3, t3 = x2[:0], torch.zeros(0, dtype=torch.long, device=DEV)
    else:                                  # "random": no lattice, a varying h
        n2 = int(n ** (2 / 3))
        dx = n ** (-1 / 3)
        x3, x2 = rnd(n - n2, 3), rnd(n2, 3)
        x2[:, 2] = 0
        t3 = torch.randint(0, 3, (n - n2,), generator=gen, device=DEV)
    xyz = torch.cat([x3, x2])
    n = xyz.shape[0]
    model = torch.zeros(n, dtype=torch.uint8, device=DEV)
    model[x3.shape[0]:] = 1
    ptype = torch.cat([t3, torch.full((x2.shape[0],), 2, device=DEV)]).to(torch.uint8)
    wall = ptype == 2
    h = torch.full((n,), 3.5 * dx, dtype=torch.float64, device=DEV)
    if shape == "random":
        h = h * (0.8 + 0.4 * rnd(n))
    else:
        jit = (rnd(n, 3) - 0.5) * (0.2 * dx)
        jit[wall, 2] = 0
        xyz = xyz + jit
    if shape == "film":
        xyz[:, 2] = 1 - torch.sqrt(1 - xyz[:, 0] ** 2 - xyz[:, 1] ** 2)
        normal = torch.tensor([0.0, 0.0, 1.0], device=DEV, dtype=torch.float64) - xyz
    pos_h = torch.cat([xyz, h[:, None]], 1).float()
    xyz = pos_h[:, :3].double()
    vp = torch.zeros(n, 4, dtype=torch.float64, device=DEV)
    for f in range(4):
        for _ in range(4):
            d = torch.randn(3, generator=cpu, dtype=torch.float64)
            r = torch.rand(2, generator=cpu, dtype=torch.float64)
            kap = (d / d.norm() * (1 + 7 * r[0])).to(DEV)
            vp[:, f] += torch.sin(xyz @ kap + 2 * math.pi * float(r[1]))
    nrm = torch.zeros(n, 4, device=DEV)
    nrm[wall, 2] = 1.0
    if normal is not None:
        nrm[:, :3] = normal.float()
    vol = torch.where(model == 0, dx ** 3, 0.3 * dx ** 3)
    hfilm = torch.where(model == 1, 0.3 * dx, 0.0)
    one = torch.ones(n, device=DEV)
    c = {"pos_h": pos_h, "model": model, "ptype": ptype, "normal": nrm, "vp": vp.float(),
         "rho": RHO * one, "eta": ETA * one, "mass": (RHO * vol).float(),
         "diam": torch.pow(6 * vol / math.pi, 1 / 3).float(), "hfilm": hfilm.float(),
         "h3d": pos_h[:, 3].clone(), "user": torch.zeros_like(model),
         "last": torch.zeros_like(model), "vol": vol.float()}
    if shape == "tray":
        # the sweeping sphere of the tray loop: film inside it is asked to become 3D,
        # 3D matter in the shell that it has just left to become a film
        d2 = (xyz - torch.tensor([1.0, 0.5, 0.0], device=DEV, dtype=torch.float64)).square().sum(1)
        c["user"][(d2 < 0.2 ** 2) & (model == 1)] = M.USER_TO_3D
        c["user"][(d2 >= 0.2 ** 2) & (d2 < 0.29 ** 2) & (model == 0) & (xyz[:, 0] < 1)] = \
            M.USER_TO_2D
    if sort:
        o = _cell_order(xyz, pos_h[:, 3].double())
        c = {k: v[o].contiguous() for k, v in c.items()}
    return c


def _inputs(case, seed):
    """The arrays of a case: one cloud, or a batch of them stored back to back."""
    if case["clouds"] == 1:
        return _cloud(case["shape"], case["n"], seed, case["shape"] != "random")
    cpu = torch.Generator().manual_seed(case["n"] + case["clouds"])
    u = torch.rand(case["clouds"], 2, generator=cpu, dtype=torch.float64).tolist()
    size = [2_000 * 100 ** a for a, _ in u]
    scale = case["n"] / sum(size)
    parts = []
    for b, (sz, (_, f)) in enumerate(zip(size, u)):
        sz, f = max(1_000.0, sz * scale), 0.1 + 0.8 * f
        m = ((1 - f) * sz) ** (1 / 3)
        parts.append(_cloud("cube", 0, 1000 * seed + b + 1, True,
                            _cube_edges(m, max(m + 2, math.sqrt(f * sz + m * m)))))
    c = {k: torch.cat([p[k] for p in parts]) for k in parts[0]}
    count = torch.tensor([0] + [p["pos_h"].shape[0] for p in parts])
    c["cloud_offset"] = torch.cumsum(count, 0).to(DEV)
    return c


def _capacity(case, model):
    """Room for the lists' entries: the support's volume per particle, and a little over."""
    n2 = int(model.sum())
    row = 220 if case["shape"] == "random" else 185
    return row * (model.numel() - n2) + 40 * n2


def prepare(case, seed):
    dt = M.F64 if case["f64"] else M.F32_REFINED
    rd = M.real_dtype(dt)
    d = {k: v.to(rd) if v.dtype == torch.float32 else v for k, v in _inputs(case, seed).items()}
    d["fields"], d["type"] = d["vp"], d["ptype"]
    n = d["pos_h"].shape[0]
    ctx = M.Context(n + n // 4)
    if case["tuned"]:
        ctx.set_tuning(**TUNED)
    cap = _capacity(case, d["model"])
    p = Pipeline(ctx, n, 1 if case["op"] == "neighbours" else cap, dt)
    s = {"op": case["op"], "d": d, "n": n, "pipe": p, "ctx": ctx, "dt": dt}
    if case["op"] == "neighbours":        # no room for coefficients
        p.col = torch.zeros(cap, dtype=torch.int32, device=DEV)
    elif case["op"] != "step":
        p.neighbours(d)
        if case["op"] == "transition":
            room = n + n // 4
            s["out"] = {k: torch.zeros((room,) + d[k].shape[1:], dtype=d[k].dtype, device=DEV)
                        for k in M.STATE_F4 + M.STATE_F1 + M.STATE_U8}
            s["old2new"] = torch.zeros(n, dtype=torch.int32, device=DEV)
            s["n_out"] = torch.zeros(1, dtype=torch.int64, device=DEV)
            s["order"] = torch.zeros(n, dtype=torch.int32, device=DEV)
            return s
        p.classify(d)
        if case["op"] == "apply":
            p.stencils(d)
        if case["op"] == "gradient":
            d["pos_h"].requires_grad_()
            d["fields"] = d["fields"].clone().requires_grad_()
    return s


def run(s):
    p, d, n = s["pipe"], s["d"], s["n"]
    if s["op"] == "step":
        p.step(d)
        return {"row_ptr": p.row_ptr, "col": p.col, "flag": p.flag, "eig": p.eig,
                "frame": p.frame, "hfilm": p.hfilm, "coef": p.coef, "status": p.status,
                "out": p.out}
    if s["op"] == "neighbours":
        p.neighbours(d, with_order=True)
        return {"row_ptr": p.row_ptr, "col": p.col, "order": p.order}
    if s["op"] == "stencils":
        p.stencils(d)
        return {"coef": p.coef, "status": p.status}
    if s["op"] == "apply":
        p.apply(d)
        return {"out": p.out}
    if s["op"] == "gradient":
        out = gfdm_operators(s["ctx"], d["pos_h"], d["fields"], p.row_ptr, p.col, d["model"],
                             p.frame, s["dt"])
        gpos, gfields = torch.autograd.grad(out[:, :, 3].square().sum(),
                                            (d["pos_h"], d["fields"]))
        return {"out": out, "gpos": gpos, "gfields": gfields}
    p.classify(d)
    M.remap_switched(s["ctx"], n, d, p.flag, p.row_ptr, p.col, s["out"],
                     s["out"]["rho"].shape[0], s["old2new"], s["n_out"], s["dt"])
    M.cell_order(s["ctx"], d["pos_h"], s["order"], s["dt"])
    return {"flag": p.flag, "eig": p.eig, "frame": p.frame, "hfilm": p.hfilm, "state": s["out"],
            "old2new": s["old2new"], "n_out": s["n_out"], "order": s["order"]}


# ------------------------------------------------------------------- the work
def _counts(case):
    """About how many 3D and film particles a case holds."""
    n, shape = float(case["n"]), case["shape"]
    if case["clouds"] > 1:
        return 0.5 * n, 0.5 * n
    if shape == "cube":
        dx = _bisect(lambda d: (0.3 / d) ** 3 + 0.91 / d ** 2, n)
        return (0.3 / dx) ** 3, 0.91 / dx ** 2
    if shape == "jet":
        dx = _bisect(lambda d: math.pi * (0.00125 / d ** 3 + 0.9975 / d ** 2), n)
        return math.pi * 0.00125 / dx ** 3, math.pi * 0.9975 / dx ** 2
    if shape == "tray":
        return 0.375 * n, 0.625 * n
    return (0.0, n) if shape == "film" else (n, 0.0)


def work(case):
    n3, n2 = _counts(case)
    e3, e2 = n3 * (ROW_3D if case["shape"] != "tray" else 90.0), n2 * ROW_2D
    n, e, r = n3 + n2, e3 + e2, 8.0 if case["f64"] else 4.0
    lists = 4 * e + 8 * n
    search = {"bytes": 4 * r * n + lists, "flops": 11 * e}
    detect = {"bytes": lists + r * n * (4 + 4 + 1 + 1 + 4 + 8 + 1) + 6 * n, "flops": 25 * e2 + 150 * n2}
    build = {"bytes": lists + r * n * 12 + 2 * n + 4 * n + 4 * r * e,
             "flops": 210 * e3 + 1200 * n3 + 90 * e2 + 1000 * n2}
    apply_ = {"bytes": lists + 4 * r * e + r * n * 20, "flops": 36 * e}
    back = {"bytes": lists + 4 * r * e + r * n * (16 + 4 + 12 + 4 + 4),
            "flops": 32 * e + 525 * e3 + 225 * e2}
    remap = {"bytes": 2 * n * (18 * r + 3) + 6 * n, "flops": 10 * n}
    parts = {"step": (search, detect, build, apply_), "neighbours": (search,),
             "stencils": (build,), "apply": (apply_,), "gradient": (build, apply_, back),
             "transition": (detect, remap)}[case["op"]]
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


# ------------------------------------------------- the same in plain 64 bits
ALPHA = 4.0        # the weight W(s) = (exp(-4 s^2) - e^-4) / (1 - e^-4)


def _lists(pos):
    """Neighbour lists |x_j - x_i| <= (h_i + h_j) / 2 of one cloud (row_ptr, col)."""
    n = pos.shape[0]
    x, h = pos[:, :3], pos[:, 3]
    lo, c = x.amin(0), float(h.max()) * (1 + 1e-6)
    q = torch.floor((x - lo) / c).long()
    dim = q.amax(0) + 1
    key = (q[:, 2] * dim[1] + q[:, 1]) * dim[0] + q[:, 0]
    skey, order = torch.sort(key, stable=True)
    begin, length = [], []
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            y, z = q[:, 1] + dy, q[:, 2] + dz
            ok = (y >= 0) & (y < dim[1]) & (z >= 0) & (z < dim[2])
            row = (z * dim[1] + y) * dim[0]
            a = torch.searchsorted(skey, row + torch.clamp(q[:, 0] - 1, min=0))
            b = torch.searchsorted(skey, row + torch.minimum(q[:, 0] + 1, dim[0] - 1), right=True)
            begin.append(a)
            length.append(torch.where(ok, b - a, 0))
    begin, length = torch.stack(begin, 1), torch.stack(length, 1)
    total = torch.cumsum(length.sum(1), 0).cpu()
    counts, cols, r0 = torch.zeros(n, dtype=torch.long, device=DEV), [], 0
    while r0 < n:
        base = int(total[r0 - 1]) if r0 else 0
        r1 = max(r0 + 1, int(torch.searchsorted(total, base + 30_000_000)))
        ln = length[r0:r1].reshape(-1)
        run_of = torch.repeat_interleave(torch.arange(ln.numel(), device=DEV), ln)
        at = torch.arange(run_of.numel(), device=DEV) - (torch.cumsum(ln, 0) - ln)[run_of]
        i = r0 + run_of // 9
        j = order[begin[r0:r1].reshape(-1)[run_of] + at]
        dd = (x[j] - x[i]).square()
        hit = (dd[:, 0] + dd[:, 1]) + dd[:, 2] <= ((h[i] + h[j]) * 0.5).square()
        i, j = i[hit], j[hit]
        both = torch.sort(i * n + j).values
        counts += torch.bincount(both // n, minlength=n)
        cols.append(both % n)
        r0 = r1
    return torch.cat([torch.zeros(1, dtype=torch.long, device=DEV), torch.cumsum(counts, 0)]), \
        torch.cat(cols)


def _rows(rows, row_ptr, col):
    """Columns of the given rows, padded with the row's own particle, and which are real."""
    ln = row_ptr[rows + 1] - row_ptr[rows]
    k = torch.arange(int(ln.max()), device=DEV)
    real = k[None, :] < ln[:, None]
    e = torch.where(real, row_ptr[rows][:, None] + k, 0)
    return torch.where(real, col[e], rows[:, None]), real, e


def _row_ops(x, hi, u, rows, j, same, film):
    """Coefficients [rows, K, 4] and outputs [rows, 4, 4] of rows of one model."""
    xi = x[rows]
    y = (x[j] - xi[:, None, :]) / hi[:, None, None]
    s2 = y.square().sum(2)
    ea = math.exp(-ALPHA)
    w = torch.where(same & (s2 <= 1), (torch.exp(-ALPHA * s2) - ea) / (1 - ea), 0.0)
    one = torch.ones_like(s2)
    if film:
        m = same.double()[:, :, None]
        z = (y - (y * m).sum(1, keepdim=True) / m.sum(1, keepdim=True)) * m
        scatter = z.transpose(1, 2) @ z
        lam, vec = torch.linalg.eigh(scatter.detach())
        n0 = vec[:, :, 0]
        # first-order change of the normal with the scatter matrix (zero at the value itself)
        gap = 1 / (lam[:, 1:] - lam[:, :1])
        pull = torch.einsum("nak,nk,nbk->nab", vec[:, :, 1:], gap, vec[:, :, 1:])
        nv = n0 - (pull @ (scatter @ n0[:, :, None]))[:, :, 0]
        nv = nv / nv.norm(dim=1, keepdim=True)
        t1 = vec[:, :, 2]
        t1 = t1 - (t1 * nv).sum(1, keepdim=True) * nv
        t1 = t1 / t1.norm(dim=1, keepdim=True)
        t2 = torch.linalg.cross(nv, t1)
        a, b = (y * t1[:, None, :]).sum(2), (y * t2[:, None, :]).sum(2)
        p = torch.stack([one, a, b, a * a, a * b, b * b], 2)
        rhs = torch.zeros(6, 3, device=DEV, dtype=torch.float64)
        rhs[1, 0] = rhs[2, 1] = 1
        rhs[3, 2] = rhs[5, 2] = 2
    else:
        a, b, c = y.unbind(2)
        p = torch.stack([one, a, b, c, a * a, b * b, c * c, a * b, a * c, b * c], 2)
        rhs = torch.zeros(10, 4, device=DEV, dtype=torch.float64)
        rhs[1, 0] = rhs[2, 1] = rhs[3, 2] = 1
        rhs[4:7, 3] = 2
    A = (p * w[:, :, None]).transpose(1, 2) @ p
    lam = torch.linalg.solve(A, rhs.expand(A.shape[0], -1, -1))
    co = w[:, :, None] * (p @ lam)
    hk = hi[:, None, None]
    if film:
        co = torch.cat([(co[:, :, :1] * t1[:, None, :] + co[:, :, 1:2] * t2[:, None, :]) / hk,
                        co[:, :, 2:] / hk ** 2], 2)
    else:
        co = torch.cat([co[:, :, :3] / hk, co[:, :, 3:] / hk ** 2], 2)
    du = u[j] - u[rows][:, None, :]
    return co, du.transpose(1, 2) @ co


def exact(case, seed):
    op = case["op"]
    n3, n2 = _counts(case)
    if op in ("neighbours", "transition") or n3 * ROW_3D + n2 * ROW_2D > 1e8:
        return None
    d = _inputs(case, seed)
    off = d["cloud_offset"].tolist() if case["clouds"] > 1 else [0, d["pos_h"].shape[0]]
    pos, u, model = d["pos_h"].double(), d["vp"].double(), d["model"]
    parts = [_lists(pos[a:b]) for a, b in zip(off[:-1], off[1:])]
    n, at, row_ptr = pos.shape[0], 0, [torch.zeros(1, dtype=torch.long, device=DEV)]
    for rp, c in parts:
        row_ptr.append(rp[1:] + at)
        at += c.numel()
    row_ptr = torch.cat(row_ptr)
    col = torch.cat([c + a for (_, c), a in zip(parts, off[:-1])])
    x, h = pos[:, :3].clone(), pos[:, 3]
    grad = op == "gradient"
    coef = torch.zeros(_capacity(case, model) if not grad else 1, 4, device=DEV,
                       dtype=torch.float64)
    out = torch.zeros(n, 4, 4, device=DEV, dtype=torch.float64)
    gx, gu = torch.zeros_like(x), torch.zeros_like(u)
    for film in (False, True):
        for rows in torch.split(torch.nonzero(model == int(film))[:, 0], 8192):
            if not rows.numel():
                continue
            j, real, e = _rows(rows, row_ptr, col)
            same = real & (model[j] == model[rows][:, None])
            xx, uu = x.detach().requires_grad_(grad), u.detach().requires_grad_(grad)
            with torch.set_grad_enabled(grad):
                co, o = _row_ops(xx, h[rows], uu, rows, j, same, film)
                if grad:
                    a, b = torch.autograd.grad(o[:, :, 3].square().sum(), (xx, uu))
                    gx += a
                    gu += b
            out[rows] = o.detach()
            if not grad:
                coef[e[real]] = co[real]
    if grad:
        return {"out": out, "gpos": torch.cat([gx, torch.zeros_like(h)[:, None]], 1),
                "gfields": gu}
    if op == "apply":
        return {"out": out}
    return dict({"coef": coef, "status": None},
                **({k: None for k in ("row_ptr", "col", "flag", "eig", "frame", "hfilm")}
                   if op == "step" else {}), **({"out": out} if op == "step" else {}))
