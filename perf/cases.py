"""Performance cases of the LGF library: the calls a flow solver makes.

A case is a dict of plain values: the operation (``op``), the shape of the
block sets (``layout`` and its sizes), the block edge, the precision, the
number of fields and the kernel's parameter.  ``prepare`` builds the inputs on
the GPU, ``run`` makes one pass through the public entry points and ``exact``
gives the same result in 64 bits from plain torch.  One context per precision
lives for the whole process, as in a solver that applies the operators to new
fields in every step; plans and spectra are built by the first pass on a
geometry.

Operations
  poisson    u = dx^2 G_L * f
  kinv       u = dx^2 G_K(alpha) * f
  intfactor  u = E(alpha) f
  step       one batch: G_L and three E(alpha) of the same field
  batch      one batch: G_L, then E(alpha), of many flat-plate problems
  refresh    u <- -C^dagger L^{-1} C u
  stage      one IF-HERK stage by the nested projection
  ib         marker forces spread onto the faces, velocities read back

Layouts (all counts in blocks)
  box        nx x ny x nz blocks, sources and targets on all of them
  scattered  nsrc source and ntgt target blocks drawn from a box (own layout_seed)
  sphere     a ball of `radius` and a wake cylinder; sources on the blocks that
             the sphere of markers touches (surface = 1) or on every block; with
             surface = 2 the touched blocks are sources and targets
  wake       the part `frac` of an nx x ny x nz box around a ball and its wake
  plates     nprob flat plates, nb_lo..nb_hi target blocks each (own layout_seed)
"""
import math
import random
from functools import lru_cache

import numpy as np
import torch

import paper_1604_01814_gb300 as lgf

DEV = "cuda:0"
STEP_ALPHAS = (0.05, 0.5, 2.0)
# the work of the largest listed case: lattice points of the box times fields
MOST_POINTS = 512 * 256 * 256 * 12


# ----------------------------------------------------------------------------
# cases
# ----------------------------------------------------------------------------
def listed():
    sphere = dict(layout="sphere", b=16, radius=4.0, wake_len=12.0, wake_radius=3.0, radius_cells=20.0, markers=5120)
    return [
        # latency: a handful of 8^3 blocks around a small body, and the plain
        # method's single 32^3 box in FP64
        dict(name="scattered_f32", op="poisson", layout="scattered", b=8, ex=4, ey=3, ez=3, nsrc=5, ntgt=7,
             layout_seed=5, prec="f32", fields=3),
        dict(name="box32_f64", op="poisson", layout="box", b=32, nx=1, ny=1, nz=1, prec="f64", fields=1),
        # a smooth dense 128^3 box: one batch of G_L and three integrating factors
        dict(name="step128_f32", op="step", layout="box", b=32, nx=4, ny=4, nz=4, prec="f32", fields=1),
        # the sphere with its wake (556 blocks of 16^3): body forces to the whole
        # flow, in both precisions
        dict(name="sphere_poisson_f32", op="poisson", surface=1, prec="f32", fields=3, **sphere),
        dict(name="sphere_poisson_f64", op="poisson", surface=1, prec="f64", fields=3, **sphere),
        # the viscous integrating factor of the whole flow, and the force
        # operator's K(alpha)^-1 from the body's blocks to themselves
        dict(name="sphere_intfactor_f32", op="intfactor", surface=0, prec="f32", fields=3, alpha=0.25, **sphere),
        dict(name="sphere_kinv_f32", op="kinv", surface=2, prec="f32", fields=3, alpha=0.25, **sphere),
        # the periodic velocity refresh and one whole stage of the time stepper
        dict(name="sphere_refresh_f32", op="refresh", surface=0, prec="f32", fields=3, **sphere),
        dict(name="sphere_stage_f32", op="stage", surface=0, prec="f32", fields=3, alpha=0.05, **sphere),
        # the immersed-boundary operators of 5120 markers
        dict(name="sphere_ib_f32", op="ib", surface=0, prec="f32", fields=3, **sphere),
        # a parameter study: 64 uneven flat-plate problems as one batch
        dict(name="plates64_f32", op="batch", layout="plates", b=16, nprob=64, nb_lo=8, nb_hi=1200, layout_seed=3,
             prec="f32", fields=3, alpha=0.25),
        # a large wake: 3 components x 4 right-hand sides of a 512x256x256 box
        dict(name="wake512_f32", op="poisson", layout="wake", b=32, nx=16, ny=8, nz=8, frac=0.4, prec="f32",
             fields=12),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _draw_layout(rng, kind, b):
    n = lambda lo, hi: int(round(_log(rng, lo / b, hi / b))) or 1   # noqa: E731  extents in points
    if kind == "box":
        return dict(nx=n(8, 256), ny=n(8, 256), nz=n(8, 256))
    if kind == "wake":
        return dict(nx=max(2, n(64, 512)), ny=max(2, n(32, 256)), nz=max(2, n(32, 256)),
                    frac=round(rng.uniform(0.2, 0.8), 3))
    if kind == "scattered":
        ex, ey, ez = n(8, 160), n(8, 128), n(8, 128)
        most = ex * ey * ez
        return dict(ex=ex, ey=ey, ez=ez, nsrc=min(most, int(_log(rng, 1, most + 1))),
                    ntgt=min(most, int(_log(rng, 1, most + 1))), layout_seed=rng.randrange(1 << 20))
    rc = _log(rng, 5.0, 28.0)   # sphere: radius of the body in cells
    radius = (rc + 4.0) / b + rng.uniform(0.7, 3.0)
    return dict(radius=round(radius, 3), wake_len=round(radius * rng.uniform(1.0, 3.5), 3),
                wake_radius=round(radius * rng.uniform(0.4, 0.9), 3), radius_cells=round(rc, 2),
                markers=int(4.0 * math.pi * rc * rc * rng.uniform(0.7, 1.1)))


def draw(rng: random.Random):
    while True:
        op = rng.choice(["poisson", "poisson", "intfactor", "step", "kinv", "refresh", "stage", "ib", "batch"])
        prec = "f64" if rng.random() < 0.25 else "f32"
        b = rng.choice([8, 16, 16, 32])
        case = dict(op=op, prec=prec, b=b)
        if op == "batch":
            case.update(layout="plates", nprob=int(_log(rng, 2, 48)), nb_lo=8, nb_hi=int(_log(rng, 60, 1200)),
                        layout_seed=rng.randrange(1 << 20), fields=3)
            case["b"] = b = min(b, 16)
        elif op in ("stage", "ib"):
            case.update(layout="sphere", surface=0, fields=3, **_draw_layout(rng, "sphere", b))
            if op == "stage":
                case["markers"] = min(case["markers"], 5120 if prec == "f32" else 2500)
        else:
            kind = rng.choice(["box", "wake", "scattered", "sphere"]) if op != "kinv" else "sphere"
            case.update(layout=kind, fields=3 if op in ("refresh", "kinv") else rng.choice([1, 2, 3, 3, 6]))
            case.update(_draw_layout(rng, kind, b))
            if kind == "sphere":
                case["surface"] = 2 if op == "kinv" else 1 if op == "poisson" and rng.random() < 0.6 else 0
        if op in ("intfactor", "kinv", "stage", "batch"):
            case["alpha"] = round(_log(rng, 0.02, 2.5 if op == "intfactor" else 0.6), 4)
        probs = _problems(_key(case))
        points = sum(float(np.prod(_box(p["b"], p["src"], p["tgt"])[1])) for p in probs) * case["fields"]
        blocks = max(p["src"].shape[0] + p["tgt"].shape[0] for p in probs)
        # FP64 runs at a small fraction of the FP32 rate
        if blocks <= 8000 and points * (8 if prec == "f64" else 1) <= 0.5 * MOST_POINTS:
            return case


# ----------------------------------------------------------------------------
# block sets
# ----------------------------------------------------------------------------
def _key(case):
    """What shapes the block sets of a case, as a hashable key."""
    return tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "prec", "alpha", "fields")))


def _grid(nx, ny, nz):
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    return np.stack([x.ravel(), y.ravel(), z.ravel()], axis=1).astype(np.int32)


def _support(X):
    """Face-lattice points within the three-point kernel of markers X [nm][3]
    (cell units) and their first axis indices: for component k, n0 [nm][3]."""
    for k in range(3):
        off = np.full(3, 0.5)
        off[k] = 0.0
        yield k, np.floor(X - off - 0.5).astype(np.int64)


def _touched(b, X):
    """Blocks holding a support point of the markers, sorted."""
    keys = []
    for _, n0 in _support(X):
        for j in _grid(3, 3, 3):
            c = np.floor_divide(n0 + j, b) + (1 << 20)
            keys.append(np.unique((c[:, 0] << 42) | (c[:, 1] << 21) | c[:, 2]))
    k = np.unique(np.concatenate(keys))
    return (np.stack([k >> 42, (k >> 21) & 0x1fffff, k & 0x1fffff], axis=1) - (1 << 20)).astype(np.int32)


def _sphere_markers(nm, radius):
    i = np.arange(nm) + 0.5
    z = 1.0 - 2.0 * i / nm
    phi = math.pi * (1.0 + 5 ** 0.5) * i
    r = np.sqrt(1.0 - z * z)
    return radius * np.stack([r * np.cos(phi), r * np.sin(phi), z], axis=1)


def _plate(rng, count, b, aspect):
    """A flat plate at 30 degrees with about `count` target blocks: the blocks
    it touches, and the nearest blocks downstream."""
    chord, a = 40.0, math.radians(30.0)
    while True:
        nc, ns = (max(2, int(round(v / 1.05)) + 1) for v in (chord, aspect * chord))
        s, w = np.meshgrid(np.linspace(-0.5, 0.5, nc) * chord, np.linspace(-0.5, 0.5, ns) * aspect * chord,
                           indexing="ij")
        X = np.stack([s.ravel() * math.cos(a), -s.ravel() * math.sin(a), w.ravel()], axis=1) + rng.uniform(-0.5, 0.5, 3)
        src = _touched(b, X)
        if src.shape[0] <= count or chord < 2.0:
            break
        chord *= 0.8
    lo, hi = src.min(0), src.max(0)
    need = max(0, count - src.shape[0])
    span = hi - lo + 1
    cand = _grid(span[0] + 2 + math.ceil(need / (span[1] * span[2])), span[1] + 2, span[2]) + lo - [0, 1, 0]
    have = {tuple(c) for c in src.tolist()}
    cand = np.array([c for c in cand.tolist() if tuple(c) not in have]).reshape(-1, 3)
    d = np.abs(cand - (lo + hi) / 2.0) @ np.array([1.0, 2.0, 0.5])
    tgt = np.concatenate([src, cand[np.argsort(d, kind="stable")[:need]]])
    return dict(b=b, src=src, tgt=tgt.astype(np.int32), X=X)


@lru_cache(maxsize=64)
def _problems(key):
    """The block sets of a case: dicts of b, src, tgt and the markers X (or None)."""
    c = dict(key)
    b, layout = c["b"], c["layout"]
    if layout == "box":
        s = _grid(c["nx"], c["ny"], c["nz"])
        return [dict(b=b, src=s, tgt=s, X=None)]
    if layout == "scattered":
        rng = np.random.default_rng(c["layout_seed"])
        g = _grid(c["ex"], c["ey"], c["ez"])
        pick = lambda n: g[np.sort(rng.choice(g.shape[0], n, replace=False))]   # noqa: E731
        return [dict(b=b, src=pick(c["nsrc"]), tgt=pick(c["ntgt"]) + rng.integers(-1, 2, 3).astype(np.int32), X=None)]
    if layout == "wake":
        g = _grid(c["nx"], c["ny"], c["nz"])
        x, y, z = (g + 0.5 - np.array([c["nx"] / 4.0, c["ny"] / 2.0, c["nz"] / 2.0])).T
        # blocks in the order in which a growing ball with its wake takes them
        r = np.where(x >= 0, np.sqrt(y * y + z * z), np.inf)
        r = np.minimum(r, np.sqrt(x * x + y * y + z * z) / 1.2)
        take = np.sort(np.argsort(r, kind="stable")[:max(1, int(round(c["frac"] * g.shape[0])))])
        return [dict(b=b, src=g[take], tgt=g[take], X=None)]
    if layout == "sphere":
        n = int(math.ceil(max(c["radius"], c["wake_len"]))) + 1
        g = _grid(2 * n + 1, 2 * n + 1, 2 * n + 1) - n
        x, y, z = (g + 0.5).T
        keep = (x * x + y * y + z * z <= c["radius"] ** 2) | (
            (x >= 0) & (x <= c["wake_len"]) & (y * y + z * z <= c["wake_radius"] ** 2))
        flow = g[keep].astype(np.int32)
        X = _sphere_markers(c["markers"], c["radius_cells"])
        body = _touched(b, X)
        if c["surface"] == 2:
            return [dict(b=b, src=body, tgt=body, X=X)]
        inside = {tuple(v) for v in flow.tolist()}
        body = np.array([v for v in body.tolist() if tuple(v) in inside], dtype=np.int32)
        return [dict(b=b, src=body if c["surface"] else flow, tgt=flow, X=X)]
    rng = np.random.default_rng(c["layout_seed"])
    counts = np.exp(rng.uniform(math.log(c["nb_lo"]), math.log(c["nb_hi"]), c["nprob"])).astype(int)
    return [_plate(rng, int(n), b, (1, 2, 4)[i % 3]) for i, n in enumerate(counts)]


def _box(b, *sets, margin=0):
    """Lowest lattice point and extents (x, y, z) of the box around block sets."""
    c = np.concatenate(sets)
    lo, hi = c.min(0) - margin, c.max(0) + margin
    return lo.astype(np.int64) * b, (hi - lo + 1).astype(np.int64) * b


def _points(b, coords, lo, n):
    """Flat indices of the blocks' points in the box [z][y][x] at lo of extents n."""
    r = torch.arange(b, device=DEV)
    o = torch.as_tensor(np.asarray(coords, dtype=np.int64) * b - lo, device=DEV)
    x, y, z = (o[:, d, None] + r for d in range(3))
    i = (z[:, :, None, None] * int(n[1]) + y[:, None, :, None]) * int(n[0]) + x[:, None, None, :]
    return i.reshape(-1)


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def _blobs(rng, b, coords, nfields, lo, n):
    """Sums of Gaussian vortices (widths of a few cells up to a twelfth of the
    box) at the points of the blocks: [nfields][nblocks b^3], float64."""
    nb = 16
    width = np.clip(n.min() / rng.uniform(12.0, 24.0, nb), 2.0, 10.0)
    axes = []
    for d in range(3):
        c = rng.uniform(0.0, float(n[d]), nb)
        axes.append(torch.as_tensor(np.exp(-(np.arange(n[d])[None] - c[:, None]) ** 2 / (2.0 * width[:, None] ** 2)),
                                    device=DEV))
    zy = (axes[2][:, :, None] * axes[1][:, None, :]).reshape(nb, -1)
    at = _points(b, coords, lo, n)
    out = torch.empty(nfields, at.numel(), dtype=torch.float64, device=DEV)
    for f in range(nfields):
        amp = torch.as_tensor(rng.normal(size=nb), device=DEV)
        out[f] = (zy.T @ (amp[:, None] * axes[0])).reshape(-1)[at]
    return out


def _phi(r):
    a = r.abs()
    near = (1.0 + torch.sqrt((1.0 - 3.0 * a * a).clamp_min(0.0))) / 3.0
    far = (5.0 - 3.0 * a - torch.sqrt((1.0 - 3.0 * (1.0 - a) ** 2).clamp_min(0.0))) / 6.0
    return torch.where(a <= 0.5, near, torch.where(a <= 1.5, far, torch.zeros_like(a)))


def _marker_stencil(X, lo, n):
    """For each face component the flat box indices [nm][27] and the weights."""
    for k, n0 in _support(X):
        off = np.full(3, 0.5)
        off[k] = 0.0
        p = torch.as_tensor(n0[:, None, :] + _grid(3, 3, 3)[None], device=DEV)
        w = _phi(p - torch.as_tensor(X - off, device=DEV)[:, None, :]).prod(-1)
        p = p - torch.as_tensor(lo, device=DEV)
        inside = ((p >= 0) & (p < torch.as_tensor(n, device=DEV))).all(-1)
        p = torch.where(inside[..., None], p, torch.zeros_like(p))
        yield k, (p[..., 2] * int(n[1]) + p[..., 1]) * int(n[0]) + p[..., 0], torch.where(inside, w, torch.zeros_like(w))


def _spread(p, coords, g, lo, n):
    """Marker values g [3][nm] on the box's faces, kept on the blocks: [3][points]."""
    out = torch.zeros(3, int(np.prod(n)), dtype=torch.float64, device=DEV)
    for k, at, w in _marker_stencil(p["X"], lo, n):
        out[k].index_add_(0, at.reshape(-1), (w * g[k][:, None]).reshape(-1))
    return out[:, _points(p["b"], coords, lo, n)]


def _inputs(case, seed):
    """Input tensors of each problem of a case, in the case's precision."""
    rng = np.random.default_rng([seed, 1604])
    dt = torch.float64 if case["prec"] == "f64" else torch.float32
    normal = lambda *shape: torch.as_tensor(rng.normal(size=shape), device=DEV)   # noqa: E731
    out = []
    for p in _problems(_key(case)):
        lo, n = _box(p["b"], p["src"])
        i = {}
        if case["op"] == "ib":
            i["g"] = normal(3, p["X"].shape[0])
            i["v"] = _blobs(rng, p["b"], p["tgt"], 3, lo, n)
        elif case["op"] == "stage":
            nm = p["X"].shape[0]
            gen = torch.Generator(DEV).manual_seed(int(seed) * 7919 + 17)
            # an inverse Cholesky factor: lower triangular, of order one
            W = torch.randn(3 * nm, 3 * nm, generator=gen, dtype=dt, device=DEV).mul_(0.5 / math.sqrt(3.0 * nm)).tril_()
            W.diagonal().add_(1.0)
            i.update(f=_blobs(rng, p["b"], p["src"], 3, lo, n), ub=0.1 * normal(3, nm), W=W)
        elif p["X"] is not None and case.get("surface", 1):
            # marker forces spread onto the body's blocks (three face components)
            i["f"] = _spread(p, p["src"], normal(3, p["X"].shape[0]), lo, n)[:case["fields"]]
            while i["f"].shape[0] < case["fields"]:
                i["f"] = torch.cat([i["f"], i["f"].flip(0) * float(rng.normal())])[:case["fields"]]
        else:
            i["f"] = _blobs(rng, p["b"], p["src"], case["fields"], lo, n)
        out.append({k: v.to(dt).contiguous() for k, v in i.items()})
    return out


# ----------------------------------------------------------------------------
# the measured call
# ----------------------------------------------------------------------------
_contexts = {}
_streams = []


def _context(prec):
    if prec not in _contexts:
        _contexts[prec] = lgf.Context(prec)
        _contexts[prec].table_build(48)
    return _contexts[prec]


def _stream():
    """The solver's own stream: batches replay a CUDA graph on it."""
    if not _streams:
        _streams.append(torch.cuda.Stream(DEV))
    return _streams[0]


def prepare(case, seed):
    ctx = _context(case["prec"])
    probs, ins = _problems(_key(case)), _inputs(case, seed)
    op, nf = case["op"], case["fields"]
    new = lambda n: torch.empty(n, dtype=ctx.dtype, device=DEV)   # noqa: E731
    state = dict(op=op, ctx=ctx, b=case["b"], alpha=case.get("alpha", 0.0), nf=nf)
    if op in ("batch", "step"):
        sizes = [p["tgt"].shape[0] * p["b"] ** 3 * nf for p in probs]
        if op == "batch":
            u = new(sum(sizes))
            parts = u.split(sizes)
            state["problems"] = [dict(b=p["b"], src=p["src"], tgt=p["tgt"], f=i["f"].reshape(-1), u=v, ncomp=nf,
                                      op=lgf.LGF_OP_POISSON_THEN_INTFACTOR, alpha=case["alpha"])
                                 for p, i, v in zip(probs, ins, parts)]
        else:
            p, f = probs[0], ins[0]["f"].reshape(-1)
            u = [new(sizes[0]) for _ in range(1 + len(STEP_ALPHAS))]
            common = dict(b=p["b"], src=p["src"], tgt=p["tgt"], f=f, ncomp=nf)
            state["problems"] = [dict(common, u=u[0], op=lgf.LGF_OP_POISSON)] + [
                dict(common, u=v, op=lgf.LGF_OP_INTFACTOR, alpha=a) for v, a in zip(u[1:], STEP_ALPHAS)]
        _stream().wait_stream(torch.cuda.current_stream())
        return dict(state, out=u)
    p, i = probs[0], ins[0]
    state.update(src=p["src"], tgt=p["tgt"], **i)
    if p["X"] is not None:
        state["X"] = torch.as_tensor(p["X"], device=DEV)
    state["out"] = new(p["tgt"].shape[0] * p["b"] ** 3 * nf)
    if op == "stage":
        state["d"], state["fm"] = new(p["tgt"].shape[0] * p["b"] ** 3), new(3 * p["X"].shape[0])
    if op == "ib":
        state["um"] = new(3 * p["X"].shape[0])
    return state


def run(s):
    op, ctx, b = s["op"], s["ctx"], s["b"]
    if op in ("batch", "step"):
        ctx.batch_apply(s["problems"], stream=_stream())
        return s["out"]
    if op == "poisson":
        return ctx.poisson_apply(b, s["src"], s["tgt"], s["f"], s["out"], ncomp=s["nf"])
    if op == "kinv":
        return ctx.kinv_apply(s["alpha"], b, s["src"], s["tgt"], s["f"], s["out"], ncomp=s["nf"])
    if op == "intfactor":
        return ctx.intfactor_apply(s["alpha"], b, s["src"], s["tgt"], s["f"], s["out"], ncomp=s["nf"])
    if op == "refresh":
        return ctx.velocity_refresh(b, s["src"], s["tgt"], s["f"], s["out"])
    if op == "stage":
        ctx.nested_projection_stage(b, s["tgt"], s["f"], s["out"], X_prev=s["X"], X=s["X"], ub=s["ub"], W1=s["W"],
                                    alpha=s["alpha"], d=s["d"], f=s["fm"])
        return [s["out"], s["d"], s["fm"]]
    ctx.ib_spread(b, s["tgt"], s["X"], s["g"], s["out"])
    ctx.ib_interp(b, s["tgt"], s["X"], s["v"], s["um"])
    return [s["out"], s["um"]]


def work(case):
    """Bytes: every input and output once.  Flops: a zero-padded FFT
    convolution of the smallest box (5 N log2 N each way, half for real
    fields), 2 per weight and axis of an integrating factor, 2 per entry of the
    force factor's two products."""
    esz = 8 if case["prec"] == "f64" else 4
    op, nf = case["op"], case["fields"]
    nbytes = flops = 0.0
    for p in _problems(_key(case)):
        b3 = p["b"] ** 3
        ns, nt = p["src"].shape[0] * b3, p["tgt"].shape[0] * b3
        m = 1.0
        for d in range(3):
            m *= float(np.ptp(p["src"][:, d]) + np.ptp(p["tgt"][:, d]) + 2) * p["b"] - 1.0
        conv = 5.0 * m * math.log2(m)
        heat = lambda alpha: 6.0 * nt * (2 * _radius(alpha, case["prec"]) + 1)   # noqa: E731
        nm = 0 if p["X"] is None else p["X"].shape[0]
        if op == "ib":
            nbytes += esz * (2 * nt * 3 + 6 * nm) + 48.0 * nm
            flops += 2 * 27 * 6.0 * nm
        elif op == "stage":
            nbytes += esz * (3 * ns + 4 * nt + (3 * nm) ** 2 + 6 * nm) + 48.0 * nm
            flops += 2 * conv + 6 * heat(case["alpha"]) + 4.0 * (3 * nm) ** 2
        elif op == "step":
            nbytes += esz * nf * (ns + nt * (1 + len(STEP_ALPHAS)))
            flops += nf * (conv + sum(heat(a) for a in STEP_ALPHAS))
        else:
            nbytes += esz * nf * (ns + nt)
            flops += nf * (0.0 if op == "intfactor" else conv)
            flops += nf * (heat(case["alpha"]) if op in ("intfactor", "batch") else 0.0)
            flops += 18.0 * (ns + nt) if op == "refresh" else 0.0
    return {"bytes": nbytes, "flops": flops}


# ----------------------------------------------------------------------------
# the same results in 64 bits
# ----------------------------------------------------------------------------
def _bessel(n, z):
    """e^{-z} I_k(z) for k = 0..n: the cosine coefficients of e^{z (cos t - 1)}
    (spectrally exact trapezoidal rule), or Hankel's expansion for large z."""
    if z > max(2048.0, 6.0 * n * n):
        k = np.arange(n + 1, dtype=np.float64)
        term, total = np.ones(n + 1), np.ones(n + 1)
        for j in range(1, 40):
            term = -term * (4.0 * k * k - (2 * j - 1) ** 2) / (8.0 * j * z)
            total += term
        return total / math.sqrt(2.0 * math.pi * z)
    m = 2 * (n + int(12.0 * math.sqrt(z)) + 64)
    t = 2.0 * math.pi * np.arange(m) / m
    return np.fft.rfft(np.exp(z * (np.cos(t) - 1.0))).real[:n + 1] / m


@lru_cache(maxsize=None)
def _radius(alpha, prec):
    w = _bessel(200, 2.0 * alpha)
    return int(np.argmax(w < (1e-7 if prec == "f32" else 1e-13) / 8.0 * w[0]))


def _green(n, alpha):
    """-int_alpha^inf prod_i e^{-2t} I_{n_i}(2t) dt at offsets 0..n_i per axis,
    [nz+1][ny+1][nx+1]: Gauss-Legendre on octaves of t, then t = T / v^2."""
    big = int(max(n))
    x, w = np.polynomial.legendre.leggauss(20)
    x, w = 0.5 * (x + 1.0), 0.5 * w
    edges = [alpha]
    for e in 0.5 * 2.0 ** np.arange(0, 64):
        if e > alpha:
            edges.append(e)
        if e >= max(1024.0, 3.0 * big * big):
            break
    t = np.concatenate([a + (c - a) * x for a, c in zip(edges, edges[1:])] + [edges[-1] / x ** 2])
    wt = np.concatenate([(c - a) * w for a, c in zip(edges, edges[1:])] + [2.0 * edges[-1] * w / x ** 3])
    B = torch.as_tensor(np.stack([_bessel(big, 2.0 * v) for v in t]), device=DEV)
    wt = torch.as_tensor(wt, device=DEV)
    Bx, By, Bz = (B[:, :int(n[d]) + 1] for d in range(3))
    out = torch.empty(int(n[2]) + 1, int(n[1]) + 1, int(n[0]) + 1, dtype=torch.float64, device=DEV)
    for z in range(out.shape[0]):
        out[z] = -((wt * Bz[:, z])[:, None] * By).T @ Bx
    return out


def _convolver(n, alpha=0.0):
    """Function of one dense field [z][y][x]: its convolution with G_K(alpha)."""
    g = _green(n, alpha)
    for d in range(3):   # even extension to 2 n per axis
        g = torch.cat([g, g.flip(d).narrow(d, 1, g.shape[d] - 2)], d)
    shape = tuple(g.shape)
    spec = torch.fft.rfftn(g)
    del g

    def apply(f):
        h = torch.fft.irfftn(torch.fft.rfftn(f, s=shape) * spec, s=shape)
        return h[:f.shape[0], :f.shape[1], :f.shape[2]]
    return apply


def _heat(f, alpha):
    """E(alpha) of dense fields [..][z][y][x], zero outside the box."""
    for d, size in zip((-3, -2, -1), f.shape[-3:]):
        w = torch.as_tensor(_bessel(size, 2.0 * alpha), device=DEV)
        i = torch.arange(size, device=DEV)
        f = torch.movedim(torch.movedim(f, d, -1) @ w[(i[:, None] - i[None]).abs()], -1, d)
    return f


def _dense(v, at, n):
    out = torch.zeros(v.shape[0], int(np.prod(n)), dtype=torch.float64, device=DEV)
    out[:, at] = v.reshape(v.shape[0], -1).double()
    return out.reshape(v.shape[0], int(n[2]), int(n[1]), int(n[0]))


def _diff(f, k, sign):
    """f(n + e_k) - f(n) (sign 1) or f(n) - f(n - e_k) (sign -1)."""
    return sign * (torch.roll(f, -sign, 2 - k) - f)


def _curl(f, sign):
    """C (sign -1) or its adjoint (sign 1) of dense fields [3][z][y][x]."""
    out = []
    for k in range(3):
        i, j = (k + 1) % 3, (k + 2) % 3
        out.append(_diff(f[j], i, sign) - _diff(f[i], j, sign))
    return torch.stack(out)


def _exact_stage(case, p, i, at, lo, n, mask):
    r = _dense(i["f"], at, n)
    solve = _convolver(n)
    div = lambda a: mask * sum(_diff(a[k], k, 1) for k in range(3))   # noqa: E731
    grad = lambda d: torch.stack([_diff(d, k, -1) for k in range(3)])   # noqa: E731
    w = _heat(mask * (r - grad(solve(div(r)))), case["alpha"]) * mask
    U = torch.stack([(wt * w[k].reshape(-1)[ix]).sum(1) for k, ix, wt in _marker_stencil(p["X"], lo, n)])
    W, y = i["W"], (U - i["ub"].double()).reshape(-1)
    rows = [W[a:a + 1024].double() @ y for a in range(0, W.shape[0], 1024)]
    f = sum(W[a:a + 1024].double().T @ v for a, v in zip(range(0, W.shape[0], 1024), rows))
    g = _dense(_spread(p, p["tgt"], f.reshape(3, -1), lo, n), at, n)
    d = solve(div(r - g))
    u = _heat(mask * (r - grad(d) - g), case["alpha"]).reshape(3, -1)[:, at]
    return [u.reshape(-1), d.reshape(-1)[at], f]


def exact(case, seed):
    op, results = case["op"], []
    for p, i in zip(_problems(_key(case)), _inputs(case, seed)):
        # one block of margin: the staggered operators look one point further
        lo, n = _box(p["b"], p["src"], p["tgt"], margin=1 if op in ("refresh", "stage", "ib") else 0)
        at_s, at = _points(p["b"], p["src"], lo, n), _points(p["b"], p["tgt"], lo, n)
        mask = _dense(torch.ones(1, at.numel(), device=DEV), at, n)[0]
        take = lambda f: f.reshape(-1)[at]   # noqa: E731
        if op == "ib":
            f = _spread(p, p["tgt"], i["g"].double(), lo, n).reshape(-1)
            v = _dense(i["v"], at, n).reshape(3, -1)
            return [f, torch.cat([(w * v[k][ix]).sum(1) for k, ix, w in _marker_stencil(p["X"], lo, n)])]
        if op == "stage":
            return _exact_stage(case, p, i, at, lo, n, mask)
        f = _dense(i["f"], at_s, n)
        if op == "refresh":
            src = _dense(torch.ones(1, at_s.numel(), device=DEV), at_s, n)[0]
            solve = _convolver(n)
            u = -_curl(torch.stack([solve(w) for w in _curl(f, -1) * src]), 1)
            return u.reshape(3, -1)[:, at].reshape(-1)
        if op == "intfactor":
            return torch.cat([take(_heat(c, case["alpha"])) for c in f])
        solve = _convolver(n, case["alpha"] if op == "kinv" else 0.0)
        if op == "batch":
            results.append(torch.cat([take(_heat(mask * solve(c), case["alpha"])) for c in f]))
            continue
        u = torch.cat([take(solve(c)) for c in f])
        if op == "step":
            return [u] + [torch.cat([take(_heat(c, a)) for c in f]) for a in STEP_ALPHAS]
        return u
    return torch.cat(results)
