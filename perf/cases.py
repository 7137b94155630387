"""Performance cases of the library: what its users call, at the sizes they call it.

``listed()`` names the cases that are timed, ``draw(rng)`` gives further ones
of the same ranges, ``prepare`` makes a case's inputs and the context a
program keeps, ``run`` is one pass through the public entry points, ``work``
is the traffic and arithmetic no implementation can avoid, and ``exact`` is a
plain 64-bit evaluation of the definition (brute force, no library code) for
the cases small enough for one.

All inputs are samples of analytic fields (spheres, boxes, tori and their
combinations) drawn from the seed, as in ``paper_2605_01919_gb300.workloads``.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2605_01919_gb300 import gfs
from paper_2605_01919_gb300 import workloads as W

DEV = "cuda"


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def listed():
    return [
        # a first look at a shape: a coarse grid and its 2x upsampling, all in
        # FP64; a few milliseconds, so launches and host round trips count
        {"name": "small_solve", "kind": "solve", "shape": "sphere", "N": 16, "tau": 2, "up": 2, "fp32": False,
         "box": True, "clamp": True},
        # a handful of probe points on a field that is already built (picking,
        # ray steps): the smallest call, all latency
        {"name": "few_points", "kind": "points", "shape": "union", "N": 32, "tau": 3, "m": 257, "fp32": True,
         "box": True, "clamp": True},
        # upsampling a 64^3 grid 4x for meshing: the largest ordinary job
        {"name": "grid_upsample", "kind": "solve", "shape": "union", "N": 64, "tau": 3, "up": 4, "fp32": False,
         "box": True, "clamp": True},
        # candidates of a noisy pseudo-SDF (CSG min/max values) and which of
        # them survive: the P build alone, with overlapping balls of both signs
        {"name": "pseudo_build", "kind": "build", "shape": "csg", "N": 49, "tau": 3, "box": True, "clamp": True},
        # one step of fitting samples to values at random points: build,
        # forward and backward to points, positions and values
        {"name": "fit_step", "kind": "fit", "shape": "torus", "N": 96, "tau": 3, "m": 1 << 21, "fp32": True,
         "box": True, "clamp": True},
        # scattered scan samples in host memory, results back in host memory
        {"name": "scatter_host", "kind": "host", "shape": "scatter", "n": 50021, "tau": 3, "m": 400168,
         "fp32": False, "box": True, "clamp": True},
        # many shapes of uneven size, half grids and half scattered, rebuilt
        # and queried in one go
        {"name": "batch", "kind": "batch", "shape": "mixed", "shapes": 16, "lo": 12, "hi": 48, "sizes": 7, "tau": 3,
         "box": True, "clamp": True},
        # greedy refinement at the centres of the surface cells, in flood-fill
        # order from the least covered cell
        {"name": "refine", "kind": "refine", "shape": "union", "N": 40, "tau": 3, "T": 1536, "box": True,
         "clamp": True},
        # repair of a noisy pseudo-SDF: find the covered samples, drop them,
        # insert them again with their own values known
        {"name": "repair", "kind": "repair", "shape": "csg", "N": 32, "tau": 3, "T": 1024, "box": True,
         "clamp": True},
        # values refined by the tangent points of the spheres of the same sign
        {"name": "tangent", "kind": "tangent", "shape": "union", "N": 64, "tau": 3, "m": 31607, "fp32": False,
         "box": True, "clamp": True},
        # the scored value, positive and negative radii ranked
        {"name": "scored", "kind": "scored", "shape": "union", "N": 48, "tau": 3, "m": 8191, "fp32": False,
         "box": True, "clamp": True},
        # exact minimum radius from the uncovered circles and points of a
        # small sample set
        {"name": "exact_radius", "kind": "radius", "shape": "union", "N": 12, "tau": 3, "m": 512, "box": True,
         "clamp": True},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "points", "build", "fit", "host", "batch", "refine", "repair", "tangent",
                       "scored", "radius"])
    shape = rng.choice(["sphere", "union", "torus", "csg", "scatter"])
    c = {"kind": kind, "shape": shape, "tau": rng.choice([2, 3, 3]), "box": rng.random() < 0.85,
         "clamp": rng.random() < 0.85}
    if kind == "solve":
        c.update(N=_logint(rng, 9, 64), up=rng.choice([2, 3, 4]), fp32=rng.random() < 0.5)
    elif kind == "points":
        c.update(N=_logint(rng, 12, 64), m=_logint(rng, 1, 20000), fp32=rng.random() < 0.5)
    elif kind == "build":
        c.update(N=_logint(rng, 9, 64))
    elif kind == "fit":
        c.update(N=_logint(rng, 12, 64), m=_logint(rng, 1000, 1 << 20), fp32=rng.random() < 0.7)
    elif kind == "host":
        n = _logint(rng, 1500, 60000)
        c.update(shape="scatter", n=n, m=rng.randint(1, 8 * n), fp32=rng.random() < 0.5)
    elif kind == "batch":
        c.update(shape="mixed", shapes=rng.randint(2, 16), lo=8, hi=rng.randint(12, 48), sizes=rng.randint(0, 9999))
    elif kind == "refine":
        c.update(shape=rng.choice(["sphere", "union", "torus"]), N=_logint(rng, 10, 40), T=1)
        c["T"] = _logint(rng, 50, min(1536, c["N"] ** 2))
    elif kind == "repair":
        c.update(shape="csg", N=_logint(rng, 12, 32), T=1)
        c["T"] = _logint(rng, 50, min(1024, c["N"] ** 3 // 8))
    elif kind == "tangent":
        c.update(N=_logint(rng, 10, 64), m=_logint(rng, 200, 31607), fp32=rng.random() < 0.3)
    elif kind == "scored":
        c.update(N=_logint(rng, 10, 48), m=_logint(rng, 100, 8191), fp32=rng.random() < 0.3)
    else:
        c.update(shape=rng.choice(["sphere", "union", "scatter"]), N=rng.randint(6, 12), m=_logint(rng, 30, 512))
    return c


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _ksum(case):
    return 10 * 4 ** case["tau"] + 2


def _nsamples(case):
    return case["n"] if "n" in case else case["N"] ** 3


def _field(shape, seed, N):
    rng = np.random.default_rng(seed)
    if shape == "sphere":
        c, r = rng.uniform(-0.1, 0.1, 3), rng.uniform(0.5, 0.65)
        return lambda P: W.sdf_sphere(P, c, r)
    if shape == "torus":
        c = rng.uniform(-0.05, 0.05, 3)
        return lambda P: W.sdf_torus(P, c, 0.5, 0.2, 2)
    if shape == "union":
        return W.union_field(seed)
    return W.union_of_primitives(rng, int(rng.integers(1, 9)))


def _samples(case, seed):
    """Positions (n, 3) and values (n,) of the case's samples, and its field (None for the pseudo-SDF)."""
    if case["shape"] == "csg":
        w = W.csg_pseudo_grid(N=case["N"], tau=case["tau"], seed=seed)
        return w.p, w.s, None
    f = _field(case["shape"], seed, case.get("N", 0))
    if case["shape"] == "scatter":
        p = np.random.default_rng([seed, 1]).uniform(-1.0, 1.0, (_nsamples(case), 3))
    else:
        p = W.grid_points(case["N"])
    return p, f(p), f


def _random_points(case, seed):
    x = np.random.default_rng([seed, 2]).uniform(-1.0, 1.0, (case["m"], 3))
    return x.astype(np.float32) if case.get("fp32") else x


def _grid_queries(case):
    """The up-times upsampled node grid, made on the device."""
    nq = case["up"] * (case["N"] - 1) + 1
    g = torch.linspace(-1.0, 1.0, nq, dtype=torch.float64, device=DEV)
    x = torch.stack(torch.meshgrid(g, g, g, indexing="ij"), dim=-1).reshape(-1, 3)
    return x.float().contiguous() if case["fp32"] else x.contiguous()


def _surface_cells(case, p, s, seed):
    """The T cells whose corners come nearest to the surface: integer coordinates in a random order, and the grid's
    origin and spacing."""
    N = case["N"]
    h = W.grid_spacing(N)
    v = np.abs(s.reshape(N, N, N))
    near = v[:-1, :-1, :-1]
    for a in (0, 1):
        for b in (0, 1):
            for c in (0, 1):
                near = np.minimum(near, v[a:N - 1 + a, b:N - 1 + b, c:N - 1 + c])
    cells = np.stack(np.unravel_index(np.argsort(near, axis=None, kind="stable")[:case["T"]], near.shape), axis=1)
    cells = cells[np.random.default_rng([seed, 3]).permutation(cells.shape[0])].astype(np.int32)
    return np.ascontiguousarray(cells), np.full(3, -1.0), h


def _batch_sizes(case):
    rng = np.random.default_rng(case["sizes"])
    sides = rng.integers(case["lo"], case["hi"] + 1, case["shapes"])
    return [int(v) for v in sides]


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def prepare(case, seed):
    seed = int(seed)
    kind = case["kind"]
    st = {"kind": kind, "case": dict(case), "seed": seed}
    ctx = gfs.Context(tau=case["tau"], box_cull=case["box"], clamp_opp=case["clamp"], tangent=kind == "tangent")
    st["ctx"] = ctx
    if kind == "batch":
        shapes = []
        for k, side in enumerate(_batch_sizes(case)):
            f = _field("scatter", seed * 1000 + k, 0)
            rng = np.random.default_rng([seed, 4, k])
            if k % 2 == 0:
                p, x = W.grid_points(side), W.grid_points(2 * side - 1)
            else:
                n = max(64, side ** 3 // 4)
                p, x = rng.uniform(-1.0, 1.0, (n, 3)), rng.uniform(-1.0, 1.0, (8 * n, 3))
            shapes.append({"p": _cuda(p), "s": _cuda(f(p)), "x": _cuda(x)})
        st["shapes"] = ctx.batch_build(shapes)
        return st
    p, s, _ = _samples(case, seed)
    if kind == "host":
        x = _random_points(case, seed)
        pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory()
        m = case["m"]
        st.update(p=pin(p), s=pin(s), x=pin(x), s_out=torch.empty(m, dtype=torch.float32).pin_memory(),
                  arg_out=torch.empty(m, dtype=torch.int64).pin_memory(),
                  fl_out=torch.empty(m, dtype=torch.int16).pin_memory())
        return st
    st.update(p=_cuda(p), s=_cuda(s))
    if kind == "solve":
        st["x"] = _grid_queries(case)
    elif kind in ("points", "fit", "tangent", "scored", "radius"):
        st["x"] = _cuda(_random_points(case, seed))
    if kind == "fit":
        st["g"] = _cuda(np.random.default_rng([seed, 5]).normal(0.0, 1.0, case["m"]).astype(np.float32))
        for k in ("p", "s", "x"):
            st[k].requires_grad_(True)
    if kind == "radius":
        st["sigma"] = _cuda(np.where(np.random.default_rng([seed, 6]).random(case["m"]) < 0.5, 1, -1).astype(np.int8))
    if kind == "refine":
        cells, origin, h = _surface_cells(case, p, s, seed)
        st.update(cells_host=cells, cells=_cuda(cells), origin=origin, h=h,
                  centres=_cuda(origin + h * (cells.astype(np.float64) + 0.5)))
    if kind == "repair":
        st["order"] = _cuda(np.random.default_rng([seed, 7]).permutation(p.shape[0]))
    if kind in ("points", "tangent", "scored"):
        # these programs build once and ask many times
        ctx.build(st["p"], st["s"])
    return st


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def _kept(ctx, spheres):
    """The surviving candidates as one byte per (sphere, direction or witness)."""
    keep = torch.zeros(spheres * (ctx.K + 1), dtype=torch.uint8, device=DEV)
    keep[ctx.survivors()] = 1
    return keep


def run(st):
    kind, ctx = st["kind"], st["ctx"]
    if kind == "solve":
        ctx.build(st["p"], st["s"])
        return ctx.query(st["x"])
    if kind == "points" or kind == "tangent":
        return ctx.query(st["x"])
    if kind == "scored":
        return ctx.query_scored(st["x"])
    if kind == "build":
        ctx.build(st["p"], st["s"])
        return _kept(ctx, st["p"].shape[0])
    if kind == "fit":
        x, p, s = st["x"], st["p"], st["s"]
        ctx.build(p.detach(), s.detach())
        v = gfs.ConsistentSDF.apply(x, p, s, ctx)
        gx, gp, gs = torch.autograd.grad(v, (x, p, s), st["g"])
        return {"v": v.detach(), "gx": gx, "gp": gp, "gs": gs}
    if kind == "host":
        ctx.solve_host(st["p"], st["s"], st["x"], st["s_out"], st["arg_out"], st["fl_out"])
        return {"s": st["s_out"], "argmin": st["arg_out"], "flags": st["fl_out"]}
    if kind == "batch":
        ctx.batch_rebuild()
        outs = ctx.batch_query()
        return [{k: o[k] for k in ("s64", "argmin", "flags")} for o in outs]
    if kind == "refine":
        ctx.build(st["p"], st["s"])
        counts = ctx.cell_coverage(st["cells"], st["origin"], st["h"])
        order = gfs.flood_order(st["cells_host"], counts.cpu().numpy())
        out = ctx.insert(st["centres"][torch.from_numpy(order).to(DEV)])
        return {"counts": counts, "order": order, "kept": _kept(ctx, st["p"].shape[0] + order.shape[0]), **out}
    if kind == "repair":
        p, s = st["p"], st["s"]
        ctx.build(p, s)
        state = ctx.sphere_uncovered()
        gone = state == 0
        ctx.build(p[~gone], s[~gone])
        # the dropped samples in a random order (then kept ones, should there be too few)
        back = st["order"][torch.sort(state[st["order"]], stable=True).indices[:st["case"]["T"]]]
        out = ctx.insert(p[back], known=s[back])
        return {"state": state, "kept": _kept(ctx, p.shape[0] + back.shape[0]), **out}
    ctx.build(st["p"], st["s"])
    return {"rmin": ctx.exact_rmin(st["x"], st["sigma"])}


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
# A candidate is made (3 multiply-adds) and meets at least one ball (8
# flops); a query point is measured against at least the survivor, the
# opposite ball, the containing ball and the far ball that decide its result
# (4 x 8 flops).  Samples come in as 32 B, points as 24 or 12 B; results are
# the FP32 and FP64 value, argmin and result word (22 B).
def work(case):
    kind = case["kind"]
    if kind == "batch":
        b = f = 0
        for k, side in enumerate(_batch_sizes(case)):
            n = side ** 3 if k % 2 == 0 else max(64, side ** 3 // 4)
            m = (2 * side - 1) ** 3 if k % 2 == 0 else 8 * n
            b += 32 * n + (24 + 18) * m
            f += 14 * _ksum(case) * n + 32 * m
        return {"bytes": b, "flops": f}
    n = _nsamples(case)
    cand = 14 * _ksum(case)
    if kind == "solve":
        m = (case["up"] * (case["N"] - 1) + 1) ** 3
        return {"bytes": 32 * n + ((12 if case["fp32"] else 24) + 22) * m, "flops": cand * n + 32 * m}
    if kind == "build":
        return {"bytes": (32 + _ksum(case) + 1) * n, "flops": cand * n}
    if kind == "fit":
        m, xb = case["m"], 12 if case["fp32"] else 24
        return {"bytes": 2 * 32 * n + (2 * xb + 8) * m, "flops": cand * n + 64 * m}
    if kind == "host":
        return {"bytes": 32 * n + ((12 if case["fp32"] else 24) + 14) * case["m"],
                "flops": cand * n + 32 * case["m"]}
    if kind in ("refine", "repair"):
        T = case["T"]
        return {"bytes": 32 * n + (24 + 18) * T + (_ksum(case) + 1) * (n + T), "flops": cand * (n + T) + 32 * T}
    if kind == "radius":
        return {"bytes": 32 * n + 33 * case["m"], "flops": cand * n + 32 * case["m"]}
    # points, tangent, scored: the state is built, a point needs its own deciding samples
    return {"bytes": ((12 if case.get("fp32") else 24) + 22 + 4 * 32) * case["m"], "flops": 32 * case["m"]}


# --------------------------------------------------------------------------
# the definition in 64 bits, by brute force
# --------------------------------------------------------------------------
TOL = 1e-6
_CHUNK = 1 << 24


def _directions(tau):
    phi = (1.0 + math.sqrt(5.0)) / 2.0
    v = []
    for a in (-1.0, 1.0):
        for b in (-phi, phi):
            v += [(a, b, 0.0), (0.0, a, b), (b, 0.0, a)]
    v = np.array(v) / math.sqrt(1.0 + phi * phi)
    d = np.linalg.norm(v[:, None] - v[None], axis=-1)
    adj = np.abs(d - d[d > 1e-9].min()) < 1e-6
    faces = [(i, j, k) for i in range(12) for j in range(i) for k in range(j) if adj[i, j] and adj[j, k] and adj[i, k]]
    pts = [tuple(r) for r in v]
    for _ in range(tau):
        mid, nxt = {}, []
        for f in faces:
            e = []
            for i, j in ((f[0], f[1]), (f[1], f[2]), (f[2], f[0])):
                key = (min(i, j), max(i, j))
                if key not in mid:
                    m = np.array(pts[i]) + np.array(pts[j])
                    pts.append(tuple(m / np.linalg.norm(m)))
                    mid[key] = len(pts) - 1
                e.append(mid[key])
            nxt += [(f[0], e[0], e[2]), (f[1], e[1], e[0]), (f[2], e[2], e[1]), (e[0], e[1], e[2])]
        faces = nxt
    return torch.tensor(np.array(pts), dtype=torch.float64, device=DEV)


def _dist2(a, b):
    d = a[:, 0, None] - b[None, :, 0]
    r = d * d
    d = a[:, 1, None] - b[None, :, 1]
    r += d * d
    d = a[:, 2, None] - b[None, :, 2]
    r += d * d
    return r


def _uncovered(q, own, p, rt):
    """Which rows of q lie in no ball (p, rt) but their own, rt the shrunk radius (-1: never covers)."""
    idx = torch.arange(q.shape[0], device=DEV)
    n = p.shape[0]
    order = torch.randperm(n, generator=torch.Generator().manual_seed(1)).to(DEV)
    r2 = torch.where(rt > 0, rt * rt, torch.full_like(rt, -1.0))
    b = 0
    step = 64
    while b < n and idx.numel():
        sel = order[b:b + step]
        keep = []
        rows = max(1, _CHUNK // sel.numel())
        for part in idx.split(rows):
            hit = _dist2(q[part], p[sel]) < r2[sel][None]
            hit &= own[part][:, None] != sel[None]
            keep.append(part[~hit.any(1)])
        idx = torch.cat(keep)
        b += sel.numel()
        step = min(4 * step, 16384)
    return idx


def _survivors(p, s, U, box):
    """Surviving candidates: their sphere and their direction."""
    n, K = p.shape[0], U.shape[0]
    r = s.abs()
    rt = torch.where(r > TOL, r - TOL, torch.full_like(r, -1.0))
    sph, dire = [], []
    rows = max(1, (1 << 23) // K)
    for a in range(0, n, rows):
        e = min(n, a + rows)
        q = (p[a:e, None, :] + r[a:e, None, None] * U[None]).reshape(-1, 3)
        own = torch.arange(a, e, device=DEV).repeat_interleave(K)
        k = torch.arange(K, device=DEV).repeat(e - a)
        if box:
            ok = (q.abs() <= 1.0).all(1)
            q, own, k = q[ok], own[ok], k[ok]
        live = _uncovered(q, own, p, rt)
        sph.append(own[live])
        dire.append(k[live])
    return torch.cat(sph), torch.cat(dire)


def _nearest(x, q):
    """Distance to and index of the nearest row of q."""
    best = torch.full((x.shape[0],), math.inf, dtype=torch.float64, device=DEV)
    arg = torch.full((x.shape[0],), -1, dtype=torch.int64, device=DEV)
    if q.shape[0] == 0:
        return best, arg
    rows = max(1, min(x.shape[0], 4096))
    cols = max(1, _CHUNK // rows)
    for a in range(0, x.shape[0], rows):
        for b in range(0, q.shape[0], cols):
            d, j = _dist2(x[a:a + rows], q[b:b + cols]).min(1)
            d = d.sqrt()
            low = d < best[a:a + rows]
            best[a:a + rows] = torch.where(low, d, best[a:a + rows])
            arg[a:a + rows] = torch.where(low, j + b, arg[a:a + rows])
    return best, arg


def _spheres(x, p, s):
    """Per point: containment by sign, nearest tangent distance |x - p| - r of each sign and its sphere, and the
    sphere the point coincides with (-1: none)."""
    m, r = x.shape[0], s.abs()
    cov = torch.zeros((2, m), dtype=torch.bool, device=DEV)
    near = torch.full((2, m), math.inf, dtype=torch.float64, device=DEV)
    arg = torch.full((2, m), -1, dtype=torch.int64, device=DEV)
    same = torch.full((m,), -1, dtype=torch.int64, device=DEV)
    rows = max(1, min(m, 4096))
    cols = max(1, _CHUNK // rows)
    for a in range(0, m, rows):
        for b in range(0, p.shape[0], cols):
            d = _dist2(x[a:a + rows], p[b:b + cols]).sqrt()
            hit, j = (d == 0).max(1)
            same[a:a + rows] = torch.where(hit & (same[a:a + rows] < 0), j + b, same[a:a + rows])
            t = d - r[None, b:b + cols]
            for c in (0, 1):
                mine = (s[b:b + cols] > 0) if c == 0 else (s[b:b + cols] < 0)
                tc = torch.where(mine[None], t, torch.full_like(t, math.inf))
                v, j = tc.min(1)
                cov[c, a:a + rows] |= v < -TOL
                low = v < near[c, a:a + rows]
                near[c, a:a + rows] = torch.where(low, v, near[c, a:a + rows])
                arg[c, a:a + rows] = torch.where(low, j + b, arg[c, a:a + rows])
    return cov, near, arg, same


def _values(x, p, s, surv, U, clamp):
    """FP64 value at each point, its sign, and the sphere, direction (-1: none) and code (0 survivor, 1 opposite
    tangent, 2 sample, 3 outside, 4 invalid, 5 containing tangent) that set it."""
    cov, near, arg, same = _spheres(x, p, s)
    sph, dire = surv
    q = p[sph] + s[sph].abs()[:, None] * U[dire]
    m = x.shape[0]
    value = torch.zeros(m, dtype=torch.float64, device=DEV)
    code = torch.full((m,), 3, dtype=torch.int64, device=DEV)
    who = torch.full((m,), -1, dtype=torch.int64, device=DEV)
    kdir = torch.full((m,), -1, dtype=torch.int64, device=DEV)
    for c in (0, 1):
        ask = torch.nonzero(cov[c] & ~cov[1 - c] & (same < 0)).flatten()
        if not ask.numel():
            continue
        mine = torch.nonzero((s[sph] >= 0) if c == 0 else (s[sph] <= 0)).flatten()
        ds, j = _nearest(x[ask], q[mine])
        ub = near[1 - c, ask]
        have = j >= 0
        use_s = have & ((ds <= ub) if clamp else torch.ones_like(have))
        use_u = ~use_s & (ub < math.inf) & bool(clamp)
        v = torch.where(use_s, ds, torch.where(use_u, ub, -near[c, ask])).clamp_min(0.0)
        value[ask] = v if c == 0 else -v
        code[ask] = torch.where(use_s, 0, torch.where(use_u, 1, 5))
        g = mine[j.clamp_min(0)] if mine.numel() else torch.zeros_like(j)
        si = sph[g] if sph.numel() else torch.zeros_like(j)
        who[ask] = torch.where(use_s, si, torch.where(use_u, arg[1 - c, ask], arg[c, ask]))
        if dire.numel():
            kdir[ask] = torch.where(use_s, dire[g], -1)
    bad = cov[0] & cov[1] & (same < 0)
    value[bad] = math.nan
    code[bad] = 4
    at = same >= 0
    value[at] = s[same[at]]
    code[at] = 2
    who[at] = same[at]
    return value, code, who, kdir


def _case_values(case, seed):
    p, s, _ = _samples(case, seed)
    p, s = _cuda(p), _cuda(s)
    x = _grid_queries(case) if case["kind"] == "solve" else _cuda(_random_points(case, seed))
    x = x.double()
    U = _directions(case["tau"])
    surv = _survivors(p, s, U, case["box"])
    return p, s, x, U, _values(x, p, s, surv, U, case["clamp"])


def exact(case, seed):
    kind, seed = case["kind"], int(seed)
    if kind not in ("solve", "points", "host", "fit"):
        # ids and states are whole numbers; the insertion, tangent, scored and
        # exact-radius values need every candidate point against every ball at
        # each step or query point
        return None
    n = _nsamples(case)
    m = (case["up"] * (case["N"] - 1) + 1) ** 3 if kind == "solve" else case["m"]
    # about 1% of the candidates survive; each point meets each survivor and ball
    if n > 60000 or m * n * (1.0 + 0.01 * _ksum(case)) > 2.5e11:
        return None
    p, s, x, U, (value, code, who, kdir) = _case_values(case, seed)
    if kind in ("solve", "points"):
        return {"s": value, "s64": value, "argmin": None, "flags": None}
    if kind == "host":
        return {"s": value.cpu(), "argmin": None, "flags": None}
    g = _cuda(np.random.default_rng([seed, 5]).normal(0.0, 1.0, case["m"]).astype(np.float32)).double()
    gx = torch.zeros_like(x)
    gp = torch.zeros_like(p)
    gs = torch.zeros_like(s)
    sig = torch.sign(value)
    i = torch.nonzero(code == 2).flatten()
    gs.index_add_(0, who[i], g[i])
    i = torch.nonzero((code == 0) & (sig != 0)).flatten()
    u = U[kdir[i]]
    v = x[i] - (p[who[i]] + s[who[i]].abs()[:, None] * u)
    v = v / v.norm(dim=1, keepdim=True)
    d = (g[i] * sig[i])[:, None] * v
    gx[i] = d
    gp.index_add_(0, who[i], -d)
    gs.index_add_(0, who[i], -(d * u).sum(1) * torch.sign(s[who[i]]))
    for c, way in ((1, 1.0), (5, -1.0)):
        i = torch.nonzero((code == c) & (sig != 0)).flatten()
        v = x[i] - p[who[i]]
        v = v / v.norm(dim=1, keepdim=True)
        d = way * (g[i] * sig[i])[:, None] * v
        gx[i] = d
        gp.index_add_(0, who[i], -d)
        gs.index_add_(0, who[i], -way * g[i] * sig[i] * torch.sign(s[who[i]]))
    return {"v": value, "gx": gx, "gp": gp, "gs": gs}
