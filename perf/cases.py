"""The calls that a user of this package spends time in, as cases to be measured.

Families of cases (every one through the public entry points of the package):
  voxelize   Context.voxelize: level 0 of a fiber yarn, a woven yarn, or a heightfield mesh
  lod        Context.build_lod on a level 0 that is in hand
  pyramid    voxelize + build_lod, the whole call
  adjoint    Context.backward: gradients of a loss on the masses and moments of some levels
  batch      Batch.run + Batch.level: several instances in one captured graph

Sizes follow the package's own workloads (synth/): the 768k-capsule yarn at 512^3, the woven
patch's yarns (4-voxel radius), heightfields from 64 x 64 vertices at 128^3 to 1024 x 1024 at
1024^3, the yarn at 256^3 for the adjoint, batches of uneven instances.
"""
import math

import torch

import paper_2604_13191_gb300 as vx

FIELDS = ("keys", "mask", "mass", "moment", "occ", "occ_proj", "lobe_count", "lobes", "compact")


class Grid:
    """Cubic grid: voxel (i, j, k) covers origin + voxel_size * [i, i+1] x [j, j+1] x [k, k+1]."""

    def __init__(self, origin, resolution):
        self.origin, self.voxel_size, self.resolution, self.sub_res = origin, 1.0 / resolution, resolution, 8


def listed():
    return [
        # the smallest call: a few strands in a preview grid; launches and host work
        dict(name="voxelize-strands", kind="voxelize", geom="yarn", fibers=4, segs=120, R=64, radius=0.004, weights=True),
        # a mid-size yarn with per-primitive weights, odd sizes
        dict(name="voxelize-yarn-odd", kind="voxelize", geom="yarn", fibers=21, segs=777, R=256, radius=0.004, weights=True),
        # the headline yarn: 3 plies x 64 fibers x 4,000 segments at 512^3
        dict(name="voxelize-yarn", kind="voxelize", geom="yarn", fibers=64, segs=4000, R=512, radius=0.004, weights=False),
        # one yarn of the woven patch at its voxel scale: capsules of 4 voxels' radius
        dict(name="voxelize-woven", kind="voxelize", geom="woven", fibers=80, segs=700, R=1024, radius=0.004, weights=False),
        # the small brushed-metal mesh: 7,938 triangles at 128^3
        dict(name="voxelize-mesh-small", kind="voxelize", geom="mesh", n=64, R=128, weights=False),
        # a large mesh: 2.09 M triangles at 1024^3
        dict(name="voxelize-mesh", kind="voxelize", geom="mesh", n=1024, R=1024, weights=False),
        # all levels of the headline yarn with SGGX-H, 4 lobes, 5,000 directions
        dict(name="lod-yarn-K4", kind="lod", geom="yarn", fibers=64, segs=4000, R=512, radius=0.004, K=4, N=5000, merge="pooled"),
        # plain moment aggregation of a mesh (one lobe per voxel)
        dict(name="lod-mesh-K1", kind="lod", geom="mesh", n=701, R=512, K=1, N=0, merge="pooled"),
        # the whole call on a small asset: a user's interactive preview
        dict(name="pyramid-small", kind="pyramid", geom="yarn", fibers=9, segs=301, R=64, radius=0.006, K=4, N=1024, merge="mass"),
        # gradients of the yarn at 256^3 with 4 coarser levels
        dict(name="adjoint-yarn", kind="adjoint", geom="yarn", fibers=64, segs=4000, R=256, radius=0.004, levels=4),
        # gradients of a mesh's vertices and weights
        dict(name="adjoint-mesh", kind="adjoint", geom="mesh", n=300, R=256, levels=3),
        # instances of uneven size in one graph, 4 lobes
        dict(name="batch", kind="batch", fibers=8, segs=600, n=160, R=128, K=4, N=2000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["yarn", "yarn", "woven", "mesh", "lod-yarn", "lod-mesh", "pyramid", "adjoint-yarn",
                         "adjoint-mesh", "batch"])
    if family == "yarn":
        R = rng.choice([64, 128, 256, 512])
        fibers = _log(rng, 4, 64)
        return dict(kind="voxelize", geom="yarn", fibers=fibers, segs=_log(rng, 90, 4000), R=R,
                    radius=round(rng.uniform(0.2, 2.05) / R, 6), weights=fibers < 32 or rng.random() < 0.5)
    if family == "woven":
        return dict(kind="voxelize", geom="woven", fibers=_log(rng, 8, 80), segs=_log(rng, 100, 700), R=1024,
                    radius=round(rng.uniform(0.002, 0.004), 6), weights=rng.random() < 0.5)
    if family == "mesh":
        n = _log(rng, 40, 1000)
        return dict(kind="voxelize", geom="mesh", n=n, R=128 if n < 120 else rng.choice([256, 512, 1024]),
                    weights=rng.random() < 0.5)
    if family == "lod-yarn":
        R = rng.choice([128, 256, 512])
        return dict(kind="lod", geom="yarn", fibers=_log(rng, 8, 56), segs=_log(rng, 400, 4000), R=R,
                    radius=round(rng.uniform(0.4, 2.0) / R, 6), K=rng.choice([2, 3, 4]),
                    N=rng.randint(1000, 5000), merge=rng.choice(["pooled", "mass"]))
    if family == "lod-mesh":
        return dict(kind="lod", geom="mesh", n=_log(rng, 64, 900), R=rng.choice([128, 256, 512]), K=rng.choice([1, 1, 2]),
                    N=rng.randint(1000, 3000), merge="pooled")
    if family == "pyramid":
        return dict(kind="pyramid", geom="yarn", fibers=_log(rng, 4, 24), segs=_log(rng, 100, 1500), R=64,
                    radius=round(rng.uniform(0.002, 0.012), 6), K=rng.choice([1, 2, 4]), N=rng.randint(500, 5000),
                    merge=rng.choice(["pooled", "mass"]))
    if family == "adjoint-yarn":
        R = rng.choice([64, 128, 256])
        return dict(kind="adjoint", geom="yarn", fibers=_log(rng, 4, 60), segs=_log(rng, 100, 4000), R=R,
                    radius=round(rng.uniform(0.3, 1.1) / R, 6), levels=rng.randint(0, 5))
    if family == "adjoint-mesh":
        return dict(kind="adjoint", geom="mesh", n=_log(rng, 40, 300), R=rng.choice([128, 256]), levels=rng.randint(0, 5))
    return dict(kind="batch", fibers=_log(rng, 3, 16), segs=_log(rng, 150, 1200), n=_log(rng, 40, 250),
                R=rng.choice([64, 128, 256]), K=rng.choice([1, 2, 4]), N=rng.randint(500, 3000))


# ---------------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(0x5EED + 7919 * int(seed))
    return g


def _uniform(g, n, lo=0.0, hi=1.0):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _yarn(g, fibers, segs, radius, scale=1.0, crimp=0.0):
    """Three plies of `fibers` fibers twisted around the x axis, polylines of `segs` segments.  The
    strands lie where they lie in every draw (so that a level has as many voxels); the seed decides
    the order in which the fibers come."""
    F = 3 * fibers
    order, g = torch.randperm(F, generator=g, device="cuda"), _gen(-1 - fibers)
    x = torch.linspace(0.0021, 0.9983, segs + 1, device="cuda", dtype=torch.float64)[None, :]
    ply = torch.arange(F, device="cuda", dtype=torch.float64).div(fibers, rounding_mode="floor")[:, None]
    f = (torch.arange(F, device="cuda", dtype=torch.float64) % fibers)[:, None]
    start = _uniform(g, 1, 0.0, 2.0 * math.pi)
    th = 2.0 * math.pi * ply / 3.0 + 4.0 * math.pi * x + start
    rho = scale * (0.1 * torch.sqrt((f + 0.5) / fibers) + _uniform(g, F, 0.0, 0.05)[:, None])
    ph = f * math.pi * (3.0 - math.sqrt(5.0)) - 4.0 * math.pi * x
    y = 0.5 + scale * 0.15 * torch.cos(th) + rho * torch.cos(ph)
    z = 0.5 + scale * 0.15 * torch.sin(th) + rho * torch.sin(ph) + crimp * torch.sin(16.0 * math.pi * x)
    r = torch.full_like(y, radius) * (1.0 + 0.05 * (_uniform(g, F)[:, None] - 0.5))
    ctrl = torch.stack([x.expand_as(y), y, z, r], dim=-1)[order].reshape(-1, 4).float().contiguous()
    return ctrl, torch.arange(F + 1, device="cuda", dtype=torch.int64) * (segs + 1)


def _mesh(g, n):
    """Brushed-metal heightfield: n x n vertices, ridges along x, two triangles per cell with
    unshared vertices, tilted a little.  The seed decides at which row of cells the list begins."""
    first, g = int(_uniform(g, 1, 0, n - 1)), _gen(-1 - n)
    h = 0.02 * torch.randn((n, n), generator=g, device="cuda", dtype=torch.float64)
    h = sum(torch.roll(h, k, 1) for k in range(-8, 8)) / 16.0
    s = _uniform(g, 4)
    v = torch.linspace(0.0, 1.0, n, device="cuda", dtype=torch.float64)
    X, Y = (0.004 + 0.004 * s[0] + 0.987 * v)[None, :].expand(n, n), (0.003 + 0.005 * s[1] + 0.986 * v)[:, None].expand(n, n)
    P = torch.stack([X, Y, 0.5 + h + 0.02 * (s[2] - 0.5) * X + 0.02 * (s[3] - 0.5) * Y, torch.zeros_like(X)], -1)
    a, b, c, d = P[:-1, :-1], P[:-1, 1:], P[1:, 1:], P[1:, :-1]
    cells = torch.stack([torch.stack([a, b, c], 2), torch.stack([a, c, d], 2)], 2)
    return torch.roll(cells, -first, 0).reshape(-1, 3, 4).float().contiguous()


def _geometry(case, g):
    """(arguments of Context.voxelize, primitive count)."""
    if case["geom"] == "mesh":
        kw = dict(tri_verts=_mesh(g, case["n"]))
        n = kw["tri_verts"].shape[0]
    else:
        woven = case["geom"] == "woven"
        ctrl, off = _yarn(g, case["fibers"], case["segs"], case["radius"], 0.2 if woven else 1.0, 0.03 if woven else 0.0)
        kw = dict(ctrl=ctrl, fiber_offsets=off)
        n = 3 * case["fibers"] * case["segs"]
    if case.get("weights") or case["kind"] != "voxelize":
        kw["weights"] = _uniform(g, n, 0.5, 2.0).float()
    return kw, n


def _directions(n):
    k = torch.arange(n, device="cuda", dtype=torch.float64)
    z = 1.0 - (2.0 * k + 1.0) / n
    r = torch.sqrt(torch.clamp(1.0 - z * z, min=0.0))
    ph = k * math.pi * (3.0 - math.sqrt(5.0))
    return torch.stack([r * torch.cos(ph), r * torch.sin(ph), z], 1).float().contiguous()


def _lod_args(case):
    return dict(K=case["K"], merge=case.get("merge", "pooled"), dirs=_directions(case["N"]) if case["K"] > 1 else None)


def prepare(case, seed):
    g = _gen(seed)
    s = dict(case=case, ctx=vx.Context(torch.device("cuda", torch.cuda.current_device())))
    if case["kind"] == "batch":
        inst = []
        for i in range(3):
            c, o = _yarn(g, case["fibers"] * (i + 1), case["segs"], 1.5 / case["R"])
            inst.append(dict(kind="fibers", grid=Grid((0.0, 0.0, 0.0), case["R"]), ctrl=c, fiber_offsets=o))
            inst.append(dict(kind="triangles", grid=Grid((0.0, 0.0, 0.0), case["R"] >> (i & 1)),
                             tri_verts=_mesh(g, max(8, case["n"] // (i + 1)))))
        a = _lod_args(case)
        s["batch"] = s["ctx"].batch(inst, K=a["K"], dirs=a["dirs"])
        s["grids"] = [i["grid"].resolution for i in inst]
        return s
    s["grid"] = Grid((0.0, 0.0, 0.0), case["R"])
    s["geom"], _ = _geometry(case, g)
    if case["kind"] in ("lod", "pyramid"):
        s["lod"] = _lod_args(case)
    if case["kind"] in ("lod", "adjoint"):
        s["level0"] = s["ctx"].voxelize(s["grid"], **s["geom"])
    if case["kind"] == "adjoint":
        s["keys"] = s["level0"].keys.clone()
        del s["level0"]
        s["gm"], s["gM"] = [], []
        for l in range(case["levels"] + 1):
            n = int(torch.unique_consecutive(s["keys"] >> (3 * l)).numel())
            s["gm"].append(_uniform(g, n, -1.0, 1.0).float())
            s["gM"].append(_uniform(g, 6 * n, -1.0, 1.0).float().reshape(n, 6))
    return s


# ---------------------------------------------------------------------------- one pass
def _fields(level):
    return {f: getattr(level, f) for f in FIELDS}


def _levels(levels, most):
    """The levels' arrays; those past `most` joined (they are small)."""
    out = [_fields(lv) for lv in levels[:most]]
    rest = levels[most:]
    if rest:
        out.append({f: torch.cat([getattr(lv, f) for lv in rest]) for f in FIELDS})
    return out


def run(state):
    ctx, kind = state["ctx"], state["case"]["kind"]
    if kind == "voxelize":
        return _fields(ctx.voxelize(state["grid"], **state["geom"]))
    if kind == "lod":
        return _levels(ctx.build_lod(state["level0"], **state["lod"]), 5)
    if kind == "pyramid":
        level0 = ctx.voxelize(state["grid"], **state["geom"])
        return _levels([level0] + ctx.build_lod(level0, **state["lod"]), 7)
    if kind == "adjoint":
        return ctx.backward(state["grid"], keys0=state["keys"], grad_mass=state["gm"], grad_moment=state["gM"], **state["geom"])
    b = state["batch"]
    b.run()
    finest = [b.level(i, 0) for i in range(len(state["grids"]))]
    coarse = [b.level(i, l) for i, R in enumerate(state["grids"]) for l in range(1, R.bit_length())]
    return _levels(finest + coarse, len(finest))


# ---------------------------------------------------------------------------- work
def _sizes(case):
    """(primitives, level-0 voxels, bytes of a primitive), the voxels from the geometry's extent."""
    R = case["R"]
    if case.get("geom") == "mesh":
        n = case["n"]
        return 2 * (n - 1) ** 2, int((1.2 + 0.0056 * n) * R * R), 48
    prims = 3 * case["fibers"] * case["segs"]
    length = (0.5 if case["geom"] == "woven" else 2.5) * R * 3 * case["fibers"]
    return prims, int(length * math.pi * (case["radius"] * R + 0.6) ** 2), 16


def work(case):
    if case["kind"] == "batch":
        parts = [dict(kind="pyramid", geom="yarn", fibers=case["fibers"] * (i + 1), segs=case["segs"], R=case["R"],
                      radius=1.5 / case["R"], K=case["K"], N=case["N"]) for i in range(3)]
        parts += [dict(kind="pyramid", geom="mesh", n=max(8, case["n"] // (i + 1)), R=case["R"] >> (i & 1), K=case["K"],
                       N=case["N"]) for i in range(3)]
        w = [work(p) for p in parts]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    prims, voxels, size = _sizes(case)
    if case["kind"] == "adjoint":
        # primitives, level-0 keys and every level's gradients in; gradients out
        return {"bytes": prims * (2 * size + 8) + voxels * (8 + 28 * 1.3), "flops": 150.0 * prims * 3}
    w = {"bytes": 0.0, "flops": 0.0}
    if case["kind"] in ("voxelize", "pyramid"):
        # each voxel's 512 sub-cells are decided at least once, about ten operations each
        w["bytes"] += prims * size + voxels * 158.0
        w["flops"] += voxels * 5120.0
    if case["kind"] in ("lod", "pyramid"):
        w["bytes"] += voxels * 158.0 + voxels * 0.3 * (106.0 + 52.0 * case["K"])
        if case["K"] > 1:
            # about one lobe sampling of N directions (45 operations each) per seven voxels
            w["flops"] += voxels / 7.0 * case["N"] * 45.0
    return w


# ---------------------------------------------------------------------------- 64 bits
def _morton(i):
    k = torch.zeros_like(i[..., 0])
    for b in range(11):
        for a in range(3):
            k |= ((i[..., a] >> b) & 1) << (3 * b + a)
    return k


def _pairs(lo, hi, R, chunk):
    """Chunks of (primitive, voxel index triple) over the inclusive voxel boxes [lo, hi]."""
    lo, hi = lo.floor().long().clamp(0, R), hi.floor().long().clamp(-1, R - 1)
    n = (hi - lo + 1).clamp(min=0)
    tot = n.prod(1)
    ends = tot.cumsum(0)
    p0 = 0
    while p0 < lo.shape[0]:
        base = int(ends[p0 - 1]) if p0 else 0
        p1 = max(p0 + 1, int(torch.searchsorted(ends, base + chunk, right=True)))
        p = torch.repeat_interleave(torch.arange(p0, p1, device=lo.device), tot[p0:p1])
        q = torch.arange(p.shape[0], device=lo.device) + base - (ends - tot)[p]
        nn = n[p].clamp(min=1)
        yield p, lo[p] + torch.stack([q % nn[:, 0], q // nn[:, 0] % nn[:, 1], q // (nn[:, 0] * nn[:, 1])], 1)
        p0 = p1


def _outer(t):
    return torch.stack([t[:, 0] ** 2, t[:, 1] ** 2, t[:, 2] ** 2, t[:, 0] * t[:, 1], t[:, 0] * t[:, 2], t[:, 1] * t[:, 2]], 1)


def _clip_segment(a, b):
    """Share of the segment a-b inside the unit box, per row."""
    d = b - a
    sd = torch.where(d == 0, torch.ones_like(d), d)
    t0, t1 = -a / sd, (1.0 - a) / sd
    near, far = torch.minimum(t0, t1), torch.maximum(t0, t1)
    out = ((d == 0) & ((a < 0) | (a > 1))).any(1)
    near = torch.where(d == 0, torch.zeros_like(near), near).amax(1)
    far = torch.where(d == 0, torch.ones_like(far), far).amin(1)
    # an end that lies on a face is an end of the segment (it does not slide along it)
    near, far = torch.where(near > 0, near, torch.zeros_like(near)), torch.where(far < 1, far, torch.ones_like(far))
    return torch.where(out | (far <= near), torch.zeros_like(near), far - near)


def _segment_box2(a, b):
    """Squared distance of segment a-b from the unit box (its minimum over the pieces between
    the parameters where a coordinate passes a face)."""
    d = b - a
    sd = torch.where(d == 0, torch.full_like(d, 1e-300), d)
    t = torch.cat([-a / sd, (1.0 - a) / sd, torch.zeros_like(a[:, :1]), torch.ones_like(a[:, :1])], 1).clamp(0.0, 1.0).sort(1).values
    best = torch.full_like(t[:, 0], math.inf)
    for i in range(t.shape[1] - 1):
        l, u = t[:, i:i + 1], t[:, i + 1:i + 2]
        m = a + 0.5 * (l + u) * d
        face, on = (m > 1).double(), ((m < 0) | (m > 1)).double()
        den = (on * d * d).sum(1, keepdim=True)
        s = torch.where(den > 0, (on * d * (face - a)).sum(1, keepdim=True) / torch.where(den > 0, den, torch.ones_like(den)), l)
        q = a + torch.maximum(torch.minimum(s, u), l) * d
        e = q - q.clamp(0.0, 1.0)
        best = torch.minimum(best, (e * e).sum(1))
    return best


def _triangle_gap(v):
    """Largest separation of the triangles v [n, 3, 3] from the unit box over the 13 axes of the
    separating-axis test (positive: apart)."""
    w = v - 0.5
    f = [w[:, 1] - w[:, 0], w[:, 2] - w[:, 1], w[:, 0] - w[:, 2]]
    axes = [torch.eye(3, device=v.device, dtype=v.dtype)[i].expand_as(f[0]) for i in range(3)]
    axes += [torch.linalg.cross(e, g) for e in list(axes) for g in f] + [torch.linalg.cross(f[0], f[1])]
    best = torch.full_like(w[:, 0, 0], -math.inf)
    for n in axes:
        size = n.abs().sum(1)
        p = (w * n[:, None, :]).sum(2)
        gap = torch.maximum(p.amin(1), -p.amax(1)) - 0.5 * size
        best = torch.maximum(best, torch.where(size > 1e-12, gap / size.clamp(min=1e-300), torch.full_like(gap, -math.inf)))
    return best


def _clip_area(v):
    """Area of the triangles v [n, 3, 3] inside the unit box (Sutherland-Hodgman, nine slots)."""
    n, M = v.shape[0], 9
    P = torch.cat([v, v[:, :1].expand(n, M - 3, 3)], 1)
    cnt = torch.full((n,), 3, device=v.device, dtype=torch.long)
    slot = torch.arange(M, device=v.device)[None, :]
    for axis in range(3):
        for c, sign in ((0.0, 1.0), (1.0, -1.0)):
            nxt = torch.where(slot + 1 < cnt[:, None], slot + 1, torch.zeros_like(slot))
            Q = P.gather(1, nxt[..., None].expand(-1, -1, 3))
            live = slot < cnt[:, None]
            x, y = P[..., axis], Q[..., axis]
            xin, yin = (x - c) * sign >= 0, (y - c) * sign >= 0
            cross = live & (xin != yin)
            den = torch.where(cross, y - x, torch.ones_like(x))
            s = torch.where(cross, (c - x) / den, torch.zeros_like(x))
            I = P + s[..., None] * (Q - P)
            both = torch.stack([P, I], 2).reshape(n, 2 * M, 3)
            keep = torch.stack([live & xin, cross], 2).reshape(n, 2 * M)
            order = torch.sort((~keep).long(), dim=1, stable=True).indices[:, :M]
            P, cnt = both.gather(1, order[..., None].expand(-1, -1, 3)), keep.sum(1)
    live = (slot < cnt[:, None])[..., None]
    first = P[:, :1]
    E = torch.where(live, P - first, torch.zeros_like(P))
    C = torch.linalg.cross(E[:, 1:-1], E[:, 2:]).sum(1)
    big = (C * C).sum(1)
    return 0.5 * torch.sqrt(torch.where(big > 0, big, torch.ones_like(big))) * (big > 0)


def _normal(v):
    n = torch.linalg.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 1])
    return n / n.norm(dim=1, keepdim=True)


def _coordinates(case, kw):
    """Grid coordinates of the primitives ((A, B, r) or the vertices), 64-bit, and their weights."""
    R = case["R"]
    if "tri_verts" in kw:
        v = kw["tri_verts"][..., :3].double() * R
        geom, n = (v,), v.shape[0]
    else:
        c, off = kw["ctrl"].double() * R, kw["fiber_offsets"]
        last = torch.zeros(c.shape[0], dtype=torch.bool, device=c.device)
        last[off[1:] - 1] = True
        i = torch.arange(c.shape[0], device=c.device)[~last]
        geom, n = (c[i, :3], c[i + 1, :3], 0.5 * (c[i, 3] + c[i + 1, 3])), i.shape[0]
    w = kw.get("weights")
    return geom, torch.ones(n, device="cuda", dtype=torch.float64) if w is None else w.double()


def _lobe(mass, moment):
    ok = (mass > 0)[:, None]
    S = torch.where(ok, moment / torch.where(ok, mass[:, None], torch.ones_like(mass[:, None])), torch.zeros_like(moment))
    d = torch.sqrt(S[:, :3])
    r = [torch.where(d[:, a] * d[:, b] > 0, S[:, k] / torch.where(d[:, a] * d[:, b] > 0, d[:, a] * d[:, b], torch.ones_like(mass)),
                     torch.zeros_like(mass)) for k, a, b in ((3, 0, 1), (4, 0, 2), (5, 1, 2))]
    return torch.cat([S, mass[:, None]], 1)[:, None, :], torch.cat([d, torch.stack(r, 1)], 1)[:, None, :]


def _numbers(mass, moment, lobes=True):
    out = dict.fromkeys(FIELDS)
    out["mass"], out["moment"] = mass, moment
    if lobes:
        out["lobes"], out["compact"] = _lobe(mass, moment)
    return out


def _exact_level0(case, kw):
    """(sorted keys, mass, moment) of level 0 in 64 bits; None where it would take long, or where
    a voxel's existence is within the rounding of 32-bit coordinates."""
    geom, w = _coordinates(case, kw)
    R = case["R"]
    if len(geom) == 1:
        lo, hi = geom[0].amin(1) - 1e-3, geom[0].amax(1) + 1e-3
        T = _outer(_normal(geom[0]))
    else:
        A, B, r = geom
        lo, hi = torch.minimum(A, B) - r[:, None] - 1e-3, torch.maximum(A, B) + r[:, None] + 1e-3
        T = _outer((B - A) / (B - A).norm(dim=1, keepdim=True))
    if float((hi - lo + 1).prod(1).sum()) > 3e7:
        return None
    keys, sure, meas, prim = [], [], [], []
    for p, ijk in _pairs(lo, hi, R, 1 << 20):
        if len(geom) == 1:
            v = geom[0][p] - ijk[:, None, :]
            gap = _triangle_gap(v)
            mu = _clip_area(v)
        else:
            a, b = A[p] - ijk, B[p] - ijk
            gap = torch.sqrt(_segment_box2(a, b)) - r[p]
            mu = math.pi * r[p] ** 2 * _clip_segment(a, b) * (b - a).norm(dim=1)
        at = gap < 1e-6
        keys.append(_morton(ijk[at]))
        sure.append(gap[at] < -1e-6 if len(geom) > 1 else gap[at] < -1e-7)
        meas.append(mu[at])
        prim.append(p[at])
    keys, sure, meas, prim = (torch.cat(x) for x in (keys, sure, meas, prim))
    uniq, at = torch.unique(keys, return_inverse=True)
    known = torch.zeros(uniq.shape[0], dtype=torch.long, device=keys.device).scatter_add_(0, at, sure.long())
    if int((known == 0).sum()):
        return None
    c = w[prim] * meas
    mass = torch.zeros(uniq.shape[0], device=keys.device, dtype=torch.float64).index_add_(0, at, c)
    moment = torch.zeros(uniq.shape[0], 6, device=keys.device, dtype=torch.float64).index_add_(0, at, c[:, None] * T[prim])
    return uniq, mass, moment


def _exact_levels(keys, mass, moment, R, K):
    out = []
    while R > 1:
        keys, at = torch.unique_consecutive(keys >> 3, return_inverse=True)
        mass = torch.zeros(keys.shape[0], device=keys.device, dtype=torch.float64).index_add_(0, at, mass)
        moment = torch.zeros(keys.shape[0], 6, device=keys.device, dtype=torch.float64).index_add_(0, at, moment)
        out.append(_numbers(mass, moment, K == 1))
        R //= 2
    return out


def _joined(levels, most):
    rest = levels[most:]
    out = levels[:most]
    if rest:
        out.append({f: None if rest[0][f] is None else torch.cat([x[f] for x in rest]) for f in FIELDS})
    return out


def _exact_adjoint(case, state):
    """Gradients by automatic differentiation of the 64-bit measures."""
    R, keys = case["R"], state["keys"]
    gm = torch.zeros(keys.shape[0], device="cuda", dtype=torch.float64)
    gM = torch.zeros(keys.shape[0], 6, device="cuda", dtype=torch.float64)
    for l, (m, M) in enumerate(zip(state["gm"], state["gM"])):
        at = torch.unique_consecutive(keys >> (3 * l), return_inverse=True)[1]
        gm += m.double()[at]
        gM += M.double()[at]
    geom, w = _coordinates(case, state["geom"])
    geom, w = [x.requires_grad_(True) for x in geom], w.requires_grad_(True)
    pts = geom[0].detach() if len(geom) == 1 else torch.stack([geom[0].detach(), geom[1].detach()], 1)
    for p, ijk in _pairs(pts.amin(1), pts.amax(1), R, 1 << (18 if len(geom) == 1 else 20)):
        k = _morton(ijk)
        v = torch.searchsorted(keys, k).clamp(max=keys.shape[0] - 1)
        at = keys[v] == k
        p, ijk, v = p[at], ijk[at], v[at]
        if len(geom) == 1:
            t = geom[0][p] - ijk[:, None, :]
            mu, T = _clip_area(t), _outer(_normal(t))
        else:
            a, b = geom[0][p] - ijk, geom[1][p] - ijk
            dn = (b - a).norm(dim=1)
            mu, T = math.pi * geom[2][p] ** 2 * _clip_segment(a, b) * dn, _outer((b - a) / dn[:, None])
        (w[p] * mu * (gm[v] + (gM[v] * T).sum(1))).sum().backward()
    if len(geom) == 1:
        g = torch.zeros(geom[0].shape[0], 3, 4, device="cuda", dtype=torch.float64)
        g[..., :3] = geom[0].grad * R
        return g, w.grad
    c, off = state["geom"]["ctrl"], state["geom"]["fiber_offsets"]
    last = torch.zeros(c.shape[0], dtype=torch.bool, device="cuda")
    last[off[1:] - 1] = True
    i = torch.arange(c.shape[0], device="cuda")[~last]
    g = torch.zeros(c.shape[0], 4, device="cuda", dtype=torch.float64)
    half = 0.5 * geom[2].grad[:, None]
    g.index_add_(0, i, torch.cat([geom[0].grad, half], 1) * R)
    g.index_add_(0, i + 1, torch.cat([geom[1].grad, half], 1) * R)
    return g, w.grad


def exact(case, seed):
    """What run() returns, in 64 bits: masses, moments, single lobes and gradients.  Keys, masks and
    counts are whole numbers and have none; nor have merged lobes (they follow integer decisions).
    The input level of a `lod` case and the keys of an `adjoint` case are those of prepare()."""
    if case["kind"] == "batch":
        return None
    if case["kind"] == "lod":
        s = prepare(case, seed)
        lv = s["level0"]
        return _joined(_exact_levels(lv.keys, lv.mass.double(), lv.moment.double(), case["R"], case["K"]), 5)
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, prepare(case, seed))
    kw, _ = _geometry(case, _gen(seed))
    got = _exact_level0(case, kw)
    if got is None:
        return None
    level0 = _numbers(got[1], got[2])
    if case["kind"] == "voxelize":
        return level0
    return _joined([level0] + _exact_levels(*got, case["R"], case["K"]), 7)
