"""Kernels at the sizes and positions where their fast paths hand over to the definition, against
the CPU oracle.  Whole numbers and FP32 sums are compared bit for bit."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2604_13191_gb300 as vx  # noqa: E402

DEV = torch.device("cuda", 0)


def _same_level0(got, ref):
    g = got.host()
    for f, r in (("keys", "keys"), ("mask", "mask"), ("occ", "occ"), ("proj", "proj")):
        assert np.array_equal(g[f], ref[r]), f
    for f in ("mass", "moment"):
        assert np.array_equal(g[f].view(np.uint32), ref[f].view(np.uint32)), f


@pytest.mark.parametrize("n,R,size,snap", [
    (1, 8, (0.5, 0.5), 0),          # one triangle
    (300, 16, (0.2, 3.0), 8),       # vertices on sub-cell planes: every axis test at its boundary
    (300, 16, (0.2, 3.0), 16),      # vertices on sub-cell centres
    (60, 64, (8.0, 40.0), 8),       # triangles many voxels wide
    (400, 32, (0.001, 0.1), 0),     # far smaller than a sub-cell
    (900, 4, (0.3, 1.0), 0),        # voxels of several batches of 32 triangles
    (120, 4, (0.2, 0.5), 2),        # groups of voxels at the edge of 32, vertices on voxel planes
])
def test_triangle_masks_at_the_boundaries(n, R, size, snap):
    tris, grid = synth.random_triangles(n, R, seed=100 + n + R, size=size)
    if snap:
        tris[..., :3] = np.round(tris[..., :3] * (R * snap)) / (R * snap)
    tris[n // 2] = tris[n // 2, :1]                       # a triangle without area
    rng = np.random.default_rng(n)
    w = synth.Workload("tris", "triangles", grid, tri_verts=tris, K=1,
                       weights=rng.uniform(0.5, 2.0, n).astype(np.float32))
    ctx = vx.Context(DEV)
    got = ctx.voxelize(grid, tri_verts=torch.from_numpy(tris).to(DEV), weights=torch.from_numpy(w.weights).to(DEV))
    _same_level0(got, oracle.voxelize(w))
    ctx.close()


@pytest.mark.parametrize("n_fibers,pts,R,radius,step,snap", [
    (1, 2, 8, (0.3, 0.3), (0.5, 0.5), 0),         # one capsule
    (40, 20, 16, (0.4, 1.5), (0.1, 2.0), 8),      # ends on sub-cell planes
    (40, 20, 32, (2.0, 4.0), (0.1, 0.5), 0),      # radius of several voxels: covered voxels
    (60, 12, 16, (0.02, 0.2), (2.0, 9.0), 0),     # long and thin: most sub-cells go to step 3
    (30, 30, 4, (0.1, 0.4), (0.05, 0.4), 0),      # voxels of several batches of 32 capsules
    (20, 6, 64, (0.3, 0.9), (20.0, 60.0), 4),     # tens of voxels long, ends on sub-cell corners
    (25, 20, 8, (0.125, 0.125), (0.125, 0.5), 8), # radius and steps of whole sub-cells
])
def test_capsule_masks_at_the_boundaries(n_fibers, pts, R, radius, step, snap):
    ctrl, off, grid = synth.random_segments(n_fibers, pts, R, seed=300 + n_fibers + R, radius=radius, step=step)
    if snap:
        ctrl[:, :3] = np.round(ctrl[:, :3] * (R * snap)) / (R * snap)
    ctrl[1, :3] = ctrl[0, :3]                             # a segment without length
    rng = np.random.default_rng(n_fibers)
    n = synth.fiber_segment_count(off)
    w = synth.Workload("caps", "fibers", grid, ctrl=ctrl, fiber_offsets=off, K=1,
                       weights=rng.uniform(0.0, 2.0, n).astype(np.float32))
    ctx = vx.Context(DEV)
    got = ctx.voxelize(grid, ctrl=torch.from_numpy(ctrl).to(DEV), fiber_offsets=torch.from_numpy(off).to(DEV),
                       weights=torch.from_numpy(w.weights).to(DEV))
    _same_level0(got, oracle.voxelize(w))
    ctx.close()


def _adjoint_case(kind, seed, R, levels, n, **kw):
    rng = np.random.default_rng(seed)
    ctx = vx.Context(DEV)
    if kind == "fibers":
        ctrl, off, grid = synth.random_segments(n, kw.get("pts", 12), R, seed=seed, radius=kw["radius"], step=kw["step"])
        geom = dict(ctrl=torch.from_numpy(ctrl).to(DEV), fiber_offsets=torch.from_numpy(off).to(DEV))
        count = synth.fiber_segment_count(off)
    else:
        tris, grid = synth.random_triangles(n, R, seed=seed, size=kw["size"])
        geom = dict(tri_verts=torch.from_numpy(tris).to(DEV))
        count = n
    geom["weights"] = torch.from_numpy(rng.uniform(0.5, 2.0, count).astype(np.float32)).to(DEV)
    keys = ctx.voxelize(grid, **geom).keys.clone()
    gm, gM = [], []
    for l in range(levels + 1):
        v = int(torch.unique_consecutive(keys >> (3 * l)).numel())
        gm.append(torch.from_numpy(rng.uniform(-1, 1, v).astype(np.float32)).to(DEV))
        gM.append(torch.from_numpy(rng.uniform(-1, 1, (v, 6)).astype(np.float32)).to(DEV))
    return ctx, grid, geom, keys, gm, gM


@pytest.mark.parametrize("kind,n,R,levels,kw", [
    ("fibers", 1, 8, 0, dict(pts=2, radius=(0.4, 0.4), step=(0.6, 0.6))),
    ("fibers", 3, 256, 5, dict(pts=3, radius=(0.3, 0.5), step=(90.0, 140.0))),    # few and long
    ("fibers", 40, 64, 6, dict(pts=30, radius=(0.2, 2.0), step=(0.05, 6.0))),
    ("fibers", 900, 32, 3, dict(pts=100, radius=(0.1, 0.4), step=(0.02, 0.6))),   # a segment per lane
    ("triangles", 1, 8, 0, dict(size=(0.6, 0.6))),
    ("triangles", 6, 128, 4, dict(size=(30.0, 50.0))),                            # few and large
    ("triangles", 3000, 32, 5, dict(size=(0.1, 2.0))),
])
def test_adjoint_walks_every_voxel(kind, n, R, levels, kw):
    """The gradient with respect to the weights is each primitive's own loss, so it is computed
    again from the forward pass of that primitive alone: sum over its voxels and the levels'
    gradients of their ancestors.  A voxel that the walk misses would show as a missing term.
    Tolerance: masses of up to a few hundred FP32 terms (1e-5) of the sum of magnitudes."""
    ctx, grid, geom, keys, gm, gM = _adjoint_case(kind, 7 + n, R, levels, n, **kw)
    g_geom, g_w = ctx.backward(grid, keys0=keys, grad_mass=gm, grad_moment=gM, **geom)
    assert bool(torch.isfinite(g_geom).all())
    gm0 = torch.zeros(keys.shape[0], dtype=torch.float64, device=DEV)
    gM0 = torch.zeros(keys.shape[0], 6, dtype=torch.float64, device=DEV)
    for l in range(levels + 1):
        at = torch.unique_consecutive(keys >> (3 * l), return_inverse=True)[1]
        gm0 += gm[l].double()[at]
        gM0 += gM[l].double()[at]
    count = g_w.shape[0]
    pick = range(count) if count <= 40 else np.random.default_rng(1).choice(count, 40, replace=False)
    for p in pick:
        p = int(p)
        if kind == "fibers":
            off = geom["fiber_offsets"]
            pts = kw["pts"]
            c = (p // (pts - 1)) * pts + p % (pts - 1)
            one = dict(ctrl=geom["ctrl"][c:c + 2].contiguous(), fiber_offsets=off.new_tensor([0, 2]))
        else:
            one = dict(tri_verts=geom["tri_verts"][p:p + 1].contiguous())
        lv = ctx.voxelize(grid, **one)
        at = torch.searchsorted(keys, lv.keys)
        assert bool((keys[at] == lv.keys).all())
        terms = lv.mass.double() * gm0[at] + (lv.moment.double() * gM0[at]).sum(1)
        size = float((lv.mass.double() * gm0[at].abs() + (lv.moment.double() * gM0[at]).abs().sum(1)).sum())
        assert abs(float(g_w[p]) - float(terms.sum())) <= 1e-5 * size + 1e-7, p
    # the pair limit refuses what it refused: one voxel of more pairs than a pass may hold
    ctx.set_max_pairs_per_pass(10 ** 9)
    again = ctx.backward(grid, keys0=keys, grad_mass=gm, grad_moment=gM, **geom)
    assert torch.equal(again[0], g_geom) and torch.equal(again[1], g_w)
    if count > 1000:
        ctx.set_max_pairs_per_pass(1)
        with pytest.raises(vx.VxError) as e:
            ctx.backward(grid, keys0=keys, grad_mass=gm, grad_moment=gM, **geom)
        assert e.value.status == 3
    ctx.close()


@pytest.mark.parametrize("N,scale", [(1, 1.0), (31, 1.0), (333, 0.3), (1000, 5.0), (2049, 1.0)])
def test_lobe_sampling_paths(N, scale):
    """Direction counts below and around a warp, odd ones, and directions that are not unit vectors
    (outside the range of the packed reciprocal): every level against the oracle."""
    ctrl, off, grid = synth.random_segments(12, 40, 16, seed=5, radius=(0.2, 0.8), step=(0.2, 1.5))
    dirs = (synth.sample_directions(max(N, 2))[:N] * np.float32(scale)).astype(np.float32)
    ctx = vx.Context(DEV)
    L0 = ctx.voxelize(grid, ctrl=torch.from_numpy(ctrl).to(DEV), fiber_offsets=torch.from_numpy(off).to(DEV))
    got = ctx.build_lod(L0, K=2, dirs=torch.from_numpy(dirs).to(DEV))
    refs = oracle.build_pyramid(oracle.voxelize_fibers(ctrl, off, grid, K=1), 16, 2, dirs)
    for lv, r in zip(got, refs):
        g = lv.host()
        assert np.array_equal(g["keys"], r["keys"]) and np.array_equal(g["lobe_count"], r["lobe_count"])
        assert np.max(np.abs(g["lobes"] - r["lobes"])[..., :6]) <= 1e-5
    ctx.close()


@pytest.mark.parametrize("N", [20001, 65535])
def test_lobe_counts_at_the_thresholds(N):
    """Histogram counts are compared at FP32 rounding: with many directions some samples fall within
    one rounding of a threshold, and a mesh's nearly equal lobes turn a count that is off by one
    into another merge.  Every lobe equals the oracle's bit for bit."""
    tris = synth.heightfield(30, seed=N, sigma=0.1)
    grid = synth.Grid((0.0, 0.0, -0.5), 1.0 / 32, 32)
    dirs = synth.sample_directions(N)
    ctx = vx.Context(DEV)
    L0 = ctx.voxelize(grid, tri_verts=torch.from_numpy(tris).to(DEV))
    got = ctx.build_lod(L0, K=2, dirs=torch.from_numpy(dirs).to(DEV))
    w = synth.Workload("hf", "triangles", grid, tri_verts=tris, K=2)
    refs = oracle.build_pyramid(oracle.voxelize(w, K=1), 32, 2, dirs)
    for lv, r in zip(got, refs):
        g = lv.host()
        assert np.array_equal(g["lobe_count"], r["lobe_count"])
        for k in range(2):
            sel = r["lobe_count"] > k
            assert np.array_equal(g["lobes"][sel, k].view(np.uint32), r["lobes"][sel, k].astype(np.float32).view(np.uint32))
    ctx.close()


@pytest.mark.parametrize("n", [2, 33, 4095, 4096, 4097, 8192, 12290])
@pytest.mark.parametrize("R", [4, 8, 64, 256])
def test_pair_sort_at_the_tile_edges(n, R):
    """One pair per triangle (each lies inside a voxel), so that n is the sort's length: below, at and
    above a tile, with key digits of 6, 9, 9 + 9 and 8 + 8 + 8 bits.  Half of the pairs share one
    voxel, whose FP32 sums depend on the order that a stable sort keeps."""
    rng = np.random.default_rng(n + R)
    cell = rng.integers(0, R, (n, 3))
    cell[rng.random(n) < 0.5] = cell[0]
    v = (cell[:, None, :] + rng.uniform(0.3, 0.7, (n, 3, 3))) / R
    tris = np.zeros((n, 3, 4), np.float32)
    tris[..., :3] = v
    grid = synth.Grid((0.0, 0.0, 0.0), 1.0 / R, R)
    w = synth.Workload("cells", "triangles", grid, tri_verts=tris, K=1)
    ctx = vx.Context(DEV)
    _same_level0(ctx.voxelize(grid, tri_verts=torch.from_numpy(tris).to(DEV)), oracle.voxelize(w))
    ctx.close()


@pytest.mark.parametrize("kind,n,R", [("tri", 1, 4), ("tri", 14593, 16), ("tri", 29185, 32), ("cap", 1, 4), ("cap", 2, 64),
                                      ("cap", 14595, 32), ("cap", 29190, 16)])
def test_candidates_of_groups(kind, n, R):
    """The count pass takes 1, 2 or 4 primitives per warp at these lengths (the last group is short), and
    two capsules whose ranges hold more than 65,536 voxels: every level-0 value against the oracle."""
    if kind == "tri":
        tris, grid = synth.random_triangles(n, R, seed=n, size=(0.05, 1.2))
        tris[::7, 2, :3] = tris[::7, 0, :3]                       # without area
        w = synth.Workload("count", "triangles", grid, tri_verts=tris, K=1)
        geom = dict(tri_verts=torch.from_numpy(tris).to(DEV))
    else:
        if n == 2:
            ctrl = np.array([[0.1, 0.1, 0.1, 0.05], [0.9, 0.85, 0.8, 0.05], [0.2, 0.9, 0.15, 0.02]], np.float32)
            off, grid = np.array([0, 3], np.int64), synth.Grid((0.0, 0.0, 0.0), 1.0 / R, R)
        else:
            ctrl, off, grid = synth.random_segments(max(n // 139, 1), min(n, 139) + 1, R, seed=n, radius=(0.05, 0.8))
        w = synth.Workload("count", "fibers", grid, ctrl=ctrl, fiber_offsets=off, K=1)
        geom = dict(ctrl=torch.from_numpy(ctrl).to(DEV), fiber_offsets=torch.from_numpy(off).to(DEV))
    ctx = vx.Context(DEV)
    _same_level0(ctx.voxelize(grid, **geom), oracle.voxelize(w))
    ctx.close()


@pytest.mark.parametrize("n", [131072, 131073])
def test_pair_sort_with_and_without_its_own_offsets(n):
    """32 tiles (each block sums the tile counts itself) and 33 (a scan does): the level equals, bit
    for bit, the one whose pairs are sorted window by window in shorter pieces."""
    R = 64
    rng = np.random.default_rng(n)
    v = (rng.integers(0, R, (n, 1, 3)) + rng.uniform(0.3, 0.7, (n, 3, 3))) / R
    tris = np.zeros((n, 3, 4), np.float32)
    tris[..., :3] = v
    grid = synth.Grid((0.0, 0.0, 0.0), 1.0 / R, R)
    geom = torch.from_numpy(tris).to(DEV)
    ctx = vx.Context(DEV)
    whole = ctx.voxelize(grid, tri_verts=geom).host()
    ctx.set_max_pairs_per_pass(n // 3)
    parts = ctx.voxelize(grid, tri_verts=geom).host()
    assert whole["occ"].shape[0] > 90000 and np.all(np.diff(whole["keys"].astype(np.int64)) > 0)
    for f in ("keys", "mask", "mass", "moment", "occ", "proj", "lobes"):
        assert np.array_equal(np.asarray(whole[f]).view(np.uint8), np.asarray(parts[f]).view(np.uint8)), f
    ctx.close()


@pytest.mark.parametrize("a,b,r", [
    ((-4e19, -4e19, -4e19), (-4.1e19, -4e19, -4e19), 6e19),      # every sum of squares overflows
    ((4e19, 0, 0), (4e19, 1e19, 0), 7e19),                       # the squares of one axis do
    ((3, -4e19, -4e19), (5, -4e19, -4e19), 6e19),                # those of two
    ((-4e19, 3, -4e19), (-4e19, 5, -4e19), 6e19),
    ((-4e19, -4e19, 3), (4e19, 4e19, 3), 6e19),                  # the axis runs through the grid
    ((1e19, 1e19, 1e19), (1e19, 1e19, 1.2e19), 2e19),            # only the radius does
    ((2e19, 1e19, 1e19), (2e19, 1e19, 1e19), 3e19),              # without length
])
def test_capsule_radius_whose_square_overflows(a, b, r):
    """r^2 is infinite in FP32: the comparisons of steps 1 and 2 hold against an infinite budget and against
    none that is not a number, and step 3's minimum is at most r^2 whatever it is.  Stated here in
    numpy's FP32, sub-cell by sub-cell."""
    R, f32 = 8, np.float32
    ctrl = np.array([[*a, r], [*b, r]], f32)
    i = np.arange(R)
    vox = np.stack(np.meshgrid(i, i, i, indexing="ij"), -1).reshape(-1, 3).astype(f32)
    lo = np.arange(8).astype(f32) * f32(0.125)
    hi = (np.arange(8) + 1).astype(f32) * f32(0.125)
    with np.errstate(over="ignore", invalid="ignore"):
        def squares(p, q):                                       # [voxel, axis, interval]
            mn, mx = np.minimum(p, q)[..., None], np.maximum(p, q)[..., None]
            g = np.maximum(np.maximum(lo - mx, mn - hi), f32(0))
            return g * g
        A, B = ctrl[0, :3] - vox, ctrl[1, :3] - vox
        rr = f32(ctrl[0, 3] * ctrl[0, 3])
        assert np.isinf(rr)
        bits = np.zeros((R ** 3, 8, 8, 8), bool)                 # [voxel, sz, sy, sx]
        for s in (squares(A, B), squares(A, A), squares(B, B)):
            T = rr - (s[:, 1, None, :] + s[:, 2, :, None])       # [voxel, sz, sy]
            bits |= s[:, 0, None, None, :] <= T[..., None]
    words = np.packbits(bits.reshape(R ** 3, 512), axis=1, bitorder="little").view(np.uint64)
    key = np.zeros(R ** 3, np.uint64)
    for t in range(3):
        for ax in range(3):
            key |= ((vox[:, ax].astype(np.uint64) >> np.uint64(t)) & np.uint64(1)) << np.uint64(3 * t + ax)
    order = np.argsort(key)
    order = order[words[order].any(1)]
    ctx = vx.Context(DEV)
    got = ctx.voxelize(synth.Grid((0.0, 0.0, 0.0), 1.0, R), ctrl=torch.from_numpy(ctrl).to(DEV),
                       fiber_offsets=torch.tensor([0, 2], device=DEV)).host()
    assert np.array_equal(got["keys"].astype(np.uint64), key[order])
    assert np.array_equal(got["mask"].view(np.uint64).reshape(-1, 8), words[order])
    ctx.close()


def _sheet(n, axis, level, lo, hi):
    """n x n vertices of a plane sheet at right angles to `axis`, two triangles per cell."""
    u = np.linspace(lo, hi, n)
    P = np.full((n, n, 3), level)
    P[..., (axis + 1) % 3], P[..., (axis + 2) % 3] = u[None, :], u[:, None]
    a, b, c, d = P[:-1, :-1], P[:-1, 1:], P[1:, 1:], P[1:, :-1]
    t = np.zeros((n - 1, n - 1, 2, 3, 4), np.float32)
    t[..., 0, 0, :3], t[..., 0, 1, :3], t[..., 0, 2, :3] = a, b, c
    t[..., 1, 0, :3], t[..., 1, 1, :3], t[..., 1, 2, :3] = a, c, d
    return t.reshape(-1, 3, 4)


@pytest.mark.parametrize("n,R,level,lo,hi", [
    (30, 16, 0.3337, 0.06, 0.94),     # edges along two axes, nothing on a plane
    (17, 16, 0.5, 0.0, 1.0),          # everything on voxel planes
    (30, 16, 17 / 128, 0.06, 0.94),   # the sheets on sub-cell planes
    (3, 32, 0.61, 0.1, 0.9),          # edges of many voxels
])
def test_edges_along_the_axes(n, R, level, lo, hi):
    """A box's faces: edges parallel to an axis (their edge axis in that family is zero, and separates
    nothing) and diagonals in the coordinate planes."""
    tris = np.concatenate([_sheet(n, ax, z, lo, hi) for ax in range(3) for z in (level, 1.0 - level)])
    grid = synth.Grid((0.0, 0.0, 0.0), 1.0 / R, R)
    ctx = vx.Context(DEV)
    got = ctx.voxelize(grid, tri_verts=torch.from_numpy(tris).to(DEV))
    _same_level0(got, oracle.voxelize(synth.Workload("box", "triangles", grid, tri_verts=tris, K=1)))
    ctx.close()


def test_edges_along_the_axes_cost_nothing():
    """A flat sheet whose edges lie along the axes takes no longer than the same sheet turned a little (its
    zero edge axes sent every row to the definition, and the sheet took 1.3 times as long)."""
    n, R = 2048, 1024
    flat = _sheet(n, 2, 0.50031, 0.05, 0.95)
    turned = flat.copy()
    turned[..., 0], turned[..., 1] = flat[..., 0] + 0.01 * flat[..., 1], flat[..., 1] - 0.01 * flat[..., 0]
    turned[..., 2] += 0.01 * (flat[..., 0] - flat[..., 1])
    grid = synth.Grid((0.0, 0.0, 0.0), 1.0 / R, R)
    ctx = vx.Context(DEV)
    best = []
    for t in (flat, turned):
        geom = torch.from_numpy(t).to(DEV)
        times = []
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            ctx.voxelize(grid, tri_verts=geom)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        best.append(min(times))
    assert best[0] < 1.15 * best[1], best
    ctx.close()


@pytest.mark.parametrize("kind,R", [("tri", 4), ("tri", 8), ("tri", 64), ("cap", 4), ("cap", 8), ("cap", 64)])
def test_one_primitive_with_extent(kind, R):
    """The smallest batch and the shortest group: one pair's lane, or one primitive in every voxel."""
    grid = synth.Grid((0.0, 0.0, 0.0), 1.0 / R, R)
    if kind == "tri":
        tris = np.array([[[1.2, 1.3, 1.25, 0.0], [1.9, 1.4, 1.8, 0.0], [1.3, 2.6, 1.6, 0.0]]], np.float32) / np.float32(R)
        w = synth.Workload("one", "triangles", grid, tri_verts=tris, K=1)
        geom = dict(tri_verts=torch.from_numpy(tris).to(DEV))
    else:
        ctrl = np.array([[1.3, 1.4, 1.6, 0.2], [1.7, 2.6, 1.4, 0.3]], np.float32) / np.float32(R)
        off = np.array([0, 2], np.int64)
        w = synth.Workload("one", "fibers", grid, ctrl=ctrl, fiber_offsets=off, K=1)
        geom = dict(ctrl=torch.from_numpy(ctrl).to(DEV), fiber_offsets=torch.from_numpy(off).to(DEV))
    ref = oracle.voxelize(w)
    assert ref["keys"].shape[0] >= 2 and float(ref["mass"].min()) >= 0.0 and float(ref["mass"].sum()) > 0.1
    ctx = vx.Context(DEV)
    _same_level0(ctx.voxelize(grid, **geom), ref)
    ctx.close()
