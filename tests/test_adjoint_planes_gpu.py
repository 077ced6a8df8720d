"""The adjoint where primitives meet voxel planes exactly: coordinates on planes, negative zeros."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2604_13191_gb300 as vx  # noqa: E402

DEV = torch.device("cuda", 0)


def _loss(keys, seed):
    rng = np.random.default_rng(seed)
    n = keys.shape[0]
    return (torch.from_numpy(rng.uniform(-1, 1, n).astype(np.float32)).to(DEV),
            torch.from_numpy(rng.uniform(-1, 1, (n, 6)).astype(np.float32)).to(DEV))


def _geom(kind, p, weights):
    t = torch.from_numpy(np.ascontiguousarray(p)).to(DEV)
    w = torch.from_numpy(weights).to(DEV)
    if kind == "triangles":
        return dict(tri_verts=t, weights=w)
    return dict(ctrl=t.reshape(-1, 4), fiber_offsets=torch.arange(p.shape[0] + 1, device=DEV) * 2, weights=w)


def _snapped(kind, n, R, snap, extent, seed, lo=0.0):
    """n primitives with coordinates that are multiples of 1 / snap voxels, from `lo` voxels on."""
    rng = np.random.default_rng(seed)
    k = 3 if kind == "triangles" else 2
    p = rng.uniform(lo, R - 1.0, (n, 1, 3)) + rng.uniform(-0.5, 0.5, (n, k, 3)) * extent
    out = np.zeros((n, k, 4), np.float32)
    out[..., :3] = np.round(p * snap) / snap / R
    if kind == "fibers":
        out[..., 3] = 0.3 / R
    return out, rng.uniform(0.5, 2.0, n).astype(np.float32)


@pytest.mark.parametrize("kind", ["triangles", "fibers"])
@pytest.mark.parametrize("snap", [1, 2, 8])
def test_negative_zeros(kind, snap):
    """A coordinate of -0 is one of +0 (the grid begins at 0, so both lie on its first planes)."""
    R, n = 8, 3000
    p, w = _snapped(kind, n, R, snap, 5.0, snap, lo=-2.0)
    neg = p.copy()
    neg[p == 0.0] = -0.0
    assert int((p[..., :3] == 0.0).sum()) > 100
    grid = synth.Grid((0.0, 0.0, 0.0), 1.0 / R, R)
    ctx = vx.Context(DEV)
    keys = ctx.voxelize(grid, **_geom(kind, p, w)).keys.clone()
    gm, gM = _loss(keys, 3)
    got = []
    for x in (p, neg):
        g, gw = ctx.backward(grid, keys0=keys, grad_mass=[gm], grad_moment=[gM], **_geom(kind, x, w))
        got.append((g.cpu().numpy(), gw.cpu().numpy()))
    assert np.array_equal(got[0][1], got[1][1])
    assert np.array_equal(got[0][0], got[1][0], equal_nan=True)
    ctx.close()


def _clip_gradient(U, vox, gm, gM):
    """d/dU of area(U cut by the voxel) * (gm + gM . T(n)), and that value: Sutherland-Hodgman on voxel-local
    coordinates in plain FP64 operations, the area's derivative from the polygon's edges on voxel planes."""
    U = [[float(c) for c in v] for v in U]
    e1, e2 = [[U[j][k] - U[0][k] for k in range(3)] for j in (1, 2)]
    poly = [([U[j][k] - vox[k] for k in range(3)], (0.0, 1.0, 0.0)[j], (0.0, 0.0, 1.0)[j], -1) for j in range(3)]
    for c in range(6):
        k, bound = c >> 1, float(c & 1)
        inside = [p[0][k] <= 1.0 if c & 1 else p[0][k] >= 0.0 for p in poly]
        out = []
        for i, p in enumerate(poly):
            j = (i + 1) % len(poly)
            q = poly[j]
            if inside[i]:
                out.append(p)
            if inside[i] != inside[j]:
                l = (bound - p[0][k]) / (q[0][k] - p[0][k])
                x = [bound if a == k else p[0][a] + l * (q[0][a] - p[0][a]) for a in range(3)]
                out.append((x, p[1] + l * (q[1] - p[1]), p[2] + l * (q[2] - p[2]), c if inside[i] else p[3]))
        poly = out
        if not poly:
            return np.zeros((3, 3)), 0.0
    A, dA = 0.0, np.zeros((3, 3))
    for i, p in enumerate(poly):
        q = poly[(i + 1) % len(poly)]
        A += p[1] * q[2] - q[1] * p[2]
        if p[3] < 0:
            continue
        k = p[3] >> 1
        g = np.hypot(e1[k], e2[k])
        if g == 0.0:
            continue
        f = np.hypot(q[1] - p[1], q[2] - p[2]) / g * (-1.0 if p[3] & 1 else 1.0)
        s, t = 0.5 * (p[1] + q[1]), 0.5 * (p[2] + q[2])
        dA[:, k] += [f * (1.0 - s - t), f * s, f * t]
    A *= 0.5
    n = np.array([e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2], e1[0] * e2[1] - e1[1] * e2[0]])
    J = float(np.sqrt((n * n).sum()))
    if len(poly) < 3 or not J > 0.0 or not A > 0.0:
        return np.zeros((3, 3)), 0.0
    n /= J
    M = np.array([[gM[0], gM[3] / 2, gM[4] / 2], [gM[3] / 2, gM[1], gM[5] / 2], [gM[4] / 2, gM[5] / 2, gM[2]]])
    gt = 2.0 * M @ n
    G = gm + n @ M @ n
    q = (gt - n * (n @ gt)) / J
    out = np.zeros((3, 3))
    for j in range(3):
        d = np.array(U[(j + 1) % 3]) - np.array(U[(j + 2) % 3])
        out[j] = (np.cross(d, n) * A + J * dA[j]) * G + J * A * np.cross(d, q)
    return out, J * A * G


@pytest.mark.parametrize("snap", [1, 2, 4, 8])
@pytest.mark.parametrize("lanes", [5, 0])
def test_triangles_on_the_grid(snap, lanes):
    """Vertices on multiples of 1 / snap: planes cut triangles in voxel edges and corners, where rounding
    decides which plane an edge belongs to and whether a touching piece is empty.  The gradients equal those
    of the plain operations: FP64 sums of a few dozen terms (1e-13) rounded to FP32 (2^-24), against the
    largest of the row's terms."""
    R, few = 8, 60
    n = few if lanes == 5 else 80000
    p, w = _snapped("triangles", n, R, snap, 5.0, 10 + snap)
    grid = synth.Grid((0.0, 0.0, 0.0), 1.0 / R, R)
    ctx = vx.Context(DEV)
    geom = _geom("triangles", p, w)
    keys = ctx.voxelize(grid, **geom).keys.clone()
    gm, gM = _loss(keys, 4)
    g, gw = ctx.backward(grid, keys0=keys, grad_mass=[gm], grad_moment=[gM], **geom)
    g, gw = g.cpu().numpy().reshape(n, 3, 4)[..., :3], gw.cpu().numpy()
    index = {int(k): i for i, k in enumerate(keys.cpu().numpy())}
    gm, gM = gm.cpu().numpy().astype(np.float64), gM.cpu().numpy().astype(np.float64)
    U = (p[:few, :, :3] * np.float32(R)).astype(np.float32)
    for i in range(few):
        ref, val, size, big = np.zeros((3, 3)), 0.0, 0.0, 0.0
        lo = np.maximum(np.floor(U[i].min(0)) - 1, 0).astype(int)
        hi = np.minimum(np.floor(U[i].max(0)), R - 1).astype(int)
        for v in np.ndindex(*np.maximum(hi - lo + 1, 0)):
            v = [int(a + b) for a, b in zip(lo, v)]
            key = sum(((v[a] >> t) & 1) << (3 * t + a) for t in range(3) for a in range(3))
            if key in index:
                d, x = _clip_gradient(U[i], v, gm[index[key]], gM[index[key]])
                ref, val, size, big = ref + d, val + x, max(size, np.abs(d).max()), max(big, abs(x))
        assert np.abs(g[i] - ref * float(w[i]) * R).max() <= 2.0 ** -22 * (size * float(w[i]) * R) + 1e-12, i
        assert abs(gw[i] - val) <= 2.0 ** -22 * big + 1e-12, i
    ctx.close()


@pytest.mark.parametrize("lanes", [5, 0])
@pytest.mark.parametrize("snap", [0, 1, 8])
def test_segment_ends_on_planes(snap, lanes):
    """With one loss weight for every voxel the loss is that weight times pi r^2 |B - A| (times the segment's
    weight), however the planes cut it: its gradients with respect to both ends, the radius and the weight.  Ends
    lie on the planes of a box that cuts the segments off, or on multiples of 1 / snap.  FP64 sums of up to
    50 pieces, whose sliding ends cancel from pieces up to 1 / 1e-3 larger: 1e-12 of the gradient, and the FP32
    rounding (2^-24)."""
    R, n = 16, (3000 if lanes == 5 else 80000)
    rng = np.random.default_rng(snap + 7)
    P = np.clip(rng.uniform(2, 14, (n, 1, 3)) + rng.uniform(-4, 4, (n, 2, 3)), 3, 13)
    if snap:
        P = np.round(P * snap) / snap
    P = P.astype(np.float32)
    # (a segment without length has no gradient; one in a voxel plane lies in the voxels on both sides)
    flat = ((P[:, 0] == P[:, 1]) & (P[:, 0] == np.round(P[:, 0]))).any(1)
    d = P[:, 1].astype(np.float64) - P[:, 0]
    length = np.sqrt((d * d).sum(1))
    # near-parallel to a plane: the pieces' sliding ends are large and cancel
    steep = (np.abs(d) < 1e-3) & (d != 0)
    use = ~flat & (length > 0.01) & ~steep.any(1)
    assert use.sum() > n // 3
    ctrl = np.zeros((n, 2, 4), np.float32)
    ctrl[..., :3], ctrl[..., 3] = P / np.float32(R), np.float32(0.25 / R)
    w = rng.uniform(0.5, 2.0, n).astype(np.float32)
    grid = synth.Grid((0.0, 0.0, 0.0), 1.0 / R, R)
    ctx = vx.Context(DEV)
    geom = _geom("fibers", ctrl, w)
    keys = ctx.voxelize(grid, **geom).keys.clone()
    ones, none = torch.ones(keys.shape[0], device=DEV), torch.zeros(keys.shape[0], 6, device=DEV)
    g, gw = ctx.backward(grid, keys0=keys, grad_mass=[ones], grad_moment=[none], **geom)
    g, gw = g.cpu().numpy().reshape(n, 2, 4).astype(np.float64), gw.cpu().numpy().astype(np.float64)
    r = 0.25
    c = np.pi * r * r * w.astype(np.float64) * R
    with np.errstate(invalid="ignore", divide="ignore"):
        t = d / length[:, None]
    for got, ref in ((g[:, 0, :3], -c[:, None] * t), (g[:, 1, :3], c[:, None] * t)):
        assert np.abs(got - ref)[use].max(1).max() <= 2.0 ** -22 * c.max()
    half = 0.5 * 2.0 * np.pi * r * length * w * R
    for e in range(2):
        assert (np.abs(g[:, e, 3] - half) <= 2.0 ** -22 * half + 1e-9)[use].all()
    mass = np.pi * r * r * length
    assert (np.abs(gw - mass) <= 2.0 ** -22 * mass + 1e-9)[use].all()
    ctx.close()
